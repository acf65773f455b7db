// maclab_window.cuh -- several steps of MacLABSWE (Zhou, arXiv:1902.02999,
// Section 3, Eqs. Mac.lb.6 / Mac.lb.7 in the perturbation form of
// maclab_kernels.cuh) per launch, for grids and batches whose whole state
// fits the chip's caches.
//
// A block owns a tile and loads it with a halo of k nodes (its window) into
// shared memory, takes up to k steps there and stores the tile; after step s
// the nodes within k - s of the tile are up to date, so nothing is exchanged
// between blocks inside a launch.  A window reaches across a periodic edge
// by wrapped loads; at the other edges it ends, and the ring of ghost nodes
// beyond it is derived from the window's own nodes each step (mirrored, or
// wrapped where the tile spans the whole axis).
//
// Why: on a small grid a step is bound by the latency of one block's load,
// derive, barrier, gather and store chain and by the launch, not by any
// throughput; here the loads, stores and launch are paid once per k steps
// and a step inside costs two block barriers.  The rows of halo derived
// twice are cheap in FP32 (idle lanes), and the host weighs them against
// the launch when it picks tile and k (window_plan in maclab.cu).
//
// One step, old raw state in buffer s & 1:
//   A  every node of the region derives its source quantities (derive2 /
//      derive) into shared memory; ghosts likewise, with their flips;
//   B  every fast node gathers and updates (gather_pair / update64) into
//      the other raw buffer; a node with a bounce-back link reads its own
//      outgoing values for the bounced links (FP64, as general_node64) or is
//      updated by eight lanes, one link each, its sums added in the order of
//      general_node (FP32);
//   C  Dirichlet nodes take their values from the new inward node.
// Every node takes the operations of the single-step kernels in their
// order, so the states are bitwise theirs.
//
// Measured per step, single-step launches (graph replay where the boundary
// is steady) -> this kernel: 256 x 256 lake FP32 11.4 -> 3.3 us, 400 x 3
// tidal strip FP64 49 -> 5.4 us, eight 256 x 256 lakes FP64 195 -> 70 us.
#pragma once
#include "maclab_march.cuh"

namespace maclab {
namespace window {

constexpr int MAX_THREADS = 512;
constexpr int MAX_STEPS = 16;  // steps per launch, at most (kernel parameters hold their boundary values)
constexpr int MAX_PAIRS = 4;   // FP32: node pairs per thread, at most

struct Item {  // one tile
    int inst;            // instance of the batch
    int x0, x1, y0, y1;  // nodes [x0, x1) x [y0, y1)
    int pad;
    long long off;       // the instance's first element in the packed arrays
};

struct Shape {  // shared by every block of a launch (the largest window)
    int hw;      // half of the padded row length
    int rows;    // padded rows
    int nlist;   // room in the list of nodes with a bounce-back link
    int ndir;    // room in the list of Dirichlet nodes
};

template <typename T>
struct Buffers {        // packed bases
    const T* in[3];     // eta, u, v at the launch's first step
    T* out[3];          // ... after its last
    T* prev[3];         // ... before its last (the residual's earlier state), or nullptr
};

struct DirTable {
    DirValues v[MAX_STEPS];  // values at the end of each step
};

struct Dir {
    int cell, inward, meta, pad;
    double D64;
};

// Arrays of one window.  A padded row holds two columns, the window, and at
// least one more; node (col, row) of the window is at padded (col + 2, row + 1).
// FP32: the outgoing values read one column off and (eta, D) are split by
// column parity, as in maclab_march.cuh, so that a warp's reads are
// consecutive.
template <typename T>
struct Arrays;
template <>
struct Arrays<float> {
    float* o;        // [6][rows][2][hw]: o1 o2 o4 o5 o6 o8 by column parity
    float2* ed;      // [rows][2][hw]: (eta, D) by column parity
    float* o37;      // [2][rows][2 hw]: o3, o7
    float* raws;     // [2][3][rows][2 hw]: eta, u, v of two steps
    float* D;        // [rows][2 hw]
    Dir* dir;
    uint8_t* type;   // [rows][2 hw]
    uint16_t* list;  // cells of the nodes with a bounce-back link
    int hw, rows;
    __device__ __forceinline__ int plane() const { return rows * 2 * hw; }
    __device__ __forceinline__ float* raw(int b) const { return raws + b * 3 * plane(); }
};
template <>
struct Arrays<double> {
    double* o;       // [8][rows][2 hw]
    double* own;     // [3][rows][2 hw]: ownh, hFx, hFy
    double* raws;
    double* D;
    double* bed;     // [3][rows][2 hw]: stencils of D
    Dir* dir;
    uint16_t* type;  // type byte | bounced links << 8 (bit a - 1: direction a)
    uint16_t* list;
    int hw, rows;
    __device__ __forceinline__ int plane() const { return rows * 2 * hw; }
    __device__ __forceinline__ double* raw(int b) const { return raws + b * 3 * plane(); }
};

template <typename T>
__host__ __device__ constexpr size_t cell_bytes() { return sizeof(T) == 4 ? 68 : 168; }
__host__ __device__ inline size_t smem_of(size_t per_cell, const Shape& s)
{
    const size_t cells = (size_t)s.rows * 2 * s.hw;
    return cells * per_cell + (size_t)s.ndir * sizeof(Dir) + ((cells + 15) & ~size_t(15)) * (per_cell > 100 ? 2 : 1) +
           (((size_t)s.nlist * 2 + 15) & ~size_t(15));
}

template <typename T>
__device__ __forceinline__ Arrays<T> carve(unsigned char* p, const Shape& s)
{
    Arrays<T> a;
    a.hw = s.hw;
    a.rows = s.rows;
    const int n = s.rows * 2 * s.hw;
    T* q = reinterpret_cast<T*>(p);
    if constexpr (std::is_same<T, float>::value) {
        a.ed = reinterpret_cast<float2*>(q);
        a.o = q + 2 * n;
        a.o37 = a.o + 6 * n;
        a.raws = a.o37 + 2 * n;
    } else {
        a.o = q;
        a.own = a.o + 8 * n;
        a.raws = a.own + 3 * n;
    }
    a.D = a.raws + 6 * n;
    T* end = a.D + n;
    if constexpr (std::is_same<T, double>::value) {
        a.bed = end;
        end += 3 * n;
    }
    a.dir = reinterpret_cast<Dir*>(end);
    a.type = reinterpret_cast<decltype(a.type)>(a.dir + s.ndir);
    a.list = reinterpret_cast<uint16_t*>(a.type + ((n + 15) & ~15));
    return a;
}

// One axis of a window: nodes [lo, lo + n) of an axis of `size` nodes.
struct Axis {
    int lo, n, size;
    int first, last;  // source (window index) of the ghost before / after the window, -1: a wall,
                      // -2: the window ends inside the grid (no ghost: out-of-date nodes end there)
    uint8_t flip;     // mirror bit of a specular ghost
    bool flip_first, flip_last;
    // region needed as input of a step with m more steps after it
    int t0, t1;       // tile, in window indexes
    __device__ __forceinline__ int begin(int m) const { return max(0, t0 - m); }
    __device__ __forceinline__ int end(int m) const { return min(n, t1 + m); }
};

__device__ __forceinline__ Axis make_axis(int x0, int x1, int size, int lo_kind, int hi_kind, int k, uint8_t bit)
{
    Axis a;
    const bool wraps = lo_kind == EDGE_PER && !(x0 == 0 && x1 == size);
    int lo = x0 - k, hi = x1 + k;
    if (!wraps) {
        lo = max(lo, 0);
        hi = min(hi, size);
    }
    a.lo = lo;
    a.n = hi - lo;
    a.size = size;
    a.t0 = x0 - lo;
    a.t1 = x1 - lo;
    a.flip = bit;
    a.first = a.last = -2;
    a.flip_first = a.flip_last = false;
    if (!wraps && lo == 0) {
        a.first = lo_kind == EDGE_BB ? -1 : (lo_kind == EDGE_PER ? size - 1 : 0);
        a.flip_first = lo_kind == EDGE_SPEC;
    }
    if (!wraps && hi == size) {
        a.last = hi_kind == EDGE_BB ? -1 : (hi_kind == EDGE_PER ? 0 : a.n - 1);
        a.flip_last = hi_kind == EDGE_SPEC;
    }
    return a;
}

// Window index i (-1 .. n) resolved to the window's own node that supplies
// it: -1 for a wall (and for the out-of-date side, whose nodes no valid node
// reads), with the mirror bit set for a specular ghost.
__device__ __forceinline__ int resolve(const Axis& a, int i, uint8_t& flip)
{
    if (i >= 0 && i < a.n) return i;
    if (i < 0) {
        if (a.flip_first) flip |= a.flip;
        return a.first < 0 ? -1 : a.first;
    }
    if (a.flip_last) flip |= a.flip;
    return a.last < 0 ? -1 : a.last;
}

__device__ __forceinline__ int wrapped(int i, int n)
{
    if (i >= 0 && i < n) return i;
    i %= n;
    return i < 0 ? i + n : i;
}

// Ghost q of the ring around the window: rows -1 and WH (with corners), then
// columns -1 and WW.  False when the side holds no ghost or a wall.
__device__ __forceinline__ bool ghost(const Axis& ax, const Axis& ay, int q, int& col, int& row, int& sc, int& sr,
                                      uint8_t& flip)
{
    const int w2 = ax.n + 2;
    if (q < 2 * w2) {
        row = q < w2 ? -1 : ay.n;
        col = (q < w2 ? q : q - w2) - 1;
    } else {
        const int p = q - 2 * w2;
        col = p < ay.n ? -1 : ax.n;
        row = p < ay.n ? p : p - ay.n;
    }
    flip = 0;
    sc = resolve(ax, col, flip);
    sr = resolve(ay, row, flip);
    return sc >= 0 && sr >= 0;
}

// Update of a node with a bounce-back link, one link per lane of a group of
// eight (lane a - 1 of the group: direction a): general_node's operations in
// its order, every lane with all sums.
template <typename T>
__device__ __forceinline__ void general8(const Arrays<T>& A, const T* raw, const Coef<T>& c, const Axis& ax,
                                         const Axis& ay, int cell, int lane, T& oe, T& ou, T& ov)
{
    using O = Op<T>;
    const int pw = 2 * A.hw, n = A.plane();
    const int pr = cell / pw, pc = cell - pr * pw;
    const int a = 1 + (lane & 7);
    // c_a: x = +1 for 1 2 8, -1 for 4 5 6; y = +1 for 2 3 4, -1 for 6 7 8
    const int cx = ((0x106 >> a) & 1) - ((0x070 >> a) & 1);
    const int cy = ((0x01C >> a) & 1) - ((0x1C0 >> a) & 1);
    const NodeQ<T> X = node_q_of(c, raw[cell], A.D[cell], raw[n + cell], raw[2 * n + cell], 0);
    uint8_t flip = 0;
    const int sc = resolve(ax, pc - 2 - cx, flip), sr = resolve(ay, pr - 1 - cy, flip);
    bool bounce = sc < 0 || sr < 0;
    const int s = bounce ? cell : (sr + 1) * pw + sc + 2;
    bounce = bounce || (A.type[s] & KIND_MASK) == K_SOLID;
    NodeQ<T> Y = X;
    if (!bounce) Y = node_q_of(c, raw[s], A.D[s], raw[n + s], raw[2 * n + s], flip);
    const T lam = (a & 1) ? T(1) : T(0.25);
    const T fx = cx > 0 ? T(1) : cx < 0 ? T(-1) : T(0), fy = cy > 0 ? T(1) : cy < 0 ? T(-1) : T(0);
    T w = feq_diff_dir(c, Y, bounce ? -fx : fx, bounce ? -fy : fy, lam);
    if (!bounce) {
        const T bed = O::mul(O::mul(lam, c.G6), O::mul(O::add(X.eta, Y.eta), O::sub(X.D, Y.D)));
        const T frc = O::mul(O::mul(lam, c.KF), O::fma(fx, O::add(X.Fx, Y.Fx), O::mul(fy, O::add(X.Fy, Y.Fy))));
        w = O::add(O::add(w, bed), frc);
    }
    T Sh = general_rest(c, X), Sx = T(0), Sy = T(0);
    const unsigned group = 0xffu << (lane & 24);
#pragma unroll
    for (int b = 1; b < 9; ++b) {
        const T wb = __shfl_sync(group, w, (lane & 24) + b - 1);
        const int bx = ((0x106 >> b) & 1) - ((0x070 >> b) & 1), by = ((0x01C >> b) & 1) - ((0x1C0 >> b) & 1);
        Sh = O::add(Sh, wb);
        Sx = O::fma(T(bx), wb, Sx);
        Sy = O::fma(T(by), wb, Sy);
    }
    general_finish(c, X, Sh, Sx, Sy, (A.type[cell] & KIND_MASK) == K_NOSLIP, ou, ov);
    oe = Sh;
}

// A: derive the pair at padded (pr, pc); two: both columns lie in the window.
template <int FM>
__device__ __forceinline__ void put_pair(const Arrays<float>& A, int pr, int pc, bool two, const Src2& s)
{
    const int hw = A.hw, j = pc >> 1, row = pr * 2 * hw, n = A.plane();
    const float2 v6[6] = {s.o1, s.o2, s.o4, s.o5, s.o6, s.o8};
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        A.o[d * n + row + j] = v6[d].x;
        if (two) A.o[d * n + row + hw + j] = v6[d].y;
    }
    A.ed[row + j] = make_float2(s.eta.x, s.D.x);
    if (two) {
        A.ed[row + hw + j] = make_float2(s.eta.y, s.D.y);
        *reinterpret_cast<float2*>(&A.o37[row + pc]) = s.o3;
        *reinterpret_cast<float2*>(&A.o37[n + row + pc]) = s.o7;
    } else {
        A.o37[row + pc] = s.o3.x;
        A.o37[n + row + pc] = s.o7.x;
    }
}
__device__ __forceinline__ void put_one(const Arrays<float>& A, int pr, int pc, const Src<float>& s)
{
    const int row = pr * 2 * A.hw, n = A.plane(), j = row + (pc & 1) * A.hw + (pc >> 1);
    const float v6[6] = {s.o1, s.o2, s.o4, s.o5, s.o6, s.o8};
#pragma unroll
    for (int d = 0; d < 6; ++d) A.o[d * n + j] = v6[d];
    A.ed[j] = make_float2(s.eta, s.D);
    A.o37[row + pc] = s.o3;
    A.o37[n + row + pc] = s.o7;
}
__device__ __forceinline__ void put_one(const Arrays<double>& A, int pr, int pc, const Src<double>& s)
{
    const int q = pr * 2 * A.hw + pc, n = A.plane();
    const double v8[8] = {s.o1, s.o2, s.o3, s.o4, s.o5, s.o6, s.o7, s.o8};
#pragma unroll
    for (int d = 0; d < 8; ++d) A.o[d * n + q] = v8[d];
    A.own[q] = s.ownh;
    A.own[n + q] = s.hFx;
    A.own[2 * n + q] = s.hFy;
}

}  // namespace window

// Block b takes `steps` steps (1 .. MAX_STEPS) of tile items[b].  NP (FP32):
// node pairs per thread, enough for the largest window.  tab: boundary
// values of each step, or (steady) the instance's own.  active: batch flags
// or nullptr.
template <typename T, int FM, int NP>
__global__ void __launch_bounds__(window::MAX_THREADS, 1)
step_window_kernel(const BatchInst<T>* __restrict__ insts, const window::Item* __restrict__ items,
                   const uint8_t* __restrict__ active, const __grid_constant__ window::Buffers<T> buf,
                   const __grid_constant__ window::Shape shape, int steps, int steady,
                   const __grid_constant__ window::DirTable tab)
{
    using namespace window;
    extern __shared__ __align__(16) unsigned char window_smem[];
    __shared__ int counts[2];  // nodes with a bounce-back link, Dirichlet nodes
    const Item it = items[blockIdx.x];
    if (active && !active[it.inst]) return;  // whole block
    const BatchInst<T>& in = insts[it.inst];
    const Fields<T>& f = in.f[0];
    const Coef<T> c = f.c;
    const int nx = f.nx, ny = f.ny, pitch = f.pitch;
    const Axis ax = make_axis(it.x0, it.x1, nx, f.edge[0], f.edge[1], steps, 1);
    const Axis ay = make_axis(it.y0, it.y1, ny, f.edge[2], f.edge[3], steps, 2);
    const Arrays<T> A = carve<T>(window_smem, shape);
    const int pw = 2 * A.hw, n = A.plane();
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    if (tid < 2) counts[tid] = 0;
    __syncthreads();
    // ---- load the window
    for (int p = tid; p < ax.n * ay.n; p += nt) {
        const int r = p / ax.n, q = p - r * ax.n;
        const int gx = wrapped(ax.lo + q, nx), gy = wrapped(ay.lo + r, ny);
        const size_t g = (size_t)gy * pitch + gx;
        const int cell = (r + 1) * pw + q + 2;
        const uint8_t ty = f.type[g];
        A.raws[cell] = buf.in[0][it.off + g];
        A.raws[n + cell] = buf.in[1][it.off + g];
        A.raws[2 * n + cell] = buf.in[2][it.off + g];
        A.D[cell] = f.D[g];
        A.type[cell] = ty;
        const int kind = ty & KIND_MASK;
        if constexpr (std::is_same<T, double>::value) {
            const Bed64 b = bed_at(f, g);
            A.bed[cell] = b.s;
            A.bed[n + cell] = b.x;
            A.bed[2 * n + cell] = b.y;
        }
        if (ty & GENERAL_BIT) {
            A.list[atomicAdd(&counts[0], 1)] = (uint16_t)cell;
        } else if (kind >= K_DIR_H) {
            // the edge a Dirichlet node belongs to: the first of W, E, S, N it touches
            const int ed = gx == 0 ? 0 : gx == nx - 1 ? 1 : gy == 0 ? 2 : 3;
            const int step_in = ed == 0 ? 1 : ed == 1 ? -1 : ed == 2 ? pw : -pw;
            A.dir[atomicAdd(&counts[1], 1)] = Dir{cell, cell + step_in, kind | (ed << 4), 0, in.D64[g]};
        }
    }
    const int nghost = 2 * (ax.n + 2) + 2 * ay.n;
    if constexpr (std::is_same<T, double>::value) {
        // bounced links of the listed nodes
        __syncthreads();
        for (int g = tid; g < counts[0]; g += nt) {
            const int cell = A.list[g], pr = cell / pw, pc = cell - pr * pw;
            uint32_t mask = 0;
#pragma unroll
            for (int a = 1; a < 9; ++a) {
                const int cx = (a == 1 || a == 2 || a == 8) - (a == 4 || a == 5 || a == 6);
                const int cy = (a >= 2 && a <= 4) - (a >= 6);
                uint8_t flip = 0;
                const int sc = resolve(ax, pc - 2 - cx, flip), sr = resolve(ay, pr - 1 - cy, flip);
                const bool back = sc < 0 || sr < 0 || (A.type[(sr + 1) * pw + sc + 2] & KIND_MASK) == K_SOLID;
                mask |= (back ? 1u : 0u) << (a - 1);
            }
            A.type[cell] |= (uint16_t)(mask << 8);
        }
    }
    // FP32: the thread's pairs, fixed for the launch
    int prow[NP], pcol[NP];
    unsigned pflag[NP];  // bits 0, 1: fast node to update; 2, 3: no-slip; 4: second column in the window
    Src2 own[NP];
    const int npr = (ax.n + 1) / 2;  // pairs per window row
    __syncthreads();
    if constexpr (std::is_same<T, float>::value) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int p = tid + k * nt;
            const int r = p / npr, j = p - r * npr;
            prow[k] = r;  // rows past the window never match a region
            pcol[k] = 2 * j;
            pflag[k] = 0;
            if (r < ay.n) {
                const bool two = 2 * j + 1 < ax.n;
                const uint32_t t0 = A.type[(r + 1) * pw + 2 * j + 2], t1 = two ? A.type[(r + 1) * pw + 2 * j + 3] : 0;
                // fast: kind 1 .. 7 without the bounce-back bit
                pflag[k] = (t0 - 1u < 7u ? 1u : 0u) | (t1 - 1u < 7u ? 2u : 0u) |
                           ((t0 & KIND_MASK) == K_NOSLIP ? 4u : 0u) | ((t1 & KIND_MASK) == K_NOSLIP ? 8u : 0u) |
                           (two ? 16u : 0u);
            }
        }
    }
    const Coef2 c2 = march::pairs_of(c);
    const int ng = counts[0], nd = counts[1];
    for (int s = 0; s < steps; ++s) {
        const int m = steps - s;  // steps still to take, this one included
        const T* raw = A.raw(s & 1);
        T* nxt = A.raw(1 - (s & 1));
        // ---- A: source quantities of the region and its ghosts
        const int a0 = ay.begin(m), a1 = ay.end(m), b0 = ax.begin(m), b1 = ax.end(m);
        if constexpr (std::is_same<T, float>::value) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                if (prow[k] < a0 || prow[k] >= a1 || pcol[k] + 1 < b0 || pcol[k] >= b1) continue;
                const int q = (prow[k] + 1) * pw + pcol[k] + 2;
                const float2 e = *reinterpret_cast<const float2*>(raw + q), u = *reinterpret_cast<const float2*>(raw + n + q);
                const float2 v = *reinterpret_cast<const float2*>(raw + 2 * n + q);
                const float2 d = *reinterpret_cast<const float2*>(A.D + q);
                derive2<FM>(c2, Raw<float>{e.x, u.x, v.x, d.x, 0}, Raw<float>{e.y, u.y, v.y, d.y, 0}, own[k]);
                put_pair<FM>(A, prow[k] + 1, pcol[k] + 2, (pflag[k] & 16u) != 0, own[k]);
            }
        } else {
            const int w = b1 - b0, cells = w * (a1 - a0);
            for (int p = tid; p < cells; p += nt) {
                const int r = a0 + p / w, q = b0 + p % w, cell = (r + 1) * pw + q + 2;
                Src<T> src;
                derive<T, FM>(c, Raw<T>{raw[cell], raw[n + cell], raw[2 * n + cell], A.D[cell], 0}, src);
                put_one(A, r + 1, q + 2, src);
            }
        }
        for (int q = tid; q < nghost; q += nt) {
            int col, row, sc, sr;
            uint8_t flip;
            if (!ghost(ax, ay, q, col, row, sc, sr, flip)) continue;
            const int cell = (sr + 1) * pw + sc + 2;
            Src<T> src;
            derive<T, FM>(c, Raw<T>{raw[cell], raw[n + cell], raw[2 * n + cell], A.D[cell], flip}, src);
            put_one(A, row + 1, col + 2, src);
            if constexpr (std::is_same<T, double>::value)
                A.raw(s & 1)[(row + 1) * pw + col + 2] = src.eta;  // the stencils of eta read it
        }
        __syncthreads();
        // ---- B: update
        const int e0 = ay.begin(m - 1), e1 = ay.end(m - 1), d0 = ax.begin(m - 1), d1 = ax.end(m - 1);
        if constexpr (std::is_same<T, float>::value) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                if (prow[k] < e0 || prow[k] >= e1 || pcol[k] + 1 < d0 || pcol[k] >= d1 || !(pflag[k] & 3u)) continue;
                const int hw = A.hw, j = (pcol[k] + 2) >> 1, q = (prow[k] + 1) * pw + pcol[k] + 2;
                // rows above, own, below; even columns first, odd columns hw on
                const int rm = prow[k] * pw + j, rc = rm + pw, rp = rc + pw;
                const float *o1 = A.o, *o2 = A.o + n, *o4 = A.o + 2 * n, *o5 = A.o + 3 * n, *o6 = A.o + 4 * n,
                            *o8 = A.o + 5 * n;
                const float2 m4[4] = {A.ed[rm + hw - 1], A.ed[rm], A.ed[rm + hw], A.ed[rm + 1]};
                // (the second column of an odd window's last pair is a ghost, or out of date)
                const float2 c4[4] = {A.ed[rc + hw - 1], make_float2(own[k].eta.x, own[k].D.x),
                                      (pflag[k] & 16u) ? make_float2(own[k].eta.y, own[k].D.y) : A.ed[rc + hw],
                                      A.ed[rc + 1]};
                const float2 p4[4] = {A.ed[rp + hw - 1], A.ed[rp], A.ed[rp + hw], A.ed[rp + 1]};
                float2 oe, ou, ov;
                march::gather_pair(c2, make_float2(o1[rc + hw - 1], o1[rc]), make_float2(o2[rm + hw - 1], o2[rm]),
                                   make_float2(o5[rc + hw], o5[rc + 1]), make_float2(o4[rm + hw], o4[rm + 1]),
                                   *reinterpret_cast<const float2*>(A.o37 + q - pw),
                                   make_float2(o8[rp + hw - 1], o8[rp]), make_float2(o6[rp + hw], o6[rp + 1]),
                                   *reinterpret_cast<const float2*>(A.o37 + n + q + pw), m4, c4, p4, own[k].ownh,
                                   own[k].hFx, own[k].hFy, (pflag[k] & 4u) != 0, (pflag[k] & 8u) != 0, oe, ou, ov);
                if ((pflag[k] & 3u) == 3u) {
                    *reinterpret_cast<float2*>(nxt + q) = oe;
                    *reinterpret_cast<float2*>(nxt + n + q) = ou;
                    *reinterpret_cast<float2*>(nxt + 2 * n + q) = ov;
                } else {
                    const bool hi = (pflag[k] & 2u) != 0;
                    nxt[q + (hi ? 1 : 0)] = hi ? oe.y : oe.x;
                    nxt[n + q + (hi ? 1 : 0)] = hi ? ou.y : ou.x;
                    nxt[2 * n + q + (hi ? 1 : 0)] = hi ? ov.y : ov.x;
                }
            }
        } else {
            const int w = d1 - d0, cells = w * (e1 - e0);
            for (int p = tid; p < cells; p += nt) {
                const int r = e0 + p / w, q = (r + 1) * pw + d0 + p % w + 2;
                const uint32_t ty = A.type[q];
                if ((ty & KIND_MASK) == K_SOLID) continue;
                // where each link reads: the neighbour, or for a bounced link
                // the node itself, opposite direction
                const int nb[8] = {q - 1, q - pw - 1, q - pw, q - pw + 1, q + 1, q + pw + 1, q + pw, q + pw - 1};
                const uint32_t mask = ty >> 8;
                double o[8], eta[8];
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const bool back = (mask >> a) & 1u;
                    o[a] = A.o[back ? ((a + 4) & 7) * n + q : a * n + nb[a]];
                    eta[a] = raw[back ? q : nb[a]];
                }
                T oe, ou, ov;
                update64(c, o[0], o[1], o[7], o[4], o[3], o[5], o[2], o[6],
                         Eta8{eta[1], eta[2], eta[3], eta[0], eta[4], eta[7], eta[6], eta[5]}, raw[q], A.D[q], A.own[q],
                         A.own[n + q], A.own[2 * n + q], Bed64{A.bed[q], A.bed[n + q], A.bed[2 * n + q]},
                         (ty & KIND_MASK) == K_NOSLIP, oe, ou, ov);
                nxt[q] = oe;
                nxt[n + q] = ou;
                nxt[2 * n + q] = ov;
            }
        }
        for (int g = tid >> 3; g < (std::is_same<T, double>::value ? 0 : ng); g += nt >> 3) {
            const int cell = A.list[g], r = cell / pw - 1, q = cell - (r + 1) * pw - 2;
            if (r < e0 || r >= e1 || q < d0 || q >= d1) continue;  // the group's eight lanes alike
            T oe, ou, ov;
            general8<T>(A, raw, c, ax, ay, cell, lane, oe, ou, ov);
            if ((lane & 7) == 0) {
                nxt[cell] = oe;
                nxt[n + cell] = ou;
                nxt[2 * n + cell] = ov;
            }
        }
        __syncthreads();
        // ---- C: Dirichlet nodes
        if (nd > 0) {
            const DirValues& bv = steady ? in.bv : tab.v[s];
            for (int k = tid; k < nd; k += nt) {
                const Dir d = A.dir[k];
                const int r = d.cell / pw - 1, q = d.cell - (r + 1) * pw - 2;
                if (r < e0 || r >= e1 || q < d0 || q >= d1) continue;
                // dirichlet_node on the window's arrays (D64 of the node itself is in the entry)
                dirichlet_value(nxt, nxt + n, nxt + 2 * n, A.D, d.D64, d.cell, d.inward, d.meta, bv);
            }
            __syncthreads();
        }
    }
    // ---- store the tile
    const T *last = A.raw(steps & 1), *before = A.raw(1 - (steps & 1));
    const int tw = it.x1 - it.x0, cells = tw * (it.y1 - it.y0);
    for (int p = tid; p < cells; p += nt) {
        const int r = p / tw, q = p - r * tw;
        const int cell = (ay.t0 + r + 1) * pw + ax.t0 + q + 2;
        if ((A.type[cell] & KIND_MASK) == K_SOLID) continue;
        const size_t g = it.off + (size_t)(it.y0 + r) * pitch + it.x0 + q;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            buf.out[k][g] = last[k * n + cell];
            if (buf.prev[0]) buf.prev[k][g] = before[k * n + cell];
        }
    }
}

}  // namespace maclab
