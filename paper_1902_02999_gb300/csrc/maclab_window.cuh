// maclab_window.cuh -- several steps of MacLABSWE (Zhou, arXiv:1902.02999,
// Section 3, Eqs. Mac.lb.6 / Mac.lb.7 in the perturbation form of
// maclab_kernels.cuh) per launch, for grids and batches whose whole state
// fits the chip's caches.
//
// A block owns a tile and loads it with a halo of k nodes (its window) into
// shared memory, takes up to k steps there and stores the tile; with m steps
// to take, the nodes within m of the tile enter the next one, so nothing is
// exchanged between blocks inside a launch.  A window reaches across a
// periodic edge by wrapped loads; at the other edges it ends, and the ring of
// ghost nodes beyond it is derived from the window's own nodes each step
// (mirrored, or wrapped where the tile spans the whole axis).
//
// Why: on a small grid a step is bound by the latency of one block's load,
// derive, barrier, gather and store chain and by the launch, not by any
// throughput; here the loads, stores and launch are paid once per k steps
// and a step inside costs two block barriers.  The rows of halo derived
// twice are cheap in FP32 (idle lanes), and the host weighs them against
// the launch when it picks tile and k (window.cu).
//
// What does not change from step to step is laid out once per handle
// (window_lists_kernel): the work of a window as a list of units (FP32: node
// pairs, FP64: nodes) that hold a node that is not solid, in order of their
// distance from the tile, so that the work of a step with m to take is the
// front of the list, packed without dry nodes; its ghosts, its nodes with a
// bounce-back link with each link's source, and its Dirichlet nodes.
//
// One step, old raw state in buffer s & 1:
//   A  every unit of the region derives its source quantities (derive2 /
//      derive64) into shared memory; ghosts likewise, with their flips;
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
// is steady) -> this kernel: 256 x 256 lake FP32 11.4 -> 1.9 us, 1001 x 333
// channel FP32 10.1 -> 5.5 us, 400 x 3 tidal strip FP64 49 -> 3.4 us, eight
// 256 x 256 lakes FP64 195 -> 63 us (both with FP64's cheaper arithmetic of
// today in the second figure).  Computing the lists' content in every launch instead took
// 3.3, 9.0, 5.4 and 70 us.  Inside a launch (clock readings, 40 x 24 tile,
// k = 6, 910 pairs): loads 2,000 cycles, a step 1,700 (A) + 2,100 (B), store
// 1,300; the FP32 pipe is busy about half of a step.
#pragma once
#include "maclab_march.cuh"

namespace maclab {
namespace window {

constexpr int MAX_THREADS = 512;
constexpr int MAX_STEPS = 16;  // steps per launch, at most (kernel parameters hold their boundary values)
constexpr int MAX_PAIRS = 4;   // FP32: node pairs per thread, at most
constexpr uint32_t NONE = 0xffffffffu;

struct Item {  // one tile
    int inst;            // instance of the batch
    int x0, x1, y0, y1;  // nodes [x0, x1) x [y0, y1)
    int pad;
    long long off;       // the instance's first element in the packed arrays
};

struct Shape {  // shared by every block of a launch (the largest window)
    int k;       // halo of the windows: steps per launch, at most
    int hw;      // half of the padded row length
    int rows;    // padded rows
    int units;   // room in a tile's list of units
    int ghosts;  // ... of ghosts
    int walls;   // ... of nodes with a bounce-back link (FP32; the most of any tile)
    int dirs;    // ... of Dirichlet nodes
    __host__ __device__ int cells() const { return rows * 2 * hw; }
};

// Per tile: how many entries lie within d of the tile (d = 0 .. k).
struct Head {
    Item item;
    uint16_t units[MAX_STEPS + 1], ghosts[MAX_STEPS + 1], walls[MAX_STEPS + 1];
    uint16_t dirs;
};
// A unit.  cell: padded window cell of its (first) node | flags << 16;
// g0, g1: offsets of its nodes in the instance's arrays (NONE: not loaded).
// half (FP32): index of the pair in an array split by column parity.
// FP64: g1 = bounced links (bit a - 1: direction a).
struct Unit {
    uint32_t cell, g0, g1, half;
};
enum : uint32_t {
    U_FAST0 = 1u << 16, U_FAST1 = 1u << 17,    // nodes the fast update writes
    U_NOSLIP0 = 1u << 18, U_NOSLIP1 = 1u << 19,
    U_TWO = 1u << 20,                          // the second column belongs to the window
    U_TILE0 = 1u << 21, U_TILE1 = 1u << 22,    // nodes of the tile (stored at the end)
    U_VEC = 1u << 23                           // g0 even and g1 = g0 + 1
};
struct Ghost {
    uint32_t cells;  // ghost | source << 16
    uint32_t flip;
};
struct Link {  // of direction lane + 1
    uint32_t src;   // source cell | flip << 16 | bounced << 18 | no-slip << 19
    uint32_t cell;
};
struct Dir {
    uint32_t cells;  // node | inward node << 16
    int meta;        // as DirNode
    int dist;
    int pad;
    double D64;
};

struct Lists {  // on the device; tile b's entries start at b times the room
    const Head* head;
    const Unit* units;
    const Ghost* ghosts;
    const Link* links;  // 8 per node
    const Dir* dirs;
};

template <typename T>
struct Buffers {        // packed bases
    const T* in[3];     // eta, u, v at the launch's first step
    T* out[3];          // ... after its last
    T* prev[3];         // ... before its last (the residual's earlier state), or nullptr
    const T* D;
    const T* bed;       // FP64: stencils of D, three planes
    size_t plane;
};

struct DirTable {
    DirValues v[MAX_STEPS];  // values at the end of each step
};

// Arrays of one window.  A padded row holds two columns, the window (from an
// even global column in FP32), and at least one more.  FP32: the outgoing
// values read one column off and (eta, D) are split by column parity, as in
// maclab_march.cuh, so that a warp's reads are consecutive.
template <typename T>
struct Arrays;
template <>
struct Arrays<float> {
    float* o;        // [6][rows][2][hw]: o1 o2 o4 o5 o6 o8 by column parity
    float2* ed;      // [rows][2][hw]: (eta, D) by column parity
    float* o37;      // [2][rows][2 hw]: o3, o7
    float* raws;     // [2][3][rows][2 hw]: eta, u, v of two steps
    float* D;        // [rows][2 hw]
    int hw, n;       // n: cells of a plane
    __device__ __forceinline__ float* raw(int b) const { return raws + b * 3 * n; }
};
template <>
struct Arrays<double> {
    double* o;       // [8][rows][2 hw]
    double* own;     // [3][rows][2 hw]: ownh, hFx, hFy
    double* raws;
    double* D;
    double* bed;     // [3][rows][2 hw]
    int hw, n;
    __device__ __forceinline__ double* raw(int b) const { return raws + b * 3 * n; }
};

template <typename T>
__host__ __device__ constexpr size_t cell_bytes() { return sizeof(T) == 4 ? 68 : 168; }

template <typename T>
__device__ __forceinline__ Arrays<T> carve(unsigned char* p, const Shape& s)
{
    Arrays<T> a;
    a.hw = s.hw;
    const int n = a.n = s.cells();
    T* q = reinterpret_cast<T*>(p);
    if constexpr (std::is_same<T, float>::value) {
        a.ed = reinterpret_cast<float2*>(q);
        a.o = q + 2 * n;
        a.o37 = a.o + 6 * n;
        a.raws = a.o37 + 2 * n;
        a.D = a.raws + 6 * n;
    } else {
        a.o = q;
        a.own = a.o + 8 * n;
        a.raws = a.own + 3 * n;
        a.D = a.raws + 6 * n;
        a.bed = a.D + n;
    }
    return a;
}

// One axis of a window: nodes [lo, lo + n) of an axis of `size` nodes.
struct Axis {
    int lo, n, size;
    int first, last;  // source (window index) of the ghost before / after the window, -1: a wall,
                      // -2: the window ends inside the grid (no ghost: out-of-date nodes end there)
    uint8_t flip;     // mirror bit of a specular ghost
    bool flip_first, flip_last;
    int t0, t1;       // the tile, in window indexes
    __host__ __device__ int dist(int i) const { return i < t0 ? t0 - i : i >= t1 ? i - t1 + 1 : 0; }
};

__host__ __device__ inline Axis make_axis(int x0, int x1, int size, int lo_kind, int hi_kind, int k, uint8_t bit)
{
    Axis a;
    const bool wraps = lo_kind == EDGE_PER && !(x0 == 0 && x1 == size);
    int lo = x0 - k, hi = x1 + k;
    if (!wraps) {
        lo = lo < 0 ? 0 : lo;
        hi = hi > size ? size : hi;
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
__host__ __device__ inline int resolve(const Axis& a, int i, uint8_t& flip)
{
    if (i >= 0 && i < a.n) return i;
    if (i < 0) {
        if (a.flip_first) flip |= a.flip;
        return a.first < 0 ? -1 : a.first;
    }
    if (a.flip_last) flip |= a.flip;
    return a.last < 0 ? -1 : a.last;
}

__host__ __device__ inline int wrapped(int i, int n)
{
    if (i >= 0 && i < n) return i;
    i %= n;
    return i < 0 ? i + n : i;
}

// Ghost q of the ring around the window: rows -1 and WH (with corners), then
// columns -1 and WW.  False when the side holds no ghost or a wall.
__host__ __device__ inline bool ghost(const Axis& ax, const Axis& ay, int q, int& col, int& row, int& sc, int& sr,
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

// Slot of this thread's entry when `has` is set: entries keep the order of
// the threads; base advances by the block's count.  Every thread calls it.
__device__ inline int block_append(bool has, int& base, int* sums)
{
    const unsigned m = __ballot_sync(0xffffffffu, has);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) sums[w] = __popc(m);
    __syncthreads();
    int before = 0, all = 0;
    for (int k = 0; k < nw; ++k) {
        if (k < w) before += sums[k];
        all += sums[k];
    }
    __syncthreads();
    const int slot = base + before + __popc(m & ((1u << lane) - 1u));
    base += all;
    return slot;
}

}  // namespace window

// The lists of tile items[blockIdx.x] (256 threads; once per handle).  Every
// entry of a list past its last one is a unit without nodes.
template <typename T>
__global__ void __launch_bounds__(256)
window_lists_kernel(const BatchInst<T>* __restrict__ insts, const window::Item* __restrict__ items,
                    const window::Shape sh, window::Head* __restrict__ heads, window::Unit* __restrict__ units,
                    window::Ghost* __restrict__ ghosts, window::Link* __restrict__ links, window::Dir* __restrict__ dirs)
{
    using namespace window;
    constexpr bool F32 = std::is_same<T, float>::value;
    __shared__ int sums[8];
    const int b = blockIdx.x, tid = threadIdx.x;
    const Item it = items[b];
    const BatchInst<T>& in = insts[it.inst];
    const Fields<T>& f = in.f[0];
    const Axis ax = make_axis(it.x0, it.x1, f.nx, f.edge[0], f.edge[1], sh.k, 1);
    const Axis ay = make_axis(it.y0, it.y1, f.ny, f.edge[2], f.edge[3], sh.k, 2);
    const int pw = 2 * sh.hw, shift = F32 ? ax.lo & 1 : 0;
    auto cell_of = [&](int q, int r) { return (r + 1) * pw + q + 2 + shift; };
    auto global_of = [&](int q, int r) {
        return (uint32_t)((size_t)wrapped(ay.lo + r, f.ny) * f.pitch + wrapped(ax.lo + q, f.nx));
    };
    Head& hd = heads[b];
    if (tid == 0) hd.item = it;
    // ---- units
    const int uw = F32 ? (ax.n + shift + 1) / 2 : ax.n, nu = uw * ay.n;
    int base = 0;
    for (int d = 0; d <= sh.k; ++d) {
        for (int u0 = 0; u0 < nu; u0 += 256) {
            const int u = u0 + tid;
            bool has = false;
            Unit e{0, NONE, NONE, 0};
            if (u < nu) {
                const int r = u / uw, j = u - r * uw, dy = ay.dist(r);
                if constexpr (F32) {
                    const int q0 = 2 * j - shift, q1 = q0 + 1;
                    const bool in0 = q0 >= 0, in1 = q1 < ax.n;
                    const int dd = min(in0 ? max(dy, ax.dist(q0)) : MAX_STEPS + 1, in1 ? max(dy, ax.dist(q1)) : MAX_STEPS + 1);
                    if (dd == d) {
                        const uint32_t g0 = in0 ? global_of(q0, r) : NONE, g1 = in1 ? global_of(q1, r) : NONE;
                        const uint32_t t0 = in0 ? f.type[g0] : 0, t1 = in1 ? f.type[g1] : 0;
                        const bool wet0 = (t0 & KIND_MASK) != K_SOLID, wet1 = (t1 & KIND_MASK) != K_SOLID;
                        has = wet0 || wet1;
                        e.g0 = wet0 ? g0 : NONE;
                        e.g1 = wet1 ? g1 : NONE;
                        // fast: kind 1 .. 7 without the bounce-back bit
                        e.half = (uint32_t)((r + 1) * pw + (q0 + 2 + shift) / 2);
                        e.cell = (uint32_t)cell_of(q0, r) | (t0 - 1u < 7u ? U_FAST0 : 0) | (t1 - 1u < 7u ? U_FAST1 : 0) |
                                 ((t0 & KIND_MASK) == K_NOSLIP ? U_NOSLIP0 : 0) |
                                 ((t1 & KIND_MASK) == K_NOSLIP ? U_NOSLIP1 : 0) | (in1 ? U_TWO : 0) |
                                 (wet0 && dy == 0 && ax.dist(q0) == 0 ? U_TILE0 : 0) |
                                 (wet1 && dy == 0 && ax.dist(q1) == 0 ? U_TILE1 : 0) |
                                 (wet0 && wet1 && !(g0 & 1) && g1 == g0 + 1 ? U_VEC : 0);
                    }
                } else {
                    if (max(dy, ax.dist(j)) == d) {
                        const uint32_t g = global_of(j, r);
                        const uint32_t t = f.type[g];
                        has = (t & KIND_MASK) != K_SOLID;
                        e.g0 = g;
                        e.cell = (uint32_t)cell_of(j, r) | ((t & KIND_MASK) == K_NOSLIP ? U_NOSLIP0 : 0) |
                                 (d == 0 ? U_TILE0 : 0);
                        uint32_t mask = 0;
                        if (t & GENERAL_BIT)
                            for (int a = 1; a < 9; ++a) {
                                uint8_t flip = 0;
                                const int sc = resolve(ax, j - c_cx[a], flip), sr = resolve(ay, r - c_cy[a], flip);
                                if (sc < 0 || sr < 0 || (f.type[global_of(sc, sr)] & KIND_MASK) == K_SOLID)
                                    mask |= 1u << (a - 1);
                            }
                        e.g1 = mask;
                    }
                }
            }
            const int slot = block_append(has, base, sums);
            if (has) units[(size_t)b * sh.units + slot] = e;
        }
        if (tid == 0) hd.units[d] = (uint16_t)base;
    }
    for (int k = base + tid; k < sh.units; k += 256) units[(size_t)b * sh.units + k] = Unit{0, NONE, F32 ? NONE : 0u, 0};
    // ---- ghosts, by the distance of their place
    const int nring = 2 * (ax.n + 2) + 2 * ay.n;
    base = 0;
    for (int d = 0; d <= sh.k; ++d) {
        for (int q0 = 0; q0 < nring; q0 += 256) {
            int col, row, sc, sr;
            uint8_t flip;
            const bool has = q0 + tid < nring && ghost(ax, ay, q0 + tid, col, row, sc, sr, flip) &&
                             max(ax.dist(col), ay.dist(row)) == d;
            const int slot = block_append(has, base, sums);
            if (has)
                ghosts[(size_t)b * sh.ghosts + slot] =
                    Ghost{(uint32_t)cell_of(col, row) | (uint32_t)cell_of(sc, sr) << 16, flip};
        }
        if (tid == 0) hd.ghosts[d] = (uint16_t)base;
    }
    // ---- nodes with a bounce-back link (FP32) and Dirichlet nodes
    const int nc = ax.n * ay.n;
    base = 0;
    for (int d = 0; d <= sh.k; ++d) {
        for (int p0 = 0; p0 < nc && F32 && sh.walls > 0; p0 += 256) {
            const int p = p0 + tid, r = p / ax.n, q = p - r * ax.n;
            bool has = p < nc && max(ax.dist(q), ay.dist(r)) == d;
            uint32_t t = 0;
            if (has) t = f.type[global_of(q, r)];
            has = has && (t & GENERAL_BIT);
            const int slot = block_append(has, base, sums);
            if (!has) continue;
            for (int a = 1; a < 9; ++a) {
                uint8_t flip = 0;
                const int sc = resolve(ax, q - c_cx[a], flip), sr = resolve(ay, r - c_cy[a], flip);
                const bool back = sc < 0 || sr < 0 || (f.type[global_of(sc, sr)] & KIND_MASK) == K_SOLID;
                const uint32_t src = back ? (uint32_t)cell_of(q, r) : (uint32_t)cell_of(sc, sr);
                links[((size_t)b * sh.walls + slot) * 8 + a - 1] =
                    Link{src | (back ? 0u : (uint32_t)flip << 16) | (back ? 1u << 18 : 0u) |
                             ((t & KIND_MASK) == K_NOSLIP ? 1u << 19 : 0u),
                         (uint32_t)cell_of(q, r)};
            }
        }
        if (tid == 0) hd.walls[d] = (uint16_t)base;
    }
    base = 0;
    for (int p0 = 0; p0 < nc && sh.dirs > 0; p0 += 256) {
        const int p = p0 + tid, r = p / ax.n, q = p - r * ax.n;
        uint32_t t = 0, g = 0;
        if (p < nc) t = f.type[g = global_of(q, r)];
        const int kind = (int)(t & KIND_MASK);
        const bool has = kind >= K_DIR_H;
        const int slot = block_append(has, base, sums);
        if (!has) continue;
        // the edge a Dirichlet node belongs to: the first of W, E, S, N it touches
        const int gx = wrapped(ax.lo + q, f.nx), gy = wrapped(ay.lo + r, f.ny);
        const int ed = gx == 0 ? 0 : gx == f.nx - 1 ? 1 : gy == 0 ? 2 : 3;
        const int inward = cell_of(q, r) + (ed == 0 ? 1 : ed == 1 ? -1 : ed == 2 ? pw : -pw);
        dirs[(size_t)b * sh.dirs + slot] = Dir{(uint32_t)cell_of(q, r) | (uint32_t)inward << 16, kind | (ed << 4),
                                               max(ax.dist(q), ay.dist(r)), 0, in.D64[g]};
    }
    if (tid == 0) hd.dirs = (uint16_t)base;
}

namespace window {

// Update of a node with a bounce-back link, one link per lane of a group of
// eight (lane & 7 = a - 1): general_node's operations in its order, every
// lane with all sums.
__device__ __forceinline__ void general8(const Arrays<float>& A, const float* raw, const Coef<float>& c, const Link l,
                                         int lane, float& oe, float& ou, float& ov)
{
    using T = float;
    using O = Op<T>;
    const int n = A.n, a = 1 + (lane & 7);
    // c_a: x = +1 for 1 2 8, -1 for 4 5 6; y = +1 for 2 3 4, -1 for 6 7 8
    const int cx = ((0x106 >> a) & 1) - ((0x070 >> a) & 1);
    const int cy = ((0x01C >> a) & 1) - ((0x1C0 >> a) & 1);
    const int x = (int)l.cell, s = (int)(l.src & 0xffffu);
    const bool bounce = (l.src >> 18) & 1u;
    const NodeQ<T> X = node_q_of(c, raw[x], A.D[x], raw[n + x], raw[2 * n + x], 0);
    const NodeQ<T> Y = node_q_of(c, raw[s], A.D[s], raw[n + s], raw[2 * n + s], (uint8_t)((l.src >> 16) & 3u));
    const T lam = (a & 1) ? T(1) : T(0.25);
    const T fx = cx > 0 ? T(1) : cx < 0 ? T(-1) : T(0), fy = cy > 0 ? T(1) : cy < 0 ? T(-1) : T(0);
    T w = feq_diff_dir(c, Y, bounce ? -fx : fx, bounce ? -fy : fy, lam);
    const T bed = O::mul(O::mul(lam, c.G6), O::mul(O::add(X.eta, Y.eta), O::sub(X.D, Y.D)));
    const T frc = O::mul(O::mul(lam, c.KF), O::fma(fx, O::add(X.Fx, Y.Fx), O::mul(fy, O::add(X.Fy, Y.Fy))));
    if (!bounce) w = O::add(O::add(w, bed), frc);
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
    general_finish(c, X, Sh, Sx, Sy, ((l.src >> 19) & 1u) != 0, ou, ov);
    oe = Sh;
}

// dirichlet_value on the window's arrays, in two parts that run side by side
// (0: eta and u, 1: v): its two divisions would be one chain otherwise, and
// with it the longest of a step at the grid's edge (2,800 cycles; 900 now).
template <typename T>
__device__ __forceinline__ void dirichlet_part(T* raw, int n, const T* D, const Dir& d, int part, double h, double q)
{
    const int x = (int)(d.cells & 0xffffu), n1 = (int)(d.cells >> 16), kind = d.meta & 15;
    T* w = raw + (part ? 2 : 1) * n;
    if (kind == K_DIR_H) {
        w[x] = w[n1];
    } else {
        if (kind == K_DIR_Q) h = (double)D[n1] + (double)raw[n1];
        w[x] = (T)(q / h);
    }
    if (!part) raw[x] = (T)(h - d.D64);
}

// A: the derived pair of the padded cell q (an even column; j in the split
// arrays); two: both columns lie in the window.
__device__ __forceinline__ void put_pair(const Arrays<float>& A, int q, int j, bool two, const Src2& s)
{
    const int hw = A.hw, n = A.n;
    const float2 v6[6] = {s.o1, s.o2, s.o4, s.o5, s.o6, s.o8};
#pragma unroll
    for (int d = 0; d < 6; ++d) {
        A.o[d * n + j] = v6[d].x;
        if (two) A.o[d * n + hw + j] = v6[d].y;
    }
    A.ed[j] = make_float2(s.eta.x, s.D.x);
    if (two) {
        A.ed[hw + j] = make_float2(s.eta.y, s.D.y);
        *reinterpret_cast<float2*>(&A.o37[q]) = s.o3;
        *reinterpret_cast<float2*>(&A.o37[n + q]) = s.o7;
    } else {
        A.o37[q] = s.o3.x;
        A.o37[n + q] = s.o7.x;
    }
}
__device__ __forceinline__ void put_one(const Arrays<float>& A, int q, const Src<float>& s)
{
    const int pw = 2 * A.hw, row = q / pw * pw, pc = q - row, n = A.n, j = row + (pc & 1) * A.hw + (pc >> 1);
    const float v6[6] = {s.o1, s.o2, s.o4, s.o5, s.o6, s.o8};
#pragma unroll
    for (int d = 0; d < 6; ++d) A.o[d * n + j] = v6[d];
    A.ed[j] = make_float2(s.eta, s.D);
    A.o37[q] = s.o3;
    A.o37[n + q] = s.o7;
}
__device__ __forceinline__ void put_one(const Arrays<double>& A, int q, const Src<double>& s)
{
    const int n = A.n;
    const double v8[8] = {s.o1, s.o2, s.o3, s.o4, s.o5, s.o6, s.o7, s.o8};
#pragma unroll
    for (int d = 0; d < 8; ++d) A.o[d * n + q] = v8[d];
    A.own[q] = s.ownh;
    A.own[n + q] = s.hFx;
    A.own[2 * n + q] = s.hFy;
}

}  // namespace window

// Block b takes `steps` steps (1 .. shape.k) of tile b of the lists.  NP
// (FP32): pairs per thread, enough for the longest list.  tab: boundary
// values of each step, or (steady) the instance's own.  active: batch flags
// or nullptr.
template <typename T, int FM, int NP>
__global__ void __launch_bounds__(window::MAX_THREADS, 1)
step_window_kernel(const BatchInst<T>* __restrict__ insts, const __grid_constant__ window::Lists lists,
                   const uint8_t* __restrict__ active, const __grid_constant__ window::Buffers<T> buf,
                   const __grid_constant__ window::Shape shape, int steps, int steady,
                   const __grid_constant__ window::DirTable tab)
{
    using namespace window;
    constexpr bool F32 = std::is_same<T, float>::value;
    extern __shared__ __align__(16) unsigned char window_smem[];
    __shared__ Head hd;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const Arrays<T> A = carve<T>(window_smem, shape);
    const int pw = 2 * A.hw, n = A.n;
    const Unit* units = lists.units + (size_t)blockIdx.x * shape.units;
    // the tile's static data: everything here may run before the launch
    // before this one has finished
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    Unit un[NP];
    if constexpr (F32) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const uint4 q = *reinterpret_cast<const uint4*>(units + tid + k * nt);
            un[k] = Unit{q.x, q.y, q.z, q.w};
        }
    }
    for (int k = tid; k < (int)(sizeof(Head) / 4); k += nt)
        reinterpret_cast<uint32_t*>(&hd)[k] = reinterpret_cast<const uint32_t*>(lists.head + blockIdx.x)[k];
    __syncthreads();
    const BatchInst<T>& in = insts[hd.item.inst];
    const Coef<T> c = in.f[0].c;
    const long long off = hd.item.off;
    const T* Dg = buf.D + off;
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
    if (active && !active[hd.item.inst]) return;  // whole block
    // ---- load the window
    Src2 own[NP];
    const T *e_in = buf.in[0] + off, *u_in = buf.in[1] + off, *v_in = buf.in[2] + off;
    if constexpr (F32) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const int q = (int)(un[k].cell & 0xffffu);
            float2 e{}, u{}, v{}, d{};
            if (un[k].cell & U_VEC) {
                e = *reinterpret_cast<const float2*>(e_in + un[k].g0);
                u = *reinterpret_cast<const float2*>(u_in + un[k].g0);
                v = *reinterpret_cast<const float2*>(v_in + un[k].g0);
                d = *reinterpret_cast<const float2*>(Dg + un[k].g0);
            } else {
                if (un[k].g0 != NONE)
                    e.x = e_in[un[k].g0], u.x = u_in[un[k].g0], v.x = v_in[un[k].g0], d.x = Dg[un[k].g0];
                if (un[k].g1 != NONE)
                    e.y = e_in[un[k].g1], u.y = u_in[un[k].g1], v.y = v_in[un[k].g1], d.y = Dg[un[k].g1];
            }
            if (q == 0) continue;  // past the list
            *reinterpret_cast<float2*>(A.raws + q) = e;
            *reinterpret_cast<float2*>(A.raws + n + q) = u;
            *reinterpret_cast<float2*>(A.raws + 2 * n + q) = v;
            *reinterpret_cast<float2*>(A.D + q) = d;
        }
    } else {
        const int total = hd.units[steps];
        const T* bg = buf.bed + off;
        for (int p = tid; p < total; p += nt) {
            const uint32_t g = units[p].g0;
            const int q = (int)(units[p].cell & 0xffffu);
            const T e = e_in[g], u = u_in[g], v = v_in[g], d = Dg[g], b0 = bg[g], b1 = bg[g + buf.plane],
                    b2 = bg[g + 2 * buf.plane];
            A.raws[q] = e;
            A.raws[n + q] = u;
            A.raws[2 * n + q] = v;
            A.D[q] = d;
            A.bed[q] = b0;
            A.bed[n + q] = b1;
            A.bed[2 * n + q] = b2;
        }
    }
    const Coef2 c2 = march::pairs_of(c);
    const int nd = hd.dirs;
    const Ghost* gl = lists.ghosts + (size_t)blockIdx.x * shape.ghosts;
    const Link* ll = lists.links + (size_t)blockIdx.x * shape.walls * 8;
    const Dir* dl = lists.dirs + (size_t)blockIdx.x * shape.dirs;
    // Dirichlet nodes: two lanes each (eta and u; v), the first round's entry
    // and steady values in registers
    const int part = tid & 1;
    Dir mine{};
    double bh = 0.0, bq = 0.0;
    if (tid >> 1 < nd) {
        mine = dl[tid >> 1];
        if (steady) {
            bh = in.bv.h[mine.meta >> 4];
            bq = part ? in.bv.qy[mine.meta >> 4] : in.bv.qx[mine.meta >> 4];
        }
    }
    __syncthreads();
    for (int s = 0; s < steps; ++s) {
        const int m = steps - s;  // steps still to take, this one included
        T* raw = A.raw(s & 1);
        T* nxt = A.raw(1 - (s & 1));
        // ---- A: source quantities of the region and its ghosts
        const int na = hd.units[m];
        if constexpr (F32) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                if (tid + k * nt >= na) break;
                const int q = (int)(un[k].cell & 0xffffu);
                const float2 e = *reinterpret_cast<const float2*>(raw + q), u = *reinterpret_cast<const float2*>(raw + n + q);
                const float2 v = *reinterpret_cast<const float2*>(raw + 2 * n + q);
                const float2 d = *reinterpret_cast<const float2*>(A.D + q);
                derive2<FM>(c2, Raw<float>{e.x, u.x, v.x, d.x, 0}, Raw<float>{e.y, u.y, v.y, d.y, 0}, own[k]);
                put_pair(A, q, (int)un[k].half, (un[k].cell & U_TWO) != 0, own[k]);
            }
            // ghosts on the block's last warps, whose pairs drop out first
            for (int g = nt - 1 - tid; g < (int)hd.ghosts[m]; g += nt) {
                const Ghost gh = gl[g];
                const int to = (int)(gh.cells & 0xffffu), q = (int)(gh.cells >> 16);
                Src<T> src;
                derive<T, FM>(c, Raw<T>{raw[q], raw[n + q], raw[2 * n + q], A.D[q], (uint8_t)gh.flip}, src);
                put_one(A, to, src);
            }
        } else {
            // nodes, then ghosts: one list, so that no warp takes two rounds
            // of FP64 instructions while another has none
            for (int p = tid; p < na + (int)hd.ghosts[m]; p += nt) {
                int q, to;
                uint8_t flip = 0;
                if (p < na) {
                    q = to = (int)(units[p].cell & 0xffffu);
                } else {
                    const Ghost gh = gl[p - na];
                    to = (int)(gh.cells & 0xffffu);
                    q = (int)(gh.cells >> 16);
                    flip = (uint8_t)gh.flip;
                }
                Src<T> src;
                derive<T, FM>(c, Raw<T>{raw[q], raw[n + q], raw[2 * n + q], A.D[q], flip}, src);
                put_one(A, to, src);
                if (to != q) raw[to] = src.eta;  // the stencils of eta read it
            }
        }
        __syncthreads();
        // ---- B: update
        const int nb = hd.units[m - 1];
        if constexpr (F32) {
#pragma unroll
            for (int k = 0; k < NP; ++k) {
                if (tid + k * nt >= nb) break;
                if (!(un[k].cell & (U_FAST0 | U_FAST1))) continue;
                const int hw = A.hw, q = (int)(un[k].cell & 0xffffu);
                // rows above, own, below; even columns first, odd columns hw on
                const int rc = (int)un[k].half, rm = rc - pw, rp = rc + pw;
                const float *o1 = A.o, *o2 = A.o + n, *o4 = A.o + 2 * n, *o5 = A.o + 3 * n, *o6 = A.o + 4 * n,
                            *o8 = A.o + 5 * n;
                const float2 m4[4] = {A.ed[rm + hw - 1], A.ed[rm], A.ed[rm + hw], A.ed[rm + 1]};
                // (the second column of an odd window's last pair is a ghost, or out of date)
                const float2 c4[4] = {A.ed[rc + hw - 1], make_float2(own[k].eta.x, own[k].D.x),
                                      (un[k].cell & U_TWO) ? make_float2(own[k].eta.y, own[k].D.y) : A.ed[rc + hw],
                                      A.ed[rc + 1]};
                const float2 p4[4] = {A.ed[rp + hw - 1], A.ed[rp], A.ed[rp + hw], A.ed[rp + 1]};
                float2 oe, ou, ov;
                march::gather_pair(c2, make_float2(o1[rc + hw - 1], o1[rc]), make_float2(o2[rm + hw - 1], o2[rm]),
                                   make_float2(o5[rc + hw], o5[rc + 1]), make_float2(o4[rm + hw], o4[rm + 1]),
                                   *reinterpret_cast<const float2*>(A.o37 + q - pw),
                                   make_float2(o8[rp + hw - 1], o8[rp]), make_float2(o6[rp + hw], o6[rp + 1]),
                                   *reinterpret_cast<const float2*>(A.o37 + n + q + pw), m4, c4, p4, own[k].ownh,
                                   own[k].hFx, own[k].hFy, (un[k].cell & U_NOSLIP0) != 0, (un[k].cell & U_NOSLIP1) != 0,
                                   oe, ou, ov);
                if ((un[k].cell & (U_FAST0 | U_FAST1)) == (U_FAST0 | U_FAST1)) {
                    *reinterpret_cast<float2*>(nxt + q) = oe;
                    *reinterpret_cast<float2*>(nxt + n + q) = ou;
                    *reinterpret_cast<float2*>(nxt + 2 * n + q) = ov;
                } else {
                    const bool hi = (un[k].cell & U_FAST1) != 0;
                    nxt[q + (hi ? 1 : 0)] = hi ? oe.y : oe.x;
                    nxt[n + q + (hi ? 1 : 0)] = hi ? ou.y : ou.x;
                    nxt[2 * n + q + (hi ? 1 : 0)] = hi ? ov.y : ov.x;
                }
            }
            // eight lanes per node, the block's last warps first (their pairs
            // lie farthest from the tile and drop out as the region shrinks)
            const int nw = hd.walls[m - 1];
            for (int g = (nt - 1 - tid) >> 3; g < nw; g += nt >> 3) {
                const Link l = ll[g * 8 + (lane & 7)];
                T oe, ou, ov;
                general8(A, raw, c, l, lane, oe, ou, ov);
                if ((lane & 7) == 0) {
                    nxt[l.cell] = oe;
                    nxt[n + l.cell] = ou;
                    nxt[2 * n + l.cell] = ov;
                }
            }
        } else {
            for (int p = tid; p < nb; p += nt) {
                const uint32_t code = units[p].cell, mask = units[p].g1;
                const int q = (int)(code & 0xffffu);
                // where each link reads: the neighbour, or for a bounced link
                // the node itself, opposite direction
                const int nbr[8] = {q - 1, q - pw - 1, q - pw, q - pw + 1, q + 1, q + pw + 1, q + pw, q + pw - 1};
                T o[8], eta[8];
#pragma unroll
                for (int a = 0; a < 8; ++a) {
                    const bool back = (mask >> a) & 1u;
                    o[a] = A.o[back ? ((a + 4) & 7) * n + q : a * n + nbr[a]];
                    eta[a] = raw[back ? q : nbr[a]];
                }
                T oe, ou, ov;
                update64(c, o[0], o[1], o[7], o[4], o[3], o[5], o[2], o[6],
                         Eta8{eta[1], eta[2], eta[3], eta[0], eta[4], eta[7], eta[6], eta[5]}, raw[q], A.D[q], A.own[q],
                         A.own[n + q], A.own[2 * n + q], Bed64{A.bed[q], A.bed[n + q], A.bed[2 * n + q]},
                         (code & U_NOSLIP0) != 0, oe, ou, ov);
                nxt[q] = oe;
                nxt[n + q] = ou;
                nxt[2 * n + q] = ov;
            }
        }
        __syncthreads();
        // ---- C: Dirichlet nodes
        if (nd > 0) {
            for (int k = tid >> 1; k < nd; k += nt >> 1) {
                const bool first = k == tid >> 1;
                const Dir d = first ? mine : dl[k];
                if (d.dist > m - 1) continue;
                const int ed = d.meta >> 4;
                double h = bh, q = bq;
                if (!steady || !first) {
                    const DirValues& bv = steady ? in.bv : tab.v[s];
                    h = bv.h[ed];
                    q = part ? bv.qy[ed] : bv.qx[ed];
                }
                dirichlet_part(nxt, n, A.D, d, part, h, q);
            }
            __syncthreads();
        }
    }
    // ---- store the tile
    const T *last = A.raw(steps & 1), *before = A.raw(1 - (steps & 1));
    T *o_e = buf.out[0] + off, *o_u = buf.out[1] + off, *o_v = buf.out[2] + off;
    const int nst = hd.units[0];
    auto store = [&](const T* from, T* e, T* u, T* v, uint32_t code, uint32_t g0, uint32_t g1) {
        const int q = (int)(code & 0xffffu);
        if constexpr (F32) {
            if ((code & U_VEC) && (code & U_TILE0) && (code & U_TILE1)) {
                *reinterpret_cast<float2*>(e + g0) = *reinterpret_cast<const float2*>(from + q);
                *reinterpret_cast<float2*>(u + g0) = *reinterpret_cast<const float2*>(from + n + q);
                *reinterpret_cast<float2*>(v + g0) = *reinterpret_cast<const float2*>(from + 2 * n + q);
                return;
            }
            if (code & U_TILE1) e[g1] = from[q + 1], u[g1] = from[n + q + 1], v[g1] = from[2 * n + q + 1];
        }
        if (code & U_TILE0) e[g0] = from[q], u[g0] = from[n + q], v[g0] = from[2 * n + q];
    };
    if constexpr (F32) {
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            if (tid + k * nt >= nst) break;
            store(last, o_e, o_u, o_v, un[k].cell, un[k].g0, un[k].g1);
            if (buf.prev[0])
                store(before, buf.prev[0] + off, buf.prev[1] + off, buf.prev[2] + off, un[k].cell, un[k].g0, un[k].g1);
        }
    } else {
        for (int p = tid; p < nst; p += nt) {
            const Unit e = units[p];
            store(last, o_e, o_u, o_v, e.cell, e.g0, 0);
            if (buf.prev[0]) store(before, buf.prev[0] + off, buf.prev[1] + off, buf.prev[2] + off, e.cell, e.g0, 0);
        }
    }
}

}  // namespace maclab
