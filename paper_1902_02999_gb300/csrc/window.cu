// window.cu -- planning and launching of the several-steps-per-launch kernel
// (maclab_window.cuh).
#include "window.h"

#include <algorithm>
#include <cmath>

namespace maclab {
namespace window {
namespace {

constexpr size_t MAX_SMEM = 227 * 1024 - 2048;

// Cost model in SM cycles, fitted to clock readings inside the kernel and to
// whole runs on a GB300 (2.07 GHz): 256 x 256 lake, 1001 x 333 channel,
// 400 x 3 strip.
constexpr double LAUNCH_CYCLES = 4000;  // launch
constexpr double BLOCK_CYCLES = 4500;   // a block's dependent loads and its store
constexpr double LOAD_CELL = 1.5;       // per window node
constexpr double STEP_CYCLES = 100;     // barriers of a step
// FP32: a round of a block's threads (a pair each, derived and updated) takes
// its latency, and each warp its issue slots
constexpr double ROUND_F32 = 900, WARP_F32 = 100;
// FP64: a warp instruction takes 66 cycles of an SM quarter and 19 of the SM
constexpr double DERIVE_F64 = 40, UPDATE_F64 = 46;

double f32_cycles(double pairs, int threads, double shared)
{
    return STEP_CYCLES + 0.5 * (ROUND_F32 * std::ceil(pairs / threads) + WARP_F32 * shared * std::ceil(pairs / 32));
}
double f64_cycles(double nodes, double instructions, double shared)
{
    const double warps = shared * std::ceil(nodes / 32);
    return STEP_CYCLES + instructions * std::max(66.0 * std::ceil(warps / 4), 19.0 * warps);
}

// tiles across an axis of n nodes for tiles of at most t; a tile that does
// not span the axis has two nodes at least
int tiles(int n, int t) { return std::max(1, std::min((n + t - 1) / t, std::max(1, n / 2))); }
int cut(int n, int nt, int i) { return (int)((int64_t)n * i / nt); }

// nodes that are not solid in [0, x) x [0, y), row length nx + 1 (empty when
// no node is solid)
struct Counts {
    std::vector<int> c;
    int w;
    explicit Counts(const GridView& g) : w(g.nx + 1)
    {
        bool dry = false;
        for (int y = 0; y < g.ny && !dry; ++y) {
            const uint8_t* t = g.type + (size_t)y * g.pitch;
            uint8_t solid = 0;
            for (int x = 0; x < g.nx; ++x) solid |= (t[x] & KIND_MASK) == K_SOLID;
            dry = solid;
        }
        if (!dry) return;
        c.assign((size_t)(g.nx + 1) * (g.ny + 1), 0);
        for (int y = 0; y < g.ny; ++y) {
            int run = 0;
            for (int x = 0; x < g.nx; ++x) {
                run += (g.type[(size_t)y * g.pitch + x] & KIND_MASK) != K_SOLID;
                c[(size_t)(y + 1) * w + x + 1] = c[(size_t)y * w + x + 1] + run;
            }
        }
    }
    // tiles that hold a node that is not solid (cx: scratch)
    int tiles_with_nodes(const GridView& g, int ntx, int nty, std::vector<int>& cx) const
    {
        if (c.empty()) return ntx * nty;
        cx.resize(ntx + 1);
        for (int a = 0; a <= ntx; ++a) cx[a] = cut(g.nx, ntx, a);
        int n = 0;
        for (int b = 0; b < nty; ++b) {
            const int* r0 = &c[(size_t)cut(g.ny, nty, b) * w];
            const int* r1 = &c[(size_t)cut(g.ny, nty, b + 1) * w];
            int before = r1[0] - r0[0];
            for (int a = 1; a <= ntx; ++a) {
                const int upto = r1[cx[a]] - r0[cx[a]];
                n += upto > before;
                before = upto;
            }
        }
        return n;
    }
    int operator()(int x0, int x1, int y0, int y1) const
    {
        if (c.empty()) return (x1 - x0) * (y1 - y0);
        return c[(size_t)y1 * w + x1] - c[(size_t)y0 * w + x1] - c[(size_t)y1 * w + x0] + c[(size_t)y0 * w + x0];
    }
};

// The most nodes with a bounce-back link in the window of any of a grid's nt
// tiles (nodes that windows wrap onto more than once count each time).
int most_walls(const GridView& g, int ntx, int nty, int k)
{
    // per column and row: the tiles whose windows hold it (once per hold)
    struct Holders {
        std::vector<int> start, tile;
        Holders(int n, int nt, int lo_kind, int hi_kind, int halo) : start(n + 2, 0)
        {
            for (int pass = 0; pass < 2; ++pass) {
                for (int t = 0; t < nt; ++t) {
                    const Axis a = make_axis(cut(n, nt, t), cut(n, nt, t + 1), n, lo_kind, hi_kind, halo, 1);
                    int x = wrapped(a.lo, n);
                    for (int i = 0; i < a.n; ++i, x = x + 1 == n ? 0 : x + 1) {
                        if (pass == 0) ++start[x + 2];
                        else tile[start[x + 1]++] = t;
                    }
                }
                if (pass == 0) {
                    for (int x = 0; x < n; ++x) start[x + 2] += start[x + 1];
                    tile.resize(start[n + 1]);
                }
            }
        }
    };
    const Holders cols(g.nx, ntx, g.edge[0], g.edge[1], k), rows(g.ny, nty, g.edge[2], g.edge[3], k);
    std::vector<int> count((size_t)ntx * nty, 0);
    for (int w = 0; w < g.walls; ++w) {
        const int y = g.wall[w] / g.nx, x = g.wall[w] - y * g.nx;
        for (int j = rows.start[y]; j < rows.start[y + 1]; ++j)
            for (int i = cols.start[x]; i < cols.start[x + 1]; ++i) ++count[(size_t)rows.tile[j] * ntx + cols.tile[i]];
    }
    return *std::max_element(count.begin(), count.end());
}

}  // namespace

Plan make_plan(const std::vector<GridView>& grids, bool batch, bool f64, int fmode, int sms)
{
    Plan best;
    int64_t nodes = 0;
    bool dirichlet = false;
    for (const GridView& g : grids) {
        nodes += (int64_t)g.nx * g.ny;
        for (int y = 0; y < g.ny; ++y)
            for (int x = 0; x < g.nx; ++x) {
                if (y > 0 && y < g.ny - 1 && x > 0 && x < g.nx - 1) {
                    x = g.nx - 2;  // Dirichlet nodes lie on the grid's edges
                    continue;
                }
                if ((g.type[(size_t)y * g.pitch + x] & KIND_MASK) < K_DIR_H) continue;
                dirichlet = true;
                const int ed = x == 0 ? 0 : x == g.nx - 1 ? 1 : y == 0 ? 2 : 3;
                if (g.edge[ed] == EDGE_PER) return best;  // its inward node may lie outside a window
            }
    }
    // (above this the single-step kernels win whatever the tiles)
    if (nodes > (int64_t)640 << 10) return best;
    std::vector<Counts> counts;
    counts.reserve(grids.size());
    bool dry = false;
    for (const GridView& g : grids) {
        counts.emplace_back(g);
        dry = dry || !counts.back().c.empty();
    }
    // without dry nodes to leave out, FP64 gains only where the tile kernel
    // leaves SMs idle
    if (f64 && !dry && nodes > (int64_t)140 << 10) return best;
    static const int TW[] = {4, 8, 12, 16, 24, 32, 40, 48, 64};
    static const int TH[] = {2, 4, 8, 12, 16, 24, 32, 48};
    static const int KS[] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 16};
    const size_t per_cell = f64 ? cell_bytes<double>() : cell_bytes<float>();
    std::vector<int> cx;
    double best_cost = 1e300, one_step = 0;
    int btw = 0, bth = 0;
    for (int tw : TW)
        for (int th : TH) {
            int64_t upper = 0;
            for (const GridView& g : grids) upper += (int64_t)tiles(g.nx, tw) * tiles(g.ny, th);
            if (upper > (f64 ? 16 : 4) * (int64_t)sms) continue;
            int64_t wet = 0;
            int mw = 0, mh = 0;
            for (size_t i = 0; i < grids.size(); ++i) {
                const GridView& g = grids[i];
                const int ntx = tiles(g.nx, tw), nty = tiles(g.ny, th);
                wet += counts[i].tiles_with_nodes(g, ntx, nty, cx);
                mw = std::max(mw, (g.nx + ntx - 1) / ntx);
                mh = std::max(mh, (g.ny + nty - 1) / nty);
            }
            if (wet == 0) continue;
            // no k can take less than a step of the bare tiles each step
            const double bare = (double)((wet + sms - 1) / sms) *
                                (f64 ? 2 * STEP_CYCLES + 19.0 * (DERIVE_F64 + UPDATE_F64) * mw * mh / 32
                                     : 2 * STEP_CYCLES + WARP_F32 * mw * mh / 64);
            if (bare >= best_cost) continue;
            for (int k : KS) {
                if (bare + (LAUNCH_CYCLES + BLOCK_CYCLES) / k >= best_cost) continue;
                // the largest window over the grids
                int ww = 0, wh = 0;
                for (const GridView& g : grids) {
                    const bool fx = tiles(g.nx, tw) == 1, fy = tiles(g.ny, th) == 1;
                    const bool px = g.edge[0] == EDGE_PER && !fx, py = g.edge[2] == EDGE_PER && !fy;
                    ww = std::max(ww, px ? mw + 2 * k : std::min(g.nx, mw + 2 * k));
                    wh = std::max(wh, py ? mh + 2 * k : std::min(g.ny, mh + 2 * k));
                }
                Shape s;
                s.k = k;
                s.hw = (ww + 6) / 2;
                s.rows = wh + 2;
                s.ghosts = 2 * (ww + 2) + 2 * wh;
                s.dirs = dirichlet ? 2 * (ww + wh) : 0;
                const size_t smem = s.cells() * per_cell;
                if (smem > MAX_SMEM) continue;
                int np = 1, threads;
                if (f64) {
                    // (eight warps keep the FP64 pipes busy)
                    threads = std::min(256, (ww * wh + s.ghosts + 31) / 32 * 32);
                    s.units = ww * wh;
                } else {
                    const int pairs = wh * ((ww + 2) / 2);
                    np = (pairs + MAX_THREADS - 1) / MAX_THREADS;
                    if (np > MAX_PAIRS) continue;
                    threads = ((pairs + np - 1) / np + 31) / 32 * 32;
                    s.units = np * threads;
                }
                // blocks of one wave that share an SM (by shared memory and
                // registers), and waves
                const int fit = std::max(1, std::min((int)(MAX_SMEM / smem), 65536 / (128 * threads)));
                const int64_t per_sm = (wet + sms - 1) / sms;
                const double waves = (double)((per_sm + fit - 1) / fit), shared = (double)std::min<int64_t>(per_sm, fit);
                // with several blocks on an SM one block's loads hide behind another's steps
                auto whole = [&](double c) {
                    return LAUNCH_CYCLES + (fit > 1 ? BLOCK_CYCLES + waves * c : waves * (BLOCK_CYCLES + c));
                };
                double cyc = LOAD_CELL * ww * wh * shared, first = 0;  // first: with the last step alone
                const double ghosts = (mw >= ww ? 2.0 * wh : 0) + (mh >= wh ? 2.0 * ww : 0);
                for (int m = k; m >= 1 && whole(cyc) < best_cost * k; --m) {
                    // nodes derived and updated with m steps to take
                    const double da = std::min(ww, mw + 2 * m) * (double)std::min(wh, mh + 2 * m);
                    const double db = std::min(ww, mw + 2 * m - 2) * (double)std::min(wh, mh + 2 * m - 2);
                    const double step = f64 ? f64_cycles(da + ghosts, DERIVE_F64, shared) + f64_cycles(db, UPDATE_F64, shared)
                                            : f32_cycles(0.5 * da, threads, shared) + f32_cycles(0.5 * db, threads, shared);
                    if (m == 1) first = LOAD_CELL * ww * wh * shared + step;
                    cyc += step;
                }
                const double cost = whole(cyc) / k;
                if (cost < best_cost) {
                    best_cost = cost;
                    one_step = whole(first);
                    best.k = k;
                    best.np = np;
                    best.threads = threads;
                    best.smem = smem;
                    best.shape = s;
                    btw = tw;
                    bth = th;
                }
            }
        }
    // against one launch per step (us, measured on a GB300): an FP32 handle's
    // row march, 9.9 us at 512 x 256 nodes, 10.9 at 512 x 512, 13.6 at 1024 x
    // 1024; an FP32 batch's tile kernel (below the node limit above the row
    // march is the slower one); the FP64 tile kernel, 29 us for every full
    // round of the chip's SMs (31 at 512 x 256, 58 at 512 x 512).  The model
    // counts a batch's many waves of blocks up to 1.4 times too dear: of 42
    // batches up to 640 k nodes this path was the faster one on all where it
    // came to less than 1.15 of the tile kernel, but for 97 of 64 x 48 (5.5
    // against 4.4 us).
    double tiles64 = 0, links = 0, fixed = 0;
    for (const GridView& g : grids) {
        tiles64 += (double)((g.nx + tile::TX - 1) / tile::TX) * ((g.ny + tile::TY - 1) / tile::TY);
        links += g.walls;
        fixed += g.dirichlet;
    }
    const double single = f64 ? 29.0 * std::max(1.0, std::ceil(tiles64 / sms))
                              : batch ? batch_tile_us(tiles64, links, fixed) : 9.5 + nodes / 220e3;
    if (best.k == 0 || best_cost / 2070.0 > (batch && !f64 ? 1.15 : 0.9) * single) return Plan();
    // A launch costs its loads and stores however few steps it takes, and a
    // call of a few steps has no graph replay: two us more for each single-step
    // launch, and up to five where a handle's row march has wall links (700 x 700
    // nodes: 12.5 without, 20.1 with walls around).  The fewest steps that this
    // path takes in less (0.9: the model counts a one-step launch a tenth too
    // dear or more).  One step: 809 x 809 nodes 16.3 us here, 13.0 on the row
    // march; four 256 x 256 grids 8.8, tiles 6.7; 600 x 600 12.4 both; 700 x 700
    // with walls 15.5 here.
    const double alone = single + 2.0 + (!f64 && !batch && links > 0 ? 0.5 + std::min(4.5, links / 500) : 0.0);
    const double more = best.k > 1 ? (best_cost * best.k - one_step) / (best.k - 1) : one_step;
    for (; best.min_steps < 64; ++best.min_steps) {
        const int64_t n = best.min_steps, l = launches(n, best.k);
        if (0.9 * (l * one_step + (n - l) * more) / 2070.0 <= n * alone) break;
    }
    best.fm = (fmode & F_CORIOLIS) ? 7 : (fmode & F_FRICTION) ? 3 : 1;
    for (size_t i = 0; i < grids.size(); ++i) {
        const GridView& g = grids[i];
        const int ntx = tiles(g.nx, btw), nty = tiles(g.ny, bth);
        if (!f64 && g.walls > 0) best.shape.walls = std::max(best.shape.walls, most_walls(g, ntx, nty, best.k));
        for (int b = 0; b < nty; ++b)
            for (int a = 0; a < ntx; ++a) {
                Item it{(int)i, cut(g.nx, ntx, a), cut(g.nx, ntx, a + 1), cut(g.ny, nty, b), cut(g.ny, nty, b + 1), 0, g.off};
                if (counts[i](it.x0, it.x1, it.y0, it.y1) > 0) best.items.push_back(it);
            }
    }
    // At most one tile per SM: ask for more than half an SM's shared memory.
    // Launches overlap at their ends, and without this the early blocks of the
    // next one pair up on some SMs while others idle (400 x 3 strip FP64, 4 x 3
    // tiles: 5.9 us per step, 3.3 with it).
    if ((int)best.items.size() <= sms) best.smem = std::max(best.smem, MAX_SMEM / 2 + 1024);
    return best;
}

namespace {
// fm 1: wind (a zero wind adds exact zeros), 3: and friction, 7: and Coriolis
template <typename T, typename F>
cudaError_t with_kernel(const Plan& p, F&& f)
{
#define MACLAB_W(FMV, NPV) \
    if (p.fm == FMV && p.np == NPV) return f((const void*)step_window_kernel<T, FMV, NPV>);
    MACLAB_W(1, 1) MACLAB_W(3, 1) MACLAB_W(7, 1)
    if constexpr (std::is_same<T, float>::value) {
        MACLAB_W(1, 2) MACLAB_W(3, 2) MACLAB_W(7, 2) MACLAB_W(1, 3) MACLAB_W(3, 3) MACLAB_W(7, 3) MACLAB_W(1, 4) MACLAB_W(3, 4) MACLAB_W(7, 4)
    }
#undef MACLAB_W
    return cudaErrorInvalidValue;
}
}  // namespace

namespace {
size_t up(size_t b) { return (b + 255) & ~size_t(255); }
}  // namespace

size_t list_bytes(const Plan& p)
{
    const size_t n = p.items.size();
    return up(n * sizeof(Item)) + up(n * sizeof(Head)) + up(n * p.shape.units * sizeof(Unit)) +
           up(n * p.shape.ghosts * sizeof(Ghost)) + up(n * p.shape.walls * 8 * sizeof(Link)) +
           up(n * p.shape.dirs * sizeof(Dir));
}

template <typename T>
cudaError_t build_lists(const Plan& p, const void* insts, void* mem, cudaStream_t stream, Lists* out)
{
    const size_t n = p.items.size();
    unsigned char* q = (unsigned char*)mem;
    auto take = [&](size_t bytes) {
        void* r = q;
        q += up(bytes);
        return r;
    };
    Item* items = (Item*)take(n * sizeof(Item));
    Head* head = (Head*)take(n * sizeof(Head));
    Unit* units = (Unit*)take(n * p.shape.units * sizeof(Unit));
    Ghost* ghosts = (Ghost*)take(n * p.shape.ghosts * sizeof(Ghost));
    Link* links = (Link*)take(n * p.shape.walls * 8 * sizeof(Link));
    Dir* dirs = (Dir*)take(n * p.shape.dirs * sizeof(Dir));
    *out = Lists{head, units, ghosts, links, dirs};
    cudaError_t e = cudaMemcpyAsync(items, p.items.data(), n * sizeof(Item), cudaMemcpyHostToDevice, stream);
    // the kernels are shared by every handle: opt in to the most any plan takes
    if (e == cudaSuccess)
        e = with_kernel<T>(p, [](const void* k) {
            return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MAX_SMEM);
        });
    if (e != cudaSuccess) return e;
    window_lists_kernel<T><<<(unsigned)n, 256, 0, stream>>>((const BatchInst<T>*)insts, items, p.shape, head, units, ghosts,
                                                            links, dirs);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch(const Plan& p, const void* insts, const Lists& lists, const uint8_t* active, const Buffers<T>& buf,
                   int steps, const DirTable* tab, cudaStream_t stream)
{
    static const DirTable none{};
    int steady = tab ? 0 : 1;
    void* args[] = {(void*)&insts, (void*)&lists, (void*)&active, (void*)&buf, (void*)&p.shape,
                    (void*)&steps, (void*)&steady, (void*)(tab ? tab : &none)};
    // a launch may begin loading its static data while the one before it ends
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)p.items.size());
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = p.smem;
    cfg.stream = stream;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return with_kernel<T>(p, [&](const void* k) { return cudaLaunchKernelExC(&cfg, k, args); });
}
template cudaError_t build_lists<float>(const Plan&, const void*, void*, cudaStream_t, Lists*);
template cudaError_t build_lists<double>(const Plan&, const void*, void*, cudaStream_t, Lists*);
template cudaError_t launch<float>(const Plan&, const void*, const Lists&, const uint8_t*, const Buffers<float>&, int,
                                   const DirTable*, cudaStream_t);
template cudaError_t launch<double>(const Plan&, const void*, const Lists&, const uint8_t*, const Buffers<double>&, int,
                                    const DirTable*, cudaStream_t);

}  // namespace window
}  // namespace maclab
