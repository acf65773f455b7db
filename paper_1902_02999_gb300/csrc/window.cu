// window.cu -- planning and launching of the several-steps-per-launch kernel
// (maclab_window.cuh).
#include "window.h"

#include <algorithm>
#include <cstring>

namespace maclab {
namespace window {
namespace {

#ifndef MACLAB_WINDOW_K
#define MACLAB_WINDOW_K 0  // tuning builds: force the steps per launch
#endif

constexpr size_t MAX_SMEM = 227 * 1024 - 2048;

// Cost model in SM cycles.
constexpr double LAUNCH_CYCLES = 5000;      // launch, dependent loads, store
constexpr double LOAD_CELL = 1.0;           // per window node loaded
constexpr double STEP_CYCLES = 500;         // barriers and the latency of one step
constexpr double CELL_F32 = 1.1;            // per node and step
constexpr double INSTR_F64 = 86;            // FP64 instructions per node and step

// nodes that are not solid in [0, x) x [0, y), row length nx + 1
struct Counts {
    std::vector<int> c;
    int w;
    explicit Counts(const GridView& g) : c((size_t)(g.nx + 1) * (g.ny + 1), 0), w(g.nx + 1)
    {
        for (int y = 0; y < g.ny; ++y) {
            int run = 0;
            for (int x = 0; x < g.nx; ++x) {
                run += (g.type[(size_t)y * g.pitch + x] & KIND_MASK) != K_SOLID;
                c[(size_t)(y + 1) * w + x + 1] = c[(size_t)y * w + x + 1] + run;
            }
        }
    }
    int operator()(int x0, int x1, int y0, int y1) const
    {
        return c[(size_t)y1 * w + x1] - c[(size_t)y0 * w + x1] - c[(size_t)y1 * w + x0] + c[(size_t)y0 * w + x0];
    }
};

// tiles across an axis of n nodes for tiles of at most t; a tile that does
// not span the axis has two nodes at least
int tiles(int n, int t) { return std::max(1, std::min((n + t - 1) / t, std::max(1, n / 2))); }
int cut(int n, int nt, int i) { return (int)((int64_t)n * i / nt); }

}  // namespace

Plan make_plan(const std::vector<GridView>& grids, bool f64, int fmode, int sms)
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
    const int64_t limit = f64 ? (int64_t)1 << 19 : (int64_t)1 << 20;
    if (nodes > limit) return best;
    std::vector<Counts> counts;
    counts.reserve(grids.size());
    for (const GridView& g : grids) counts.emplace_back(g);
    static const int TW[] = {4, 6, 8, 12, 16, 20, 24, 32, 40, 48, 64, 96, 128};
    static const int TH[] = {2, 3, 4, 6, 8, 12, 16, 20, 24, 32, 40, 48, 64};
    static const int KS[] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 16};
    const size_t per_cell = f64 ? cell_bytes<double>() : cell_bytes<float>();
    double best_cost = 1e300;
    int btw = 0, bth = 0;
    for (int tw : TW)
        for (int th : TH) {
            int64_t upper = 0;
            for (const GridView& g : grids) upper += (int64_t)tiles(g.nx, tw) * tiles(g.ny, th);
            if (upper > 16 * (int64_t)sms) continue;
            int64_t wet = 0;
            int mw = 0, mh = 0;
            for (size_t i = 0; i < grids.size(); ++i) {
                const GridView& g = grids[i];
                const int ntx = tiles(g.nx, tw), nty = tiles(g.ny, th);
                for (int b = 0; b < nty; ++b)
                    for (int a = 0; a < ntx; ++a)
                        wet += counts[i](cut(g.nx, ntx, a), cut(g.nx, ntx, a + 1), cut(g.ny, nty, b), cut(g.ny, nty, b + 1)) > 0;
                mw = std::max(mw, (g.nx + ntx - 1) / ntx);
                mh = std::max(mh, (g.ny + nty - 1) / nty);
            }
            if (wet == 0) continue;
            for (int k : KS) {
                if (MACLAB_WINDOW_K > 0 && k != MACLAB_WINDOW_K) continue;
                // the largest window over the grids
                int ww = 0, wh = 0;
                for (const GridView& g : grids) {
                    const bool fx = tiles(g.nx, tw) == 1, fy = tiles(g.ny, th) == 1;
                    const bool px = g.edge[0] == EDGE_PER && !fx, py = g.edge[2] == EDGE_PER && !fy;
                    ww = std::max(ww, px ? mw + 2 * k : std::min(g.nx, mw + 2 * k));
                    wh = std::max(wh, py ? mh + 2 * k : std::min(g.ny, mh + 2 * k));
                }
                Shape s;
                s.hw = (ww + 5) / 2;
                s.rows = wh + 2;
                s.nlist = s.rows * 2 * s.hw;
                s.ndir = dirichlet ? 2 * (ww + wh) : 0;
                const size_t smem = smem_of(per_cell, s);
                if (smem > MAX_SMEM) continue;
                int np = 1, threads;
                if (f64) {
                    threads = std::min(MAX_THREADS, (ww * wh + 31) / 32 * 32);
                } else {
                    const int pairs = wh * ((ww + 1) / 2);
                    np = pairs <= MAX_THREADS ? 1 : pairs <= 2 * MAX_THREADS ? 2 : 4;
                    if (pairs > MAX_PAIRS * MAX_THREADS) continue;
                    threads = ((pairs + np - 1) / np + 31) / 32 * 32;
                }
                // blocks of one wave that share an SM, and waves
                const int fit = std::max(1, std::min((int)(MAX_SMEM / smem), f64 ? 512 / threads : 512 / threads));
                const int64_t per_sm = (wet + sms - 1) / sms;
                const double waves = (double)((per_sm + fit - 1) / fit), shared = (double)std::min<int64_t>(per_sm, fit);
                double cyc = LAUNCH_CYCLES + LOAD_CELL * ww * wh * shared;
                for (int m = k; m >= 1; --m) {
                    // nodes derived and updated with m steps to take
                    const double cells = 0.5 * (std::min(ww, mw + 2 * m) * (double)std::min(wh, mh + 2 * m) +
                                                std::min(ww, mw + 2 * m - 2) * (double)std::min(wh, mh + 2 * m - 2));
                    if (f64) {
                        const double warps = shared * std::max(1.0, cells / 32);
                        cyc += STEP_CYCLES + INSTR_F64 * std::max(66.0 * std::min(4.0, warps) / 4, 19.0 * warps);
                    } else {
                        cyc += STEP_CYCLES + CELL_F32 * shared * cells;
                    }
                }
                const double cost = waves * cyc / k;
                if (cost < best_cost) {
                    best_cost = cost;
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
    if (best.k == 0) return best;
    best.fm = (fmode & F_CORIOLIS) ? 7 : (fmode & F_FRICTION) ? 3 : 1;
    for (size_t i = 0; i < grids.size(); ++i) {
        const GridView& g = grids[i];
        const int ntx = tiles(g.nx, btw), nty = tiles(g.ny, bth);
        for (int b = 0; b < nty; ++b)
            for (int a = 0; a < ntx; ++a) {
                Item it{(int)i, cut(g.nx, ntx, a), cut(g.nx, ntx, a + 1), cut(g.ny, nty, b), cut(g.ny, nty, b + 1), 0, g.off};
                if (counts[i](it.x0, it.x1, it.y0, it.y1) > 0) best.items.push_back(it);
            }
    }
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
        MACLAB_W(1, 2) MACLAB_W(3, 2) MACLAB_W(7, 2) MACLAB_W(1, 4) MACLAB_W(3, 4) MACLAB_W(7, 4)
    }
#undef MACLAB_W
    return cudaErrorInvalidValue;
}
}  // namespace

cudaError_t prepare_launch(const Plan& p, bool f64)
{
    // the kernels are shared by every handle: opt in to the most any plan takes
    auto opt = [&](const void* k) {
        return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)MAX_SMEM);
    };
    return f64 ? with_kernel<double>(p, opt) : with_kernel<float>(p, opt);
}

template <typename T>
cudaError_t launch(const Plan& p, const void* insts, const Item* items, const uint8_t* active, const Buffers<T>& buf,
                   int steps, const DirTable* tab, cudaStream_t stream)
{
    static const DirTable none{};
    int steady = tab ? 0 : 1;
    void* args[] = {(void*)&insts, (void*)&items, (void*)&active, (void*)&buf, (void*)&p.shape,
                    (void*)&steps, (void*)&steady, (void*)(tab ? tab : &none)};
    return with_kernel<T>(p, [&](const void* k) {
        return cudaLaunchKernel(k, dim3((unsigned)p.items.size()), dim3((unsigned)p.threads), args, p.smem, stream);
    });
}
template cudaError_t launch<float>(const Plan&, const void*, const Item*, const uint8_t*, const Buffers<float>&, int,
                                   const DirTable*, cudaStream_t);
template cudaError_t launch<double>(const Plan&, const void*, const Item*, const uint8_t*, const Buffers<double>&, int,
                                    const DirTable*, cudaStream_t);

}  // namespace window
}  // namespace maclab
