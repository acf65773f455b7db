// window.h -- host interface of the several-steps-per-launch kernel
// (maclab_window.cuh): the choice of tiles and steps per launch, and the
// launch itself (window.cu).
#pragma once
#include "maclab_window.cuh"

#include <algorithm>
#include <cstdint>
#include <vector>

namespace maclab {
namespace window {

// One grid of a handle or batch, as the planner sees it.
struct GridView {
    int nx, ny, pitch;
    const int* edge;      // W, E, S, N kinds
    const uint8_t* type;  // host [ny][pitch]
    long long off;        // first element in the packed arrays
    int walls, dirichlet; // nodes with a bounce-back link, Dirichlet nodes
    const int* wall;      // the former (j * nx + i)
};

// One step of an FP32 batch, us, of 64 x 16 tiles (one launch of the tile
// kernel) and of strip blocks (one of the row march), by the tiles, the rows
// of its strip blocks (two more each than they write; plain and with edge
// rules), the nodes with a bounce-back link and the Dirichlet nodes.  Fitted
// to 90 batches on a GB300 (0.1 to 16 M nodes; instances of 3 x 700 to 2000
// x 1500, lakes, channels, all edge kinds): 11 % standard error each.  The
// faster one by these is at most 4 % slower than the tile kernel anywhere and
// up to 2.1 times as fast as the row march (366 of 64 x 64: 14 us against 30;
// 96 lakes and channels, 8 M nodes: 114 against 78).
inline double batch_tile_us(double tiles, double walls, double dirichlet)
{
    return 2.9 + 0.0092 * tiles + (walls > 0 ? 2.8 + 4.5e-5 * walls : 0.0) + 1.3e-4 * dirichlet;
}
inline double batch_march_us(double rows, double edge_rows, double walls, double dirichlet)
{
    return 10.7 + 3.4e-4 * rows + 4.2e-4 * edge_rows + 4.2e-5 * walls + 7.6e-5 * dirichlet;
}

struct Plan {
    int k = 0;                // steps per launch, at most (0: this path is not used)
    int np = 1, threads = 0;  // kernel variant (FP32 pairs per thread) and block size
    int fm = 0;               // force terms compiled in
    size_t smem = 0;
    int min_steps = 1;        // shorter calls are cheaper in single-step launches
    Shape shape{};
    std::vector<Item> items;
};

// Launches that take n steps at most k at a time: one for a single step, two
// or more otherwise (see WindowRun).
inline int64_t launches(int64_t n, int k) { return std::max<int64_t>(n > 1 ? 2 : 1, (n + k - 1) / k); }

// Tiles and steps per launch for these grids, a batch's or one handle's
// (plan.k = 0 when the single-step kernels are the better choice).
Plan make_plan(const std::vector<GridView>& grids, bool batch, bool f64, int fmode, int sms);

// Device memory of a plan's lists, and the lists built there (once per
// handle; the stream's work must end before p.items goes).  insts: the
// device's BatchInst<T>[].
size_t list_bytes(const Plan& p);
template <typename T>
cudaError_t build_lists(const Plan& p, const void* insts, void* mem, cudaStream_t stream, Lists* out);

// `steps` (<= p.k) steps of every tile; tab: boundary values per step,
// nullptr when steady.
template <typename T>
cudaError_t launch(const Plan& p, const void* insts, const Lists& lists, const uint8_t* active, const Buffers<T>& buf,
                   int steps, const DirTable* tab, cudaStream_t stream);

}  // namespace window
}  // namespace maclab
