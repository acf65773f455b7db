// window.h -- host interface of the several-steps-per-launch kernel
// (maclab_window.cuh): the choice of tiles and steps per launch, and the
// launch itself (window.cu).
#pragma once
#include "maclab_window.cuh"

#include <vector>

namespace maclab {
namespace window {

// One grid of a handle or batch, as the planner sees it.
struct GridView {
    int nx, ny, pitch;
    const int* edge;      // W, E, S, N kinds
    const uint8_t* type;  // host [ny][pitch]
    long long off;        // first element in the packed arrays
};

struct Plan {
    int k = 0;                // steps per launch, at most (0: this path is not used)
    int np = 1, threads = 0;  // kernel variant (FP32 pairs per thread) and block size
    int fm = 0;               // force terms compiled in
    size_t smem = 0;
    Shape shape{};
    std::vector<Item> items;
};

// Tiles and steps per launch for these grids (plan.k = 0 when the
// single-step kernels are the better choice).
Plan make_plan(const std::vector<GridView>& grids, bool f64, int fmode, int sms);

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
