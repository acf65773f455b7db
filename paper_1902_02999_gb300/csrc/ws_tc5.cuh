// ws_tc5.cuh -- the warm-start network's convolutions (forward and input
// gradient) and weight gradients on tcgen05.mma, operands brought in by TMA
// tensor copies, accumulators in tensor memory.  Included by warmstart.cu
// inside its anonymous namespace (uses its ConvArgs, WgradArgs, relu2,
// smem_addr and mbarrier helpers).
//
// Both kernels split a block's 6 warps by role, each role waiting only on
// the mbarriers it needs (no block barrier in the main loop):
//   warp 0           issues the tensor copies of a stage once the MMAs that
//                    last read its buffer have completed ("empty");
//   warp 1           issues the stage's MMAs once its operands are in
//                    ("full") and commits them to the buffer's "empty"
//                    barrier;
//   warps 2..5       read the accumulators out of tensor memory afterwards
//                    (warp w owns lanes 32 (w mod 4) ..) for the epilogue.
// A layer whose input is relu(H) reads the rectified copy that the layer
// before stored beside H, so nothing touches a staged operand between its
// copy and its MMA.  (Rectifying the staged operand instead put 128 threads'
// pass over 16 to 48 KB, a proxy fence and a barrier into every stage's round
// trip.  16 samples, forward pass of 14 layers: 0.548 ms, 0.396 without it;
// training step 1.915 and 1.509 ms; one sample's forward pass 218 and 174 us.)
// Warps 0 and 1 run converged, one elected lane issuing (t5_elect).  Every
// wait is bounded: on time-out
// the block records it in *err, lets the copies in flight land (bounded)
// and leaves without writing its outputs.

constexpr int T5_THREADS = 192;
constexpr uint32_t T5_SW128 = 2, T5_SW32 = 6;  // descriptor swizzle modes: 128-byte and 32-byte

// shared-memory matrix descriptor: start, leading and stride byte offsets,
// descriptor version 1 at bit 46, swizzle mode at bit 61
__device__ __forceinline__ uint64_t t5_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo, uint32_t mode)
{
    uint64_t d = (uint64_t)((saddr >> 4) & 0x3FFF);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)mode << 61;
    return d;
}

// instruction descriptor, kind::f16: f32 accumulate, bf16 A and B; bit 15
// (16) set when A (B) is MN-major instead of K-major; N >> 3 at bit 17,
// M >> 4 at bit 24
__host__ __device__ constexpr uint32_t t5_idesc(int M, int N, bool a_mn, bool b_mn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
           ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__host__ __device__ constexpr uint32_t t5_cols(int n)
{
    return n <= 32 ? 32 : n <= 64 ? 64 : n <= 128 ? 128 : n <= 256 ? 256 : 512;
}

__device__ __forceinline__ void t5_bar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void t5_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void t5_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// One lane of a converged warp.  The issuing loops run with the whole warp
// and let this lane issue: the compiler then keeps descriptors and
// coordinates in uniform registers, which the copies and MMAs take.  Issued
// from an "if (lane == 0)" they are moved there one by one, about 200 cycles
// an MMA and a copy, which paced every stage: 790 cycles between the MMAs of
// one 64-channel stage and the next (clock readings), 345 now.
__device__ __forceinline__ bool t5_elect()
{
    uint32_t p;
    asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}
// the warp's index, uniform
__device__ __forceinline__ int t5_warp() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }
// every lane waits (bounded); the same outcome for the warp
__device__ __forceinline__ bool t5_wait_all(uint32_t bar, uint32_t parity)
{
    return __all_sync(0xffffffffu, tc_mbar_wait(bar, parity)) != 0;
}
// lane 0 waits (bounded), the warp learns the outcome
__device__ __forceinline__ bool t5_warp_wait(uint32_t bar, uint32_t parity, int lane)
{
    bool ok = true;
    if (lane == 0) ok = tc_mbar_wait(bar, parity);
    return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}
__device__ __forceinline__ void t5_load4(uint32_t dst, const CUtensorMap* map, int c0, int c1, int c2, int c3,
                                         uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
        "[%6];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
        : "memory");
}
// [64 channels][x][channel block][y][image]: a box of several channel blocks
__device__ __forceinline__ void t5_load5(uint32_t dst, const CUtensorMap* map, int x, int block, int y, int b, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
        "[%7];\n" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(x), "r"(block), "r"(y), "r"(b), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void t5_load2(uint32_t dst, const CUtensorMap* map, int c0, int c1, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::
            "r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
        : "memory");
}
// a box of shared memory to a tensor (bulk group of the issuing thread)
__device__ __forceinline__ void t5_store4(const CUtensorMap* map, int c0, int c1, int c2, int c3, uint32_t src)
{
    asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];\n" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void t5_mma(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
        : "memory");
}
__device__ __forceinline__ void t5_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
                 : "memory");
}
__device__ __forceinline__ void t5_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void t5_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
        "%14, %15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

// Block start-up shared by both kernels: tensor memory (warp 0) and the
// barriers (thread 0), one arrival each.
template <int ST>
struct T5Bars {
    uint64_t full[ST], empty[ST], done;
};
template <int ST>
__device__ __forceinline__ uint32_t t5_start(T5Bars<ST>& bars, uint32_t* tmem_slot, uint32_t cols, int* flags)
{
    const int tid = threadIdx.x;
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_addr(tmem_slot)),
                     "r"(cols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    if (tid == 0) {
        for (int k = 0; k < ST; ++k) {
            t5_bar_init(smem_addr(&bars.full[k]), 1);
            t5_bar_init(smem_addr(&bars.empty[k]), 1);
        }
        t5_bar_init(smem_addr(&bars.done), 1);
        flags[0] = flags[1] = flags[2] = 0;  // abort, stages issued, stages seen landed
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    return *tmem_slot;
}
// The block may have started before the kernel before it ended (launch_t5):
// waits until that one's results are there.  Weights and biases, written only
// by kernels that let no later one start early, may be read before.
__device__ __forceinline__ void t5_dep_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
__device__ __forceinline__ void t5_prefetch(const CUtensorMap* map)
{
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}
// Block end: after a time-out, the copies still in flight land (bounded)
// before shared and tensor memory are released.
template <int ST>
__device__ __forceinline__ void t5_finish(T5Bars<ST>& bars, uint32_t tmem, uint32_t cols, int* flags, int* err)
{
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (threadIdx.x == 0 && flags[0]) {
        for (int s = flags[2]; s < flags[1]; ++s) tc_mbar_wait(smem_addr(&bars.full[s % ST]), (uint32_t)(s / ST) & 1u);
        atomicOr(err, 1);
    }
    __syncthreads();
    if (threadIdx.x < 32)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(cols) : "memory");
}

// ---------------------------------------------------------------------------
// Convolution (forward, or input gradient with a gate): a block owns a
// tile of 128 consecutive pixels of an image (M = 128) and N output
// channels; K runs over 9 taps x C_in in chunks of KC channels of one tap,
// 64 / KC chunks a stage.  KC = 64: rows of 128 bytes, 128-byte swizzle;
// KC = 16 (16-channel input): rows of 32 bytes, 32-byte swizzle.  Both
// operands K-major; A = the activations at the tap's offset (zero fill
// outside the image), B = the weights [9 C_out][C_in].  The epilogue warps
// load the bias into shared memory and their pixel's residual row and gate
// signs into registers before the main loop, so that only the accumulator
// is waited for at the end.  The bf16 output and its rectified copy go
// through the stage buffers (free by then, in the swizzle of the tensor
// map) and out by tensor stores: a thread's own stores would be 16 bytes
// of a row of 256 each.
//   stage layout: A chunks [64 / KC] of 128 x KC bf16, then B chunks
//   [64 / KC] of N x KC bf16, every chunk on a 1024-byte boundary.
// MINB: blocks per SM; ST stages in flight.
template <int KC, int N, int ST, int MINB>
__global__ void __launch_bounds__(T5_THREADS, MINB) ws_conv5_kernel(const __grid_constant__ TmaOperands maps,
                                                                  const ConvArgs a, int* err)
{
    constexpr int CPS = 64 / KC;
    constexpr uint32_t ACH = 128 * KC * 2, BCH = N * KC * 2;
    constexpr uint32_t ABYTES = CPS * ACH, SBYTES = ABYTES + CPS * BCH;
    constexpr uint32_t MODE = KC == 64 ? T5_SW128 : T5_SW32, SBO = KC == 64 ? 1024 : 256;
    constexpr uint32_t IDESC = t5_idesc(128, N, false, false);
    constexpr uint32_t COLS = t5_cols(N);
    static_assert(N % 64 != 0 || 2 * (N / 64) * 16384u <= ST * SBYTES, "the stores' staging fits the stage buffers");
    extern __shared__ __align__(16) unsigned char t5_raw[];
    __shared__ __align__(8) T5Bars<ST> bars;
    __shared__ uint32_t tmem_slot;
    __shared__ int flags[3];
    __shared__ float sbias[N];
    const uint32_t raw = smem_addr(t5_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    unsigned char* tsm = t5_raw + (base - raw);
    const int R = a.R, Cin = a.Cin, Cout = a.Cout, dil = a.dil;
    const int P = R * R, tiles = P / 128;
    const int b = blockIdx.x / tiles, p0 = (blockIdx.x % tiles) * 128;
    const int n0 = blockIdx.y * N;
    const int tid = threadIdx.x, warp = t5_warp(), lane = tid & 31;
    const int kch = Cin / KC, KT = 9 * kch, NS = (KT + CPS - 1) / CPS;
    if (tid == 32) {
        t5_prefetch(&maps.A);
        t5_prefetch(&maps.B);
    }
    const uint32_t tmem = t5_start<ST>(bars, &tmem_slot, COLS, flags);

    if (warp == 0) {
        // running weight row and, for A, tap column and position (no
        // divisions on the issue path)
        int cb = 0, row = n0;
        auto next_b = [&] {
            cb += KC;
            if (cb == Cin) cb = 0, row += Cout;
        };
        const int px = p0 % R;
        int ci0 = 0, tx = 0, x = px - dil, y = p0 / R - dil;
        auto next_a = [&] {
            ci0 += KC;
            if (ci0 == Cin) {
                ci0 = 0;
                x += dil;
                if (++tx == 3) tx = 0, x = px - dil, y += dil;
            }
        };
        // the first stages: weights before the kernel before this one has
        // ended, activations after
#pragma unroll
        for (int buf = 0; buf < ST; ++buf) {
            if (buf >= NS) break;
            const int nc = min(CPS, KT - buf * CPS);
            const uint32_t sB = base + buf * SBYTES + ABYTES, bar = smem_addr(&bars.full[buf]);
            const bool issue = t5_elect();
            if (issue) t5_expect(bar, (uint32_t)nc * (ACH + BCH));
#pragma unroll
            for (int c = 0; c < CPS; ++c) {
                if (c >= nc) break;
                if (issue) t5_load2(sB + c * BCH, &maps.B, cb, row, bar);
                next_b();
            }
        }
        t5_dep_wait();
#pragma unroll
        for (int buf = 0; buf < ST; ++buf) {
            if (buf >= NS) break;
            const int nc = min(CPS, KT - buf * CPS);
            const uint32_t sA = base + buf * SBYTES, bar = smem_addr(&bars.full[buf]);
            const bool issue = t5_elect();
#pragma unroll
            for (int c = 0; c < CPS; ++c) {
                if (c >= nc) break;
                if (issue) t5_load4(sA + c * ACH, &maps.A, ci0, x, y, b, bar);
                next_a();
            }
        }
        int s = min(ST, NS);
        uint32_t par = 0;
        bool go = true;
        while (go && s < NS) {
#pragma unroll
            for (int buf = 0; buf < ST; ++buf) {
                if (s >= NS) break;
                if (!t5_wait_all(smem_addr(&bars.empty[buf]), par)) {
                    if (lane == 0) atomicOr(&flags[0], 1);
                    go = false;
                    break;
                }
                const int nc = min(CPS, KT - s * CPS);
                const uint32_t sA = base + buf * SBYTES, sB = sA + ABYTES, bar = smem_addr(&bars.full[buf]);
                const bool issue = t5_elect();
                if (issue) t5_expect(bar, (uint32_t)nc * (ACH + BCH));
#pragma unroll
                for (int c = 0; c < CPS; ++c) {
                    if (c >= nc) break;
                    if (issue) {
                        t5_load4(sA + c * ACH, &maps.A, ci0, x, y, b, bar);
                        t5_load2(sB + c * BCH, &maps.B, cb, row, bar);
                    }
                    next_a();
                    next_b();
                }
                ++s;
            }
            par ^= 1u;
        }
        if (lane == 0) flags[1] = s;
        __syncwarp();
    } else if (warp == 1) {
        int s = 0;
        uint32_t par = 0;
        bool go = true;
        while (go && s < NS) {
#pragma unroll
            for (int buf = 0; buf < ST; ++buf) {
                if (s >= NS) break;
                if (!t5_wait_all(smem_addr(&bars.full[buf]), par)) {
                    if (lane == 0) atomicOr(&flags[0], 1);
                    go = false;
                    break;
                }
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const int nc = min(CPS, KT - s * CPS);
                const uint32_t sA = base + buf * SBYTES, sB = sA + ABYTES;
                if (t5_elect()) {
#pragma unroll
                    for (int c = 0; c < CPS; ++c) {
                        if (c >= nc) break;
                        const uint64_t ad = t5_desc(sA + c * ACH, 16, SBO, MODE), bd = t5_desc(sB + c * BCH, 16, SBO, MODE);
#pragma unroll
                        for (int k16 = 0; k16 < KC / 16; ++k16)  // 32 bytes on: 2 in the descriptors' units
                            t5_mma(tmem, ad + 2 * k16, bd + 2 * k16, IDESC, (buf | c | k16) != 0 || s != 0 ? 1u : 0u);
                    }
                    t5_commit(smem_addr(&bars.empty[buf]));
                }
                ++s;
            }
            par ^= 1u;
        }
        if (lane == 0) flags[2] = s;
        // arrives once every MMA issued above has completed
        if (t5_elect()) t5_commit(smem_addr(&bars.done));
        __syncwarp();
    } else {
        // before the main loop: bias to shared memory, this lane's pixel's
        // residual row and gate signs to registers
        const int q = warp & 3;  // tensor-memory lanes 32 q .. 32 q + 31
        const int m = q * 32 + lane;
        const size_t o0 = ((size_t)b * P + p0 + m) * Cout + n0;
        for (int c = tid - 64; c < N; c += T5_THREADS - 64) sbias[c] = a.bias ? a.bias[n0 + c] : 0.f;
        t5_dep_wait();
        uint4 rres[N / 8];
        uint32_t gbits[(N + 31) / 32];
#pragma unroll
        for (int k = 0; k < N / 8; ++k) rres[k] = a.res ? reinterpret_cast<const uint4*>(a.res + o0)[k] : make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int k = 0; k < (N + 31) / 32; ++k) gbits[k] = 0xFFFFFFFFu;
        if (a.gate) {
#pragma unroll
            for (int k = 0; k < N / 8; ++k) {
                const uint4 g4 = reinterpret_cast<const uint4*>(a.gate + o0)[k];
                const __nv_bfloat162* gt = reinterpret_cast<const __nv_bfloat162*>(&g4);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = 8 * k + 2 * j;
                    if (!(__bfloat162float(gt[j].x) > 0.f)) gbits[c >> 5] &= ~(1u << (c & 31));
                    if (!(__bfloat162float(gt[j].y) > 0.f)) gbits[(c + 1) >> 5] &= ~(1u << ((c + 1) & 31));
                }
            }
        }
        asm volatile("bar.sync 1, 128;\n" ::: "memory");  // sbias written by the four epilogue warps
        const bool fin = t5_warp_wait(smem_addr(&bars.done), 0, lane);
        if (!fin && lane == 0) atomicOr(&flags[0], 1);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const bool good = fin && !*(volatile int*)&flags[0];
        constexpr int CW = N % 32 == 0 ? 32 : 16;  // columns read from tensor memory at a time
        constexpr int HW = N % 64 == 0 ? 64 : N;   // columns of one output box
#pragma unroll
        for (int h0 = 0; h0 < N; h0 += HW) {
            if (good) {
#pragma unroll
                for (int c0 = h0; c0 < h0 + HW; c0 += CW) {
                    uint32_t r[CW];
                    const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c0;
                    if constexpr (CW == 32) t5_ld32(ta, r);
                    else t5_ld16(ta, r);
                    float v[CW];
#pragma unroll
                    for (int j = 0; j < CW; ++j) {
                        v[j] = __uint_as_float(r[j]) + sbias[c0 + j];
                        if (!((gbits[(c0 + j) >> 5] >> ((c0 + j) & 31)) & 1u)) v[j] = 0.f;
                    }
                    if (a.res) {
                        const __nv_bfloat162* rr = reinterpret_cast<const __nv_bfloat162*>(&rres[c0 / 8]);
#pragma unroll
                        for (int j = 0; j < CW / 2; ++j) {
                            v[2 * j] += __bfloat162float(rr[j].x);
                            v[2 * j + 1] += __bfloat162float(rr[j].y);
                        }
                    }
                    if (a.Y) {
#pragma unroll
                        for (int k = 0; k < CW / 8; ++k) {
                            uint4 w2;
                            __nv_bfloat162* wb = reinterpret_cast<__nv_bfloat162*>(&w2);
#pragma unroll
                            for (int j = 0; j < 4; ++j) wb[j] = __floats2bfloat162_rn(v[8 * k + 2 * j], v[8 * k + 2 * j + 1]);
                            if constexpr (N % 64 == 0) {
                                // 16-byte chunk c of row m of a box (64 channels) at m 128 + (c ^ m % 8) 16
                                const int ch = (c0 - h0) / 8 + k;
                                uint4* to = reinterpret_cast<uint4*>(tsm + (h0 / 64) * 16384 + m * 128 + ((ch ^ (m & 7)) << 4));
                                *to = w2;
                                if (a.YR) to[(N / 64) * 1024] = make_uint4(relu2(w2.x), relu2(w2.y), relu2(w2.z), relu2(w2.w));
                            } else {
                                *reinterpret_cast<uint4*>(a.Y + o0 + c0 + 8 * k) = w2;
                            }
                        }
                    }
                    if (a.Yf) {
#pragma unroll
                        for (int j = 0; j < CW; j += 4)
                            *reinterpret_cast<float4*>(a.Yf + o0 + c0 + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
                    }
                }
            }
            if constexpr (N % 64 == 0) {
                // one box is on its way while the next is computed
                asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // the staged rows, to the tensor stores
                asm volatile("bar.sync 1, 128;\n" ::: "memory");
                if (warp == 2 && good && !*(volatile int*)&flags[0] && a.Y) {
                    if (t5_elect()) {
                        t5_store4(&maps.Y, n0 + h0, p0 % R, p0 / R, b, base + (h0 / 64) * 16384);
                        if (a.YR) t5_store4(&maps.YR, n0 + h0, p0 % R, p0 / R, b, base + (N / 64 + h0 / 64) * 16384);
                        asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
                    }
                    __syncwarp();
                }
            }
        }
        if constexpr (N % 64 == 0) {
            // shared memory is read before the block leaves (a lane without stores passes at once)
            if (warp == 2) asm volatile("cp.async.bulk.wait_group.read 0;\n" ::: "memory");
        }
    }
    t5_finish<ST>(bars, tmem, COLS, flags, err);
}

// ---------------------------------------------------------------------------
// Weight gradient dW[tap][co][ci] = sum_p G[p][co] X[p + d off(tap)][ci]
// (X = the layer's input, the rectified copy where it is relu(H); G = the
// gradient of its output).  A block owns one row of taps (dy = blockIdx.x
// - 1, all three dx), a 128-channel tile of one side and an N-channel
// tile of the other (blockIdx.z), and every 64-pixel row segment of one
// split (blockIdx.y): K = pixels, 64 a stage, both operands MN-major (the
// channels are contiguous in memory).  MG: the 128-channel M side is G's
// output channels (N = X's input channels), else it is X's input channels
// (N = G's 16 output channels, the head).  The G tile of a stage is loaded
// once for the three taps; each tap's X tile sits at its own offset, zero
// filled outside the image, and accumulates into its own N columns of
// tensor memory.  The split's sums go to part[split][tap][co][ci] and are
// added in split order afterwards, so every run sums the same way.
//   stage layout: the G tile, then the X tiles of taps dx = -1, 0, 1; a
//   128-channel tile is two 64-channel boxes of 64 rows (pixels) x 128
//   bytes (128-byte swizzle: 8-row groups 1024 bytes apart, the second box
//   8192 bytes on), a 16-channel tile one box of 64 rows x 32 bytes (32-byte
//   swizzle, 8-row groups 256 bytes apart).  A K = 16 step moves 16 rows on.
template <bool MG, int N, int ST>
__global__ void __launch_bounds__(T5_THREADS) ws_wgrad5_kernel(const __grid_constant__ TmaOperands maps,
                                                                const WgradArgs a, int* err)
{
    constexpr uint32_t MSZ = 128 * 64 * 2, NSZ = N * 64 * 2;
    constexpr uint32_t GSZ = MG ? MSZ : NSZ, XSZ = MG ? NSZ : MSZ, SBYTES = GSZ + 3 * XSZ;
    constexpr uint32_t IDESC = t5_idesc(128, N, true, true);
    constexpr uint32_t COLS = t5_cols(3 * N);
    extern __shared__ __align__(16) unsigned char t5_raw[];
    __shared__ __align__(8) T5Bars<ST> bars;
    __shared__ uint32_t tmem_slot;
    __shared__ int flags[3];
    const uint32_t raw = smem_addr(t5_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    const int R = a.R, Cin = a.Cin, Cout = a.Cout, dil = a.dil;
    const int dy = (int)blockIdx.x - 1, split = blockIdx.y;
    const int mtiles = (MG ? Cout : Cin) / 128;
    const int m0 = (blockIdx.z % mtiles) * 128, n0 = (blockIdx.z / mtiles) * N;
    const int g0c = MG ? m0 : n0, x0c = MG ? n0 : m0;  // first channel of the G and X tiles
    const int segs_row = R / 64, segs = a.B * R * segs_row;
    const int sg0 = (int)((long long)split * segs / a.splits), sg1 = (int)((long long)(split + 1) * segs / a.splits);
    const int NS = sg1 - sg0;
    const int tid = threadIdx.x, warp = t5_warp(), lane = tid & 31;
    if (tid == 32) {
        t5_prefetch(&maps.A);
        t5_prefetch(&maps.B);
    }
    const uint32_t tmem = t5_start<ST>(bars, &tmem_slot, COLS, flags);
    t5_dep_wait();

    if (warp == 0) {
        // running segment: column block, row, image
        int x0 = (sg0 % segs_row) * 64, y = (sg0 / segs_row) % R, b = sg0 / segs_row / R;
        int s = 0, buf = 0;
        uint32_t par = 1;
        for (; s < NS; ++s) {
            if (s >= ST && !t5_wait_all(smem_addr(&bars.empty[buf]), par)) {
                if (lane == 0) atomicOr(&flags[0], 1);
                break;
            }
            const uint32_t st = base + buf * SBYTES, bar = smem_addr(&bars.full[buf]);
            if (t5_elect()) {
                t5_expect(bar, SBYTES);
                // G tile (maps.A): two boxes of 64 channels in one copy, or 16 channels
                if (GSZ == MSZ) t5_load5(st, &maps.A, x0, g0c / 64, y, b, bar);
                else t5_load4(st, &maps.A, g0c, x0, y, b, bar);
                // X tiles of the three taps of this row (maps.B)
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const uint32_t xt = st + GSZ + t * XSZ;
                    const int xx = x0 + (t - 1) * dil, yy = y + dy * dil;
                    if (XSZ == MSZ) t5_load5(xt, &maps.B, xx, x0c / 64, yy, b, bar);
                    else t5_load4(xt, &maps.B, x0c, xx, yy, b, bar);
                }
            }
            __syncwarp();
            x0 += 64;
            if (x0 == R) {
                x0 = 0;
                if (++y == R) y = 0, ++b;
            }
            if (++buf == ST) buf = 0, par ^= 1u;
        }
        if (lane == 0) flags[1] = s;
        __syncwarp();
    } else if (warp == 1) {
        int s = 0, buf = 0;
        uint32_t par = 0;
        for (; s < NS; ++s) {
            if (!t5_wait_all(smem_addr(&bars.full[buf]), par)) {
                if (lane == 0) atomicOr(&flags[0], 1);
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t st = base + buf * SBYTES;
            if (t5_elect()) {
#pragma unroll
                for (int t = 0; t < 3; ++t) {
                    const uint32_t xt = st + GSZ + t * XSZ;
                    const uint32_t sa = MG ? st : xt;  // the 128-channel side
                    const uint32_t sb = MG ? xt : st;  // the N side
#pragma unroll
                    for (int k16 = 0; k16 < 4; ++k16) {
                        const uint64_t ad = t5_desc(sa + k16 * 2048, 8192, 1024, T5_SW128);
                        const uint64_t bd = N == 128 ? t5_desc(sb + k16 * 2048, 8192, 1024, T5_SW128)
                                                     : t5_desc(sb + k16 * 512, 16, 256, T5_SW32);
                        t5_mma(tmem + t * N, ad, bd, IDESC, (s | k16) != 0 ? 1u : 0u);
                    }
                }
                t5_commit(smem_addr(&bars.empty[buf]));
            }
            __syncwarp();
            if (++buf == ST) buf = 0, par ^= 1u;
        }
        if (lane == 0) flags[2] = s;
        if (t5_elect()) t5_commit(smem_addr(&bars.done));
        __syncwarp();
    } else {
        const bool fin = t5_warp_wait(smem_addr(&bars.done), 0, lane);
        if (!fin && lane == 0) atomicOr(&flags[0], 1);
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (fin && !*(volatile int*)&flags[0]) {
            const int q = warp & 3;
            const int m = m0 + q * 32 + lane;  // this lane's channel on the 128-channel side
#pragma unroll 1
            for (int t = 0; t < 3; ++t) {
                const int tap = (dy + 1) * 3 + t;
                float* out = a.part + ((size_t)split * 9 + tap) * Cout * Cin;
#pragma unroll 1
                for (int c0 = 0; c0 < N; c0 += 16) {
                    uint32_t r[16];
                    t5_ld16(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(t * N + c0), r);
                    if (MG) {  // row co = m, columns ci = n0 + c0 ..
                        float* d = out + (size_t)m * Cin + n0 + c0;
#pragma unroll
                        for (int j = 0; j < 16; j += 4)
                            *reinterpret_cast<float4*>(d + j) = make_float4(__uint_as_float(r[j]), __uint_as_float(r[j + 1]),
                                                                            __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
                    } else {  // ci = m, co = n0 + c0 + j: a warp writes 32 consecutive ci
#pragma unroll
                        for (int j = 0; j < 16; ++j) out[(size_t)(n0 + c0 + j) * Cin + m] = __uint_as_float(r[j]);
                    }
                }
            }
        }
    }
    t5_finish<ST>(bars, tmem, COLS, flags, err);
}
