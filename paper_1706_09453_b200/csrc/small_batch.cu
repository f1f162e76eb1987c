// Small batches (1 .. 16 frames): the matrix-vector regime the paper has in mind for embedded
// recognisers.  With so few frames the tiled tensor-core kernels leave almost the whole GPU idle
// and pay their set-up (tensor memory, barriers, a 192 KB weight slice per CTA) for one nearly
// empty tile; what matters here is to spread each layer's WEIGHTS over all SMs and to read them
// once.  Three plain kernels on the integer / FP32 pipes, one warp per output unit:
//
//   small_signw_kernel   y[m][n] = sum_k w[n][k] x[m][k], w = +-1 from packed bits, then the
//                        per-unit affine, Sign and packing (first layer)
//   small_xnor_kernel    d[m][n] = K - 2 popc(a[m] xor w[n])  (or 2 popc(a and w) - popc(a) for
//                        (0,1) frames), threshold, packing (binary hidden layers)
//   small_out_kernel     z[m][c] = sum_n Wout[c][n] h[m][n] + b[c] on packed h (top layer, fp32)
//
// A block of 16 warps owns 16 consecutive units, so that one ballot per frame yields half a
// packed word of the next layer's input (a 2048-wide layer then has 128 blocks).  Lane l of a warp takes the positions k = l, l + 32, ...
// of the unit's row; the per-frame partial sums are reduced with shuffles.  Integer results are
// exact; the fp32 sums differ from the oracle only by the order of fp32 additions.
//
// What bounds them is not the arithmetic but what lies between: launches, and the reductions.  So a run of equal hidden
// layers is ONE launch (small_xnor_kernel), with a barrier over its CTAs between layers, and the words of the next layer's
// weights are in registers when that opens.
// The per-frame partial sums of a unit are reduced all at once, each step halving
// the number of frames a lane is responsible for (31 shuffles for 16 frames instead of 80) in the same tree.
// Measured on B200, 440 -> 6 x 2048 -> 3307, a launch per layer and 32 units a block before: one frame 44 -> 29 us (the
// host's four launches take 20 to 25), 16 frames 85 -> 41 (run of five layers 31 -> 18 us of kernel time and four launches less,
// first layer 12 -> 6; the rest from the top layer, which takes the digit kernel beyond four frames).  The top
// layer's kernel is launched plainly: started under the run it takes from the run what it gains (3 frames 37 us against 33).
#include "bnn_common.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

constexpr int MAXM = kSmallBatchMax;   // frames per launch

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Sums of v[0 .. MT-1] over the 32 lanes, all at once; the lane for which owner_frame() says f returns the sum of v[f].
// A lane adds the same pairs in the same order as warp_sum() does.
template <int MT, typename T>
__device__ __forceinline__ T warp_sums(T (&v)[MT], int lane) {
    int o = 16;
#pragma unroll
    for (int half = MT / 2; half > 0; half >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < half; ++i) {
            const T keep = up ? v[i + half] : v[i], give = up ? v[i] : v[i + half];
            v[i] = keep + __shfl_xor_sync(0xFFFFFFFFu, give, o);
        }
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xFFFFFFFFu, v[0], o);
    return v[0];
}
// The frame whose sum a lane gets, or -1 for all lanes but one of those that get the same.
template <int MT>
__device__ __forceinline__ int owner_frame(int lane) {
    constexpr int step = 32 / MT;
    return lane % step ? -1 : lane / step;
}

// The kernels are instantiated for MT = 1, 4 and 16 frames (the smallest that holds the batch is
// launched), so that a single frame does not pay for sixteen.
// Warp m turns the block's decisions on frame m (dec[unit][frame]) into half a packed word; the grid covers both halves
// of every word.
constexpr int UNITS = 16, THREADS = 32 * UNITS;
inline int unit_blocks(int N) { return 2 * ceil_div(N, 32); }
__device__ __forceinline__ void pack_block(const unsigned char (*dec)[MAXM], int M, int n0, int N,
                                           uint32_t* __restrict__ out_bits, int ldob, int warp, int lane) {
    if (warp < M) {
        const uint32_t word = __ballot_sync(0xFFFFFFFFu, lane < UNITS && (n0 + lane < N) && dec[lane & (UNITS - 1)][warp]);
        if (lane == 0) reinterpret_cast<uint16_t*>(out_bits + (size_t)warp * ldob)[n0 >> 4] = (uint16_t)word;
    }
}

// `clear`: counters of the kernels behind this one, `n_clear` of them.
template <int MT>
__global__ void __launch_bounds__(THREADS)
small_signw_kernel(const float* __restrict__ X, int ldx, const uint32_t* __restrict__ Wp, int ldwp,
                   int M, int N, int K, const float* __restrict__ scale, const float* __restrict__ shift,
                   int sign_mode, uint32_t* __restrict__ out_bits, int ldob, int* __restrict__ clear, int n_clear) {
    pdl_trigger();
    __shared__ unsigned char dec[UNITS][MAXM];
    extern __shared__ float xs[];   // the batch's input, [MT][K]; rows >= M are zero
    __shared__ float xsum[MT];      // sum_k x[m][k], the same for every unit
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * UNITS, n = n0 + warp;
    const int kw = words_for(K);
    if (blockIdx.x == 0)
        for (int i = threadIdx.x; i < n_clear; i += THREADS) clear[i] = 0;
    // lane l holds word l of the unit's row, 32 words at a time
    const uint32_t* w = Wp + (size_t)(n < N ? n : 0) * ldwp;
    uint32_t ww = lane < kw ? __ldg(w + lane) : 0u;
    const float sc = (scale && n < N) ? scale[n] : 1.0f, sh = (shift && n < N) ? shift[n] : 0.0f;
    for (int k = threadIdx.x; k < K; k += THREADS) {
#pragma unroll
        for (int m = 0; m < MT; ++m) xs[m * K + k] = m < M ? __ldg(X + (size_t)m * ldx + k) : 0.f;
    }
    __syncthreads();
    if (warp < MT) {   // warp m adds up row m
        float t = 0.f;
        for (int k = lane; k < K; k += 32) t += xs[warp * K + k];
        t = warp_sum(t);
        if (lane == 0) xsum[warp] = t;
    }
    // sum_k w x = 2 * (sum of x where the weight bit is set) - sum_k x: one predicated add per
    // position and frame
    float acc[MT];
#pragma unroll
    for (int m = 0; m < MT; ++m) acc[m] = 0.f;
    for (int g0 = 0; g0 < kw; g0 += 32) {
        if (g0 > 0) ww = g0 + lane < kw ? __ldg(w + g0 + lane) : 0u;
        const int words = kw - g0 < 32 ? kw - g0 : 32;
#pragma unroll 4
        for (int g = 0; g < words; ++g) {
            const int k = (g0 + g) * 32 + lane;
            const bool plus = (__shfl_sync(0xFFFFFFFFu, ww, g) >> lane) & 1u;
            if (k < K && plus) {
#pragma unroll
                for (int m = 0; m < MT; ++m) acc[m] += xs[m * K + k];
            }
        }
    }
    const float sum = warp_sums<MT>(acc, lane);
    const int m = owner_frame<MT>(lane);
    __syncthreads();
    if (m >= 0) dec[warp][m] = sign_is_pos(fmaf(sc, 2.0f * sum - xsum[m], sh), sign_mode);
    __syncthreads();
    pack_block(dec, M, n0, N, out_bits, ldob, warp, lane);
}

struct SmallRun {
    XnorSmallLayer layer[kXnorStackMax];
    int n_layers;
    int* arrived;            // [n_layers - 1] counters, zero when the kernel before this one has completed (unused for one layer)
    tc::TcStatus status;
};
constexpr int kAhead = 4;    // words of a unit's row that a lane holds in registers (K <= 4096; beyond, they are loaded late)

// All CTAs must be resident at once when there is more than one layer (two per SM, see small_xnor_can_run).  Every
// wait is bounded: after status.limit clocks the CTA sets the status word and returns.
template <bool ZO, int MT>
__global__ void __launch_bounds__(THREADS, 2)
small_xnor_kernel(const uint32_t* __restrict__ Ap, int ldap, const __grid_constant__ SmallRun run, int M, int N, int K, int ldob) {
    __shared__ unsigned char dec[UNITS][MAXM];
    __shared__ int ones[MAXM];         // per frame: its number of ones (ZO)
    __shared__ int gave_up;
    extern __shared__ uint32_t as[];   // the batch's packed frames, [MT][kw]; rows >= M are zero
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int n0 = blockIdx.x * UNITS, n = n0 + warp;
    const int kw = words_for(K);
    const uint32_t tmask = tail_mask(K);
    if (threadIdx.x == 0) gave_up = 0;
    pdl_trigger();
    uint32_t wv[kAhead];
    int t;
    bool f;
    auto fetch = [&](const XnorSmallLayer& y) {
#pragma unroll
        for (int i = 0; i < kAhead; ++i) {
            const int g = lane + 32 * i;
            wv[i] = n < N && g < kw ? __ldg(y.Wp + (size_t)n * y.ldwp + g) : 0u;
        }
        t = n < N ? __ldg(y.thr + n) : 0;
        f = n < N ? ((__ldg(y.flip + (n >> 5)) >> (n & 31)) & 1u) : false;
    };
    fetch(run.layer[0]);
    pdl_wait();
    for (int l = 0; l < run.n_layers; ++l) {
        const XnorSmallLayer& y = run.layer[l];
        const uint32_t* in = l == 0 ? Ap : run.layer[l - 1].out_bits;
        const int ld = l == 0 ? ldap : ldob;
        for (int i = threadIdx.x; i < MT * kw; i += blockDim.x) {
            const int m = i / kw, g = i - m * kw;
            as[i] = m < M ? __ldcg(in + (size_t)m * ld + g) & (g == kw - 1 ? tmask : 0xFFFFFFFFu) : 0u;   // bits >= K hold anything
        }
        __syncthreads();
        if (ZO && warp < MT) {
            int p = 0;
            for (int g = lane; g < kw; g += 32) p += __popc(as[warp * kw + g]);
            p = warp_sum(p);
            if (lane == 0) ones[warp] = p;
        }
        int acc[MT];
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[m] = 0;
        auto add = [&](int g, uint32_t w) {
            const uint32_t wm = g == kw - 1 ? w & tmask : w;
#pragma unroll
            for (int m = 0; m < MT; ++m) acc[m] += __popc(ZO ? as[m * kw + g] & wm : as[m * kw + g] ^ wm);
        };
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
            if (lane + 32 * i < kw) add(lane + 32 * i, wv[i]);
        for (int g = lane + 32 * kAhead; g < kw; g += 32) add(g, n < N ? __ldg(y.Wp + (size_t)n * y.ldwp + g) : 0u);
        const int thr = t;
        const bool flip = f;
        if (l + 1 < run.n_layers) fetch(run.layer[l + 1]);       // on its way while this layer ends
        const int p = warp_sums<MT>(acc, lane);
        const int m = owner_frame<MT>(lane);
        if (ZO) __syncthreads();
        if (m >= 0) dec[warp][m] = ((ZO ? 2 * p - ones[m] : K - 2 * p) >= thr) != flip;
        __syncthreads();
        pack_block(dec, M, n0, N, y.out_bits, ldob, warp, lane);
        if (l + 1 < run.n_layers) {
            __syncthreads();
            if (threadIdx.x == 0) {
                __threadfence();
                asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(run.arrived + l) : "memory");
                const long long t0 = clock64();
#pragma unroll 1
                while (true) {
                    int v;
                    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(run.arrived + l) : "memory");
                    if (v >= (int)gridDim.x) break;
                    if (clock64() - t0 > run.status.limit) {
                        gave_up = 1;
                        atomicExch(run.status.word, 1);
                        break;
                    }
                }
            }
            __syncthreads();
            if (gave_up) return;
        }
    }
}

// One warp per class; 8 classes per block.
template <bool ZO, int MT>
__global__ void __launch_bounds__(256)
small_out_kernel(const uint32_t* __restrict__ Hp, int ldhp, const float* __restrict__ W, int ldw,
                 const float* __restrict__ bias, int M, int C, int H, float* __restrict__ Z, int ldz) {
    // fm[g][lane]: bit m set <=> frame m has a one at position 32 g + lane (frames >= M: clear).
    // Built once per block; the inner loop then needs one shared-memory load per weight.
    extern __shared__ uint16_t fm[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hw = words_for(H);
    const int c = blockIdx.x * 8 + warp;
    const float* w = W + (size_t)(c < C ? c : 0) * ldw;
    // independent loads of the class's weights in flight per lane, the first of them before the frames are gathered:
    // this kernel is bound by how fast the 4 bytes per weight arrive
    constexpr int DEEP = 16;
    float wv[DEEP];
    auto fetch = [&](int g0) {
#pragma unroll
        for (int u = 0; u < DEEP; ++u) {
            const int n = (g0 + u) * 32 + lane;
            wv[u] = n < H ? __ldg(w + n) : 0.f;
        }
    };
    fetch(0);
    const float b = bias && c < C ? __ldg(bias + c) : 0.f;
    for (int i = threadIdx.x; i < hw * 32; i += blockDim.x) {
        const int g = i >> 5, l = i & 31;
        uint32_t t = 0u;
#pragma unroll
        for (int m = 0; m < MT; ++m)
            if (m < M) t |= ((__ldg(Hp + (size_t)m * ldhp + g) >> l) & 1u) << m;
        fm[i] = (uint16_t)t;
    }
    __syncthreads();
    if (c >= C) return;
    // acc[m] = sum of the weights at the positions where frame m's bit is set (one predicated add
    // per weight and frame); with +-1 activations z = 2 acc - (sum of all weights of the class).
    float acc[MT], tot = 0.f;
#pragma unroll
    for (int m = 0; m < MT; ++m) acc[m] = 0.f;
    for (int g0 = 0; g0 < hw; g0 += DEEP) {
        if (g0 > 0) fetch(g0);
#pragma unroll
        for (int u = 0; u < DEEP; ++u) {
            if (g0 + u < hw) {
                tot += wv[u];
                const uint32_t t = fm[(g0 + u) * 32 + lane];
#pragma unroll
                for (int m = 0; m < MT; ++m)
                    if (t & (1u << m)) acc[m] += wv[u];
            }
        }
    }
    tot = warp_sum(tot);
    const float s1 = warp_sums<MT>(acc, lane);
    const int m = owner_frame<MT>(lane);
    if (m >= 0 && m < M) Z[(size_t)m * ldz + c] = (ZO ? s1 : 2.0f * s1 - tot) + b;
}

}  // namespace

#define BNN_SMALL_DISPATCH(M, CALL) \
    do { if ((M) <= 1) { constexpr int MT = 1; CALL; } else if ((M) <= 4) { constexpr int MT = 4; CALL; } \
         else { constexpr int MT = 16; CALL; } } while (0)
static int frames_bound(int M) { return M <= 1 ? 1 : (M <= 4 ? 4 : 16); }

int launch_small_signw(const float* X, int ldx, const uint32_t* Wp, int ldwp, int M, int N, int K,
                       const float* scale, const float* shift, int sign_mode,
                       uint32_t* out_bits, int ldob, int* clear, int n_clear, cudaStream_t st) {
    const size_t smem = (size_t)frames_bound(M) * K * sizeof(float);
    if (M > MAXM || smem > kSmallSmemMax) return BNN_ERR_UNSUPPORTED;
    BNN_SMALL_DISPATCH(M, (small_signw_kernel<MT><<<unit_blocks(N), THREADS, smem, st>>>(X, ldx, Wp, ldwp, M, N, K, scale, shift,
                                                                                      sign_mode, out_bits, ldob, clear, n_clear)));
    return launch_status();
}

// The CTAs of a run wait for one another.  (Its launch starts when the kernel before it has ended, which costs about 2 us
// against a programmatic dependent launch.)  A single layer may start under the kernel before it.
template <typename Kern>
static cudaError_t launch_run(Kern kern, int blocks, size_t smem, cudaStream_t st, const uint32_t* Ap, int ldap, const SmallRun& run,
                              int M, int N, int K, int ldob) {
    return run.n_layers > 1 ? launch_cooperative(kern, dim3(blocks), dim3(THREADS), smem, st, Ap, ldap, run, M, N, K, ldob)
                            : launch_pdl(kern, dim3(blocks), dim3(THREADS), smem, st, Ap, ldap, run, M, N, K, ldob);
}

int launch_small_xnor(const uint32_t* Ap, int ldap, const XnorSmallLayer* layers, int n_layers, int M, int N, int K,
                      int ldob, int zo, int* arrived, cudaStream_t st) {
    const size_t smem = (size_t)frames_bound(M) * words_for(K) * sizeof(uint32_t);
    if (M > MAXM || smem > kSmallSmemMax || n_layers > kXnorStackMax) return BNN_ERR_UNSUPPORTED;
    if (n_layers > 1 && !small_xnor_can_run(N)) return BNN_ERR_UNSUPPORTED;
    SmallRun run{};
    for (int l = 0; l < n_layers; ++l) run.layer[l] = layers[l];
    run.n_layers = n_layers;
    run.arrived = arrived;
    run.status = tc_status();
    if (!run.status.word) return BNN_ERR_CUDA;
    cudaError_t e = cudaSuccess;
    if (zo)
        BNN_SMALL_DISPATCH(M, (e = launch_run(small_xnor_kernel<true, MT>, unit_blocks(N), smem, st, Ap, ldap, run, M, N, K, ldob)));
    else
        BNN_SMALL_DISPATCH(M, (e = launch_run(small_xnor_kernel<false, MT>, unit_blocks(N), smem, st, Ap, ldap, run, M, N, K, ldob)));
    return e == cudaSuccess ? launch_status() : BNN_ERR_CUDA;
}

bool small_xnor_can_run(int N) { return ceil_div(N, 32) <= device_sm_count(); }

int launch_small_out(const uint32_t* Hp, int ldhp, const float* W, int ldw, const float* bias,
                     int M, int C, int H, float* Z, int ldz, int zo, cudaStream_t st) {
    const size_t smem = (size_t)words_for(H) * 32 * sizeof(uint16_t);
    if (M > MAXM || smem > kSmallSmemMax) return BNN_ERR_UNSUPPORTED;
    if (zo)
        BNN_SMALL_DISPATCH(M, (small_out_kernel<true, MT><<<ceil_div(C, 8), 256, smem, st>>>(Hp, ldhp, W, ldw, bias, M, C, H, Z, ldz)));
    else
        BNN_SMALL_DISPATCH(M, (small_out_kernel<false, MT><<<ceil_div(C, 8), 256, smem, st>>>(Hp, ldhp, W, ldw, bias, M, C, H, Z, ldz)));
    return launch_status();
}

}  // namespace bnn
