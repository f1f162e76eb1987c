// Binary weights x real-valued activations on the tensor cores with exact integer sums (digit_gemm.cuh):
//
//   1. x_digits_kernel writes every frame once per call as fixed-point numbers of a power-of-two scale of its own, in
//      three byte digits, in the order the tensor core reads shared memory (an image in scratch);
//   2. signw_digit_kernel multiplies the digits with the packed +-1 weights: units on the M side (tensor-memory
//      lane = unit), frame digits on the N side, 256 units x 64 (or 32) frames per tile and CTA pair.
//
// For layers that hand on real values.  (A layer with Sign units keeps the bf16 terms of signw_img_tc.cu: there a
// pre-activation near zero turns any change of rounding into another bit, so its sums stay what they were.)
// The epilogue thread owns a unit: per-unit affine (one fma), the activation, fp32 stores of 128 contiguous
// bytes.  When the layer that consumes the outputs is again of this kind (a network with binary weights and real activations, Algorithm 1), the epilogue also writes them
// as that layer's image: hardtanh and Sigmoid outputs lie in [-1, 1], so their scale is fixed (kUnitScale);
// the fp16 image of the real-valued layer on fp32 activations (out_gemm_f32_tc.cu) is written the same way.
//
// |result - exact| <= K * 2^-23 * max_k |x[m][k]| at worst (every rounding of a frame at its largest and of one
// sign; typically sqrt(K) 2^-25), plus one rounding to fp32.  Two bf16 terms, which this path used before, keep 2^-17 of
// each |x| and round the sums at every step.
//
// Bound by the tensor pipe and the board's power for large batches, by launch latency for small ones.  Measured on
// B200 against two bf16 terms on tiles of 128 frames x 512 units, 2048 -> 2048 units chained: 8192 frames 112 -> 63 us,
// 517 frames 56 -> 11 us; largest error of a sum 2^-17 -> 3e-7 of sum |x|.
#include <cuda_fp16.h>

#include "bnn_common.cuh"
#include "digit_gemm.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

using namespace tc;

constexpr float kUnitScale = 4194304.0f;   // 2^22 stands for 1: the affine takes the factor without a rounding

// Staging per epilogue warp: 32 frame scales, 32 frames x two fp16 terms of 32 units.
constexpr int STAGING = 128 + 4096;
constexpr int SMEM_BYTES = digit::RING_BYTES + digit::EPI_WARPS * STAGING + (int)sizeof(digit::Bars) + 1024;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

// Image of M frames of K values: [K / 16][3 ceil8(M)][16 bytes], then a scale per frame.
struct Image {
    int rows, chunks;
    size_t scales;
    __host__ __device__ __forceinline__ Image(int M, int K) {
        rows = 3 * ((M + digit::GRAN - 1) / digit::GRAN * digit::GRAN);
        chunks = 2 * ((K + 31) / 32);
        scales = (size_t)rows * chunks * 16;
    }
};

// ---- frames -> digits: one CTA of eight warps per granule of eight frames ---------------------------------
struct Frames {
    const float* X;
    int ldx, M, K, sdim, sleft;
    bool vec;
    // Four consecutive positions of input row m; beyond the row or the batch: 0.  With splicing (sdim > 0)
    // position k of row m is feature k % sdim of frame m - sleft + k / sdim, clamped to the frames that exist: the
    // context window of the feature front end, formed here instead of being materialised in memory.
    __device__ __forceinline__ float at(int m, int k) const {
        if (k >= K) return 0.f;
        if (sdim > 0) {
            int r = m - sleft + k / sdim;
            r = r < 0 ? 0 : (r >= M ? M - 1 : r);
            return __ldg(X + (size_t)r * ldx + k % sdim);
        }
        return __ldg(X + (size_t)m * ldx + k);
    }
    __device__ __forceinline__ float4 four(int m, int k) const {
        if (m >= M) return make_float4(0.f, 0.f, 0.f, 0.f);
        if (vec && k + 3 < K) {
            int r = m, c = k;
            if (sdim > 0) {
                r = m - sleft + k / sdim;
                r = r < 0 ? 0 : (r >= M ? M - 1 : r);
                c = k % sdim;
            }
            return __ldg(reinterpret_cast<const float4*>(X + (size_t)r * ldx + c));
        }
        return make_float4(at(m, k), at(m, k + 1), at(m, k + 2), at(m, k + 3));
    }
};

// STAGED: the eight rows are kept in (dynamic) shared memory between the search for their largest magnitudes and the
// conversion, pitch K rounded up to 4, plus 4 floats (the eight frames of a conversion step then lie in different
// banks); rows too long for five blocks of it on an SM are read twice.  8192 x 440: 12 us reading twice, 9 staged.
constexpr int STAGED_MAX = 40 * 1024;
__host__ __device__ __forceinline__ int staged_pitch(int K) { return ((K + 3) & ~3) + 4; }

template <bool STAGED>
__global__ void __launch_bounds__(256, 8)
x_digits_kernel(Frames x, uint8_t* __restrict__ img, int* __restrict__ clear, int clear_words) {
    extern __shared__ float rows[];
    __shared__ int exps[digit::GRAN];
    pdl_trigger();   // the GEMM may be scheduled as SMs free up; it waits before it reads the image
    // As the first kernel of a forward pass this one also clears the pass's counters (a few hundred
    // words): a memset node of its own in front of it costs about 4 us per step.
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < clear_words; i += gridDim.x * blockDim.x) clear[i] = 0;
    const Image im(x.M, x.K);
    const int m0 = blockIdx.x * digit::GRAN, pitch = staged_pitch(x.K);
    {   // largest magnitude of each frame as bits (orders NaN above infinity above every number): a warp per frame
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        uint32_t top = 0u;
#pragma unroll 4
        for (int k = 4 * lane; k < x.K; k += 128) {
            const float4 v = x.four(m0 + warp, k);
            if (STAGED) *reinterpret_cast<float4*>(rows + warp * pitch + k) = v;
            top = max(max(top, __float_as_uint(fabsf(v.x))), __float_as_uint(fabsf(v.y)));
            top = max(max(top, __float_as_uint(fabsf(v.z))), __float_as_uint(fabsf(v.w)));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
        if (lane == 0) {
            const float mx = __uint_as_float(top);
            exps[warp] = digit::scale_exponent(mx, 3);
            reinterpret_cast<float*>(img + im.scales)[m0 + warp] = digit::inverse_scale(mx, 3);
        }
    }
    __syncthreads();
    // thread -> frame i, half hh of a group of 32 positions: 16 values, one chunk of each digit row
    const int i = threadIdx.x & 7, hh = (threadIdx.x >> 3) & 1;
    const digit::Scale scale(exps[i]);
    uint8_t* dst0 = img + ((size_t)blockIdx.x * (3 * digit::GRAN) + i) * 16;
    for (int g = threadIdx.x >> 4; g < im.chunks / 2; g += 16) {
        float4 f[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = 32 * g + 8 * j + 4 * hh;
            if (STAGED) f[j] = k < x.K ? *reinterpret_cast<const float4*>(rows + i * pitch + k) : make_float4(0.f, 0.f, 0.f, 0.f);
            else f[j] = x.four(m0 + i, k);
        }
        uint32_t d[3][4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            uint32_t v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = digit::digits3(scale.fixed_point(t == 0 ? f[j].x : t == 1 ? f[j].y : t == 2 ? f[j].z : f[j].w));
            d[0][t] = digit::gather_bytes<0>(v[0], v[1], v[2], v[3]);
            d[1][t] = digit::gather_bytes<1>(v[0], v[1], v[2], v[3]);
            d[2][t] = digit::gather_bytes<2>(v[0], v[1], v[2], v[3]);
        }
        uint8_t* dst = dst0 + (size_t)(2 * g + hh) * im.rows * 16;
#pragma unroll
        for (int q = 0; q < 3; ++q)
            *reinterpret_cast<uint4*>(dst + q * digit::GRAN * 16) = make_uint4(d[q][0], d[q][1], d[q][2], d[q][3]);
    }
}

// ---- the GEMM ---------------------------------------------------------------------------
struct Args {
    const uint32_t* Wp; int ldwp;
    const float* in_scales;      // 2^-e per frame (not UNIT)
    const float* scale; const float* shift;
    int act;                     // NONE, HARDTANH or SIGMOID
    float* Y; int ldy;
    uint8_t* img_out;            // image of the layer that consumes the outputs, or nullptr
    int img_out_kind;            //   0: digits; 1: two fp16 terms, blocks of 256 frames (out_gemm_f32_tc.cu)
};

// UNIT: the frames' scale is kUnitScale (the image was written by the layer before); else g.in_scales gives one per
// frame.
template <bool UNIT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(digit::THREADS, 1)
signw_digit_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ digit::Work w, const __grid_constant__ Args g,
                   TcStatus status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + digit::RING_BYTES;
    digit::Bars* bars = reinterpret_cast<digit::Bars*>(staging + digit::EPI_WARPS * STAGING);
    volatile int* abort_flag = &bars->wait.abort;
    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const uint32_t ring = smem_u32(smem);
    const uint32_t tmem = digit::set_up(bars, status, warp);

    if (warp >= digit::PROD_WARP0) {
        digit::widen_bits<false>(w, g.Wp, g.ldwp, bars, tmem, rank, warp, lane);
    } else if (warp == digit::COPY_WARP) {
        // the image is the output of the kernel before this one in the stream: wait until that kernel has
        // completed and its writes are visible (the weights do not depend on it)
        pdl_wait();
        if (lane == 0) digit::copy_digits(w, &map, ring, bars, rank);
    } else if (warp >= digit::EPI_WARPS) {
        if (rank == 0 && warp <= digit::MMA_WARP2) digit::issue(w, ring, bars, tmem, warp - digit::MMA_WARP);
    } else {
        // ---------------- epilogue: thread = one unit (tensor-memory lane); of a tile's frames warps 0-3 take the
        // first half, warps 4-7 the second
        pdl_wait();
        const int M = w.b_rows, N = w.a_rows;
        const int grans = w.n / (3 * digit::GRAN), per = (grans + 1) >> 1;
        const int g0 = (warp >> 2) * per, ng = grans - g0 < per ? grans - g0 : per;
        const int nb = w.nb();
        uint8_t* mine = staging + warp * STAGING;
        float* rs = reinterpret_cast<float*>(mine);      // frame scales (not UNIT)
        const int half_off = ((lane & 15) >> 2) * 16 + (lane & 3) * 4 + (lane >> 4) * 2;     // of this unit in the fp16 image
        // byte transpose between the lanes l, l + 8, l + 16, l + 24: selectors of the two exchanges
        const uint32_t sel16 = lane & 16 ? 0x3276u : 0x5410u, sel8 = lane & 8 ? 0x3715u : 0x6240u;
        int tl = 0;
        for (digit::Tiles t(w); t.left > 0; t.next(), ++tl) {
            const int n0 = t.a * (2 * digit::ROWS) + rank * digit::ROWS + (warp & 3) * 32, n = n0 + lane;
            const int f0 = t.b * nb + g0 * digit::GRAN;
            const bool unit = n < N;
            float sc = (g.scale && unit) ? __ldg(g.scale + n) : 1.0f;
            const float sh = (g.shift && unit) ? __ldg(g.shift + n) : 0.0f;
            if (UNIT) sc *= 1.0f / kUnitScale;           // exact: fma(sc 2^-22, S, sh) = fma(sc, S 2^-22, sh)
            else {
                __syncwarp();
                rs[lane] = f0 + lane < M ? __ldg(g.in_scales + f0 + lane) : 0.f;
                __syncwarp();
            }
            const int b = tl & 1;
            if (!warp_wait_relaxed(smem_u32(&bars->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane)) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * w.n + g0 * 3 * digit::GRAN);
            const bool any = f0 < M && n0 < N;                      // uniform over the warp
            if (any)
                digit::granules(taddr, ng, 3, [&](int gi, const float (&S)[8]) {
                    float y[8];
                    if (UNIT) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = fmaf(sc, S[i], sh);
                    } else {
                        const float4 r0 = reinterpret_cast<const float4*>(rs)[2 * gi], r1 = reinterpret_cast<const float4*>(rs)[2 * gi + 1];
                        const float r[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = fmaf(sc, S[i] * r[i], sh);
                    }
                    if (g.act == BNN_ACT_HARDTANH) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = fminf(fmaxf(y[i], -1.0f), 1.0f);
                    } else if (g.act == BNN_ACT_SIGMOID) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = 1.0f / (1.0f + expf(-y[i]));
                    }
                    const int f = f0 + gi * digit::GRAN;
                    if (g.Y && unit) {
                        float* dst = g.Y + (size_t)f * g.ldy + n;
#pragma unroll
                        for (int i = 0; i < 8; ++i, dst += g.ldy)
                            if (f + i < M) *dst = y[i];
                    }
                    if (g.img_out && g.img_out_kind == 0 && f < M) {
                        // digits of the 8 frames, byte q of word i; four frames at a time: bytes gathered per digit,
                        // transposed over the four lanes whose units are neighbours in the image, stored as words
                        const Image im(M, N);
                        uint32_t v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = unit ? digit::digits3(__float2int_rn(y[i] * kUnitScale)) : 0u;
                        uint8_t* dst = g.img_out + ((size_t)(2 * (n0 >> 5) + ((lane >> 2) & 1)) * im.rows + (size_t)(f / digit::GRAN) * 24 + (lane >> 3)) * 16 + (lane & 3) * 4;
#pragma unroll
                        for (int h = 0; h < 2; ++h)
#pragma unroll
                            for (int q = 0; q < 3; ++q) {
                                uint32_t x = q == 0 ? digit::gather_bytes<0>(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3])
                                           : q == 1 ? digit::gather_bytes<1>(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3])
                                                    : digit::gather_bytes<2>(v[4 * h], v[4 * h + 1], v[4 * h + 2], v[4 * h + 3]);
                                x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 16), sel16);
                                x = __byte_perm(x, __shfl_xor_sync(0xFFFFFFFFu, x, 8), sel8);
                                *reinterpret_cast<uint32_t*>(dst + (q * 8 + h * 4) * 16) = x;
                            }
                    } else if (g.img_out && g.img_out_kind == 1) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float v = unit ? y[i] : 0.f;
                            const __half hi = __float2half_rn(v), lo = __float2half_rn(v - __half2float(hi));
                            uint8_t* p = mine + 128 + (gi * digit::GRAN + i) * 64 + half_off;
                            *reinterpret_cast<__half*>(p) = hi;
                            *reinterpret_cast<__half*>(p + 2048) = lo;
                        }
                    }
                });
            digit::release_acc(bars, b, lane);
            if (any && g.img_out && g.img_out_kind == 1) {
                __syncwarp();
                if (lane < ng * digit::GRAN && f0 + lane < M) {
                    const int f = f0 + lane;
                    uint8_t* dst = g.img_out + ((size_t)(f >> 8) * words_for(N) + (n0 >> 5)) * 32768u + (size_t)(f & 255) * 16;
                    const uint8_t* src = mine + 128 + lane * 64;
#pragma unroll
                    for (int q = 0; q < 8; ++q)       // term q / 4, chunk q % 4
                        *reinterpret_cast<uint4*>(dst + q * 4096) = *reinterpret_cast<const uint4*>(src + (q >> 2) * 2048 + (q & 3) * 16);
                }
                __syncwarp();
            }
        }
    }
    digit::tear_down(bars, status, warp, tmem);
}

}  // namespace

size_t signw_digit_bytes(int M, int K) {
    const Image im(M, K);
    return im.scales + (size_t)(im.rows / 3) * sizeof(float);
}

int launch_signw_digit(const RealGemmArgs& r, void* workspace, bool image_ready, void* out_image, int out_kind, int* clear,
                       int clear_words, cudaStream_t st) {
    auto kern = image_ready ? signw_digit_kernel<true> : signw_digit_kernel<false>;
    const int sms = device_sm_count();
    if (sms < 2 || !ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM_BYTES)) return BNN_ERR_CUDA;
    const TcStatus status = tc_status();
    if (!status.word) return BNN_ERR_CUDA;
    uint8_t* img = static_cast<uint8_t*>(workspace);
    const Image im(r.M, r.K);
    // (when the kernel before this one in the stream already wrote the image -- the layer that produced
    // these activations -- there is nothing to convert)
    if (!image_ready) {
        const bool vec = (r.lda % 4 == 0) && aligned16(r.Af) && (r.splice_dim % 4 == 0);
        const Frames x{r.Af, r.lda, r.M, r.K, r.splice_dim, r.splice_left, vec};
        const size_t staged = (size_t)digit::GRAN * staged_pitch(r.K) * sizeof(float);
        const int blocks = ceil_div(r.M, digit::GRAN);
        if (staged <= STAGED_MAX) x_digits_kernel<true><<<blocks, 256, staged, st>>>(x, img, clear, clear ? clear_words : 0);
        else x_digits_kernel<false><<<blocks, 256, 0, st>>>(x, img, clear, clear ? clear_words : 0);
    }
    const int steps = ceil_div(r.K, 32), pairs = sms / 2;
    const digit::Work w{r.N, r.M, digit::tile_rows(r.N, r.M, steps, pairs), 3, steps, 0};
    const Args a{r.Bb, r.ldb, image_ready ? nullptr : reinterpret_cast<const float*>(img + im.scales), r.scale, r.shift, r.act,
                 r.Y, r.ldy, static_cast<uint8_t*>(out_image), out_kind};
    CUtensorMap map;
    if (!encode_digit_map(&map, img, im.rows, im.chunks, w.n / 2, digit::KB / 16)) return BNN_ERR_CUDA;
    const long long tiles = (long long)ceil_div(r.N, 2 * digit::ROWS) * ceil_div(r.M, w.n / 3);
    if (launch_pdl(kern, dim3(2 * (int)(tiles < pairs ? tiles : pairs)), dim3(digit::THREADS), SMEM_BYTES, st, map, w, a, status) != cudaSuccess)
        return BNN_ERR_CUDA;
    return launch_status();
}

}  // namespace bnn
