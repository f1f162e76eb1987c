// Binary weights x real-valued activations on the tensor cores with exact integer sums (digit_dense.cuh):
//
//   1. x_digits_kernel writes every frame once per call as fixed-point numbers of a power-of-two scale of its own, in
//      three byte digits, in the order the tensor core reads shared memory (an image in scratch);
//   2. signw_digit_kernel multiplies the digits with the packed +-1 weights: units on the M side (tensor-memory
//      lane = unit), frame digits on the N side, 256 units x 64 (or 32) frames per tile and CTA pair.
//
// For layers that hand on real values.  (A layer with Sign units keeps the bf16 terms of signw_img_tc.cu: there a
// pre-activation near zero turns any change of rounding into another bit, so its sums stay what they were.)
// The epilogue thread owns a unit: per-unit affine (one fma), the activation, fp32 stores of 128 contiguous
// bytes.  When the layer that consumes the outputs is again of this kind (a network with binary weights and real
// activations, Algorithm 1), the epilogue also writes them as that layer's image.  A frame's scale then has to be chosen before
// its largest output is known: from a bound on its outputs, min(1, max |scale| * sum |x| + max |shift|) for hardtanh and
// likewise for Sigmoid, with sum |x| <= sqrt(K sum x^2), for which every kernel of such a chain adds up the squares of each
// frame's high digits as it writes them (one instruction per four units).  A scale for outputs up to 1 would do in most
// networks, but loses outputs that are all small: six layers of 2048 units with scale 0.001, relative error of the last
// one's outputs 0.75 with it, 6e-6 with scales from the bound, 1.3e-5 with two bf16 terms.  (What the bound costs: 517 frames,
// six layers, 98 -> 100 us.)
// The fp16 image of the real-valued layer on fp32 activations (out_gemm_f32_tc.cu) is written the same way.
//
// |result - exact| <= K * 1.01 * 2^-23 * max_k |x[m][k]| at worst (every rounding of a frame at its largest and of one
// sign; typically sqrt(K) 2^-25), plus one rounding to fp32.  Two bf16 terms, which this path used before, keep 2^-17 of
// each |x| and round the sums at every step.
//
// Bound by the tensor pipe and the board's power for large batches, by launch latency for small ones.  Measured on
// B200 against two bf16 terms on tiles of 128 frames x 512 units, 2048 -> 2048 units chained: 8192 frames 112 -> 63 us,
// 517 frames 56 -> 11 us; largest error of a sum 2^-17 -> 3e-7 of sum |x|.
#include <cfloat>

#include <cuda_fp16.h>

#include "bnn_common.cuh"
#include "digit_dense.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

using namespace tc;
namespace dense = digit::dense;

// Staging per epilogue warp: 32 frame scales of the input, then 32 of the output and 32 x 8 sums, or 32 frames x two fp16
// terms of 32 units.
constexpr int STAGING = 128 + 4096;
constexpr int SMEM_BYTES = dense::RING_BYTES + digit::EPI_WARPS * STAGING + (int)sizeof(dense::Bars) + 1024;
constexpr int BOUNDS_WARP = digit::COPY_WARP + 1;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

// Image of M frames of K values: [K / 16][3 ceil8(M)][16 bytes], then 2^-e per frame.  The images that layers of a chain hand
// one another start with what the next scales are chosen from: the UnitBounds of the layer that reads the image, and two
// arrays of a word per frame, the sum of the squares of the frame's high digits (at most 2^29) and, in the top bit, whether an
// output is a NaN, which has no digits: the reader then takes the frame's scale for a NaN.  Whoever writes the image
// adds to one array; its reader clears the other one, for the image that is written in the same place next
// (launch_signw_digit).  There is room: the digits leave 32 bytes or more a frame of what bf16 terms take.
struct Image {
    int rows, chunks;
    size_t digits, scales;       // offsets
    __host__ __device__ __forceinline__ Image(int M, int K, bool chained) {
        const int frames = (M + digit::GRAN - 1) / digit::GRAN * digit::GRAN;
        rows = 3 * frames;
        chunks = 2 * ((K + 31) / 32);
        digits = chained ? (16 + (size_t)frames * 8 + 255) & ~size_t(255) : 0;
        scales = digits + (size_t)rows * chunks * 16;
    }
    __host__ __device__ __forceinline__ size_t sums(int which) const { return 16 + (size_t)(rows / 3) * 4 * (which & 1); }
};

// The per-unit affine of a layer.
struct Affine {
    const float* scale;
    const float* shift;
    int N;
};
// What bounds the outputs of a layer besides its input: the largest |scale| and |shift| and the largest shift, as bits.
struct UnitBounds {
    uint32_t scale, shift, top_shift;
    static constexpr uint32_t kTop = 0x80000000u, kInf = 0x7F800000u;
    __device__ __forceinline__ UnitBounds(uint32_t sc, uint32_t sh, uint32_t top) : scale(sc), shift(sh), top_shift(top) {}
    // By `threads` threads; the parts are joined by the caller.
    __device__ __forceinline__ UnitBounds(const Affine& a, int thread, int threads) {
        scale = a.scale ? 0u : 0x3F800000u;
        shift = 0u;
        top_shift = a.shift ? 0u : kTop;
#pragma unroll 8
        for (int n = thread; n < a.N; n += threads) {
            if (a.scale) scale = max(scale, __float_as_uint(fabsf(__ldg(a.scale + n))));     // orders NaN above infinity above every number
            if (a.shift) {
                const uint32_t b = __float_as_uint(__ldg(a.shift + n));
                shift = max(shift, b & ~kTop);
                top_shift = max(top_shift, b & kTop ? ~b : b | kTop);                        // order of the signed numbers
            }
        }
        scale = __reduce_max_sync(0xFFFFFFFFu, scale);
        shift = __reduce_max_sync(0xFFFFFFFFu, shift);
        top_shift = __reduce_max_sync(0xFFFFFFFFu, top_shift);
    }
    __device__ __forceinline__ explicit UnitBounds(const uint8_t* img) {
        const uint4 v = __ldcg(reinterpret_cast<const uint4*>(img));
        scale = v.x; shift = v.y; top_shift = v.z;
    }
    __device__ __forceinline__ void store(uint8_t* img) const { *reinterpret_cast<uint4*>(img) = make_uint4(scale, shift, top_shift, 0u); }
    // Exponent of the scale of a frame whose inputs' magnitudes add up to at most `sum`.  (Up to 100: beyond, 2^-e leaves the
    // range of numbers that keep their precision.)
    __device__ __forceinline__ int exponent(float sum, bool sigmoid) const {
        const float d = __uint_as_float(scale) * sum, sh = __uint_as_float(shift);
        const float top = __uint_as_float(top_shift & kTop ? top_shift & ~kTop : ~top_shift);
        // roundings of the sums, the affine and the activation stay far below the margins
        float b = sigmoid ? expf(d + top + 1e-6f * (d + sh)) : d + sh;
        b *= 1.0001f;
        const int e = digit::scale_exponent(max(scale, shift) < kInf && b < 1.0f ? b : 1.0f);
        return e > 100 ? 100 : e;
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

// A NaN among a layer's outputs is handed on as the number below all others, of which the high digit alone is not zero.  The
// outputs of Sigmoid units are not negative, so their high digits with the top bit set are NaNs, and a part of a frame's
// sum of squares (at most 8 * 4 * 127^2 together) is replaced by one that shows in the sum.
constexpr float kNaNDigits = -8388608.0f;
constexpr int kNaNSquare = 1 << 27;
constexpr uint32_t kNaNOutput = 0x80000000u;     // in a frame's sum

// At least sum_k |v| * 2^-e, given 2^-e and the sum of the squares of the high digits (|v| <= 65536 |high| + 32896).
__device__ __forceinline__ float magnitude_bound(float inv_scale, uint32_t squares, int K) {
    const float root = sqrtf((float)K);
    return inv_scale * root * fmaf(65536.0f, sqrtf((float)squares), 32896.0f * root);
}

// STAGED: the eight rows are kept in (dynamic) shared memory between the search for their largest magnitudes and the
// conversion, pitch K rounded up to 4, plus 4 floats (the eight frames of a conversion step then lie in different
// banks); rows too long for five blocks of it on an SM are read twice.  8192 x 440: 12 us reading twice, 9 staged.
constexpr int STAGED_MAX = 40 * 1024;
__host__ __device__ __forceinline__ int staged_pitch(int K) { return ((K + 3) & ~3) + 4; }

// sums, next_sums (a chain of layers) or nullptr: this image's sums are written, those of the image that the layer behind
// this kernel writes are cleared; one more block finds the bounds of that layer, `units`.
template <bool STAGED>
__global__ void __launch_bounds__(256, 8)
x_digits_kernel(Frames x, uint8_t* __restrict__ img, uint32_t* __restrict__ sums, uint32_t* __restrict__ next_sums,
                Affine units, int* __restrict__ clear, int clear_words) {
    extern __shared__ float rows[];
    __shared__ int exps[digit::GRAN];
    __shared__ uint32_t parts[3];
    pdl_trigger();   // the GEMM may be scheduled as SMs free up; it waits before it reads the image
    // As the first kernel of a forward pass this one also clears the pass's counters (a few hundred
    // words): a memset node of its own in front of it costs about 4 us per step.
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < clear_words; i += gridDim.x * blockDim.x) clear[i] = 0;
    const Image im(x.M, x.K, sums != nullptr);
    if (blockIdx.x * digit::GRAN >= x.M) {
        if (threadIdx.x < 3) parts[threadIdx.x] = 0u;
        __syncthreads();
        UnitBounds b(units, threadIdx.x, 256);
        if ((threadIdx.x & 31) == 0) {
            atomicMax(&parts[0], b.scale);
            atomicMax(&parts[1], b.shift);
            atomicMax(&parts[2], b.top_shift);
        }
        __syncthreads();
        b.scale = parts[0]; b.shift = parts[1]; b.top_shift = parts[2];
        if (threadIdx.x == 0) b.store(img);
        return;
    }
    const int m0 = blockIdx.x * digit::GRAN, pitch = staged_pitch(x.K);
    {   // largest magnitude of each frame as bits (orders NaN above infinity above every number): a warp per frame
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
        uint32_t top = 0u;
        float all = 0.f;
#pragma unroll 4
        for (int k = 4 * lane; k < x.K; k += 128) {
            const float4 v = x.four(m0 + warp, k);
            if (STAGED) *reinterpret_cast<float4*>(rows + warp * pitch + k) = v;
            top = max(max(top, __float_as_uint(fabsf(v.x))), __float_as_uint(fabsf(v.y)));
            top = max(max(top, __float_as_uint(fabsf(v.z))), __float_as_uint(fabsf(v.w)));
            all += (fabsf(v.x) + fabsf(v.y)) + (fabsf(v.z) + fabsf(v.w));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
            all += __shfl_xor_sync(0xFFFFFFFFu, all, o);
        }
        if (lane == 0) {
            const float mx = __uint_as_float(top);
            exps[warp] = digit::scale_exponent(mx);
            reinterpret_cast<float*>(img + im.scales)[m0 + warp] = top < 0x7F800000u ? dense::inverse_scale(exps[warp]) : __int_as_float(0x7FC00000);
            if (sums) {
                // what gives magnitude_bound() the sum of the magnitudes itself; roundings stay far below 0.001
                const dense::Scale scale(exps[warp]);
                const float t = all * scale.a * scale.b * (1.001f / 65536.0f);
                sums[m0 + warp] = (uint32_t)fminf(t * t / (float)x.K, 0x1p29f) + 1u;     // (the magnitudes may add up to infinity)
                next_sums[m0 + warp] = 0u;
            }
        }
    }
    __syncthreads();
    // thread -> frame i, half hh of a group of 32 positions: 16 values, one chunk of each digit row
    const int i = threadIdx.x & 7, hh = (threadIdx.x >> 3) & 1;
    const dense::Scale scale(exps[i]);
    uint8_t* dst0 = img + im.digits + ((size_t)blockIdx.x * (3 * digit::GRAN) + i) * 16;
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
    const uint8_t* img;
    const float* in_scales;      // 2^-e per frame
    const uint32_t* in_sums;     // per frame, in the image of a chain
    uint32_t* spare_sums;        // to be cleared, or nullptr
    const float* scale; const float* shift;
    Affine next;                 // of the layer that reads the digits handed on
    int hardtanh;                // (not SIGMOID) 0: no activation
    int K;
    float* Y; int ldy;
    uint8_t* img_out;            // image of the layer that consumes the outputs, or nullptr
    int img_out_kind;            //   0: digits; 1: two fp16 terms, blocks of 256 frames (out_gemm_f32_tc.cu)
    uint32_t* out_sums;          // of that image (digits)
};

// (What is handed on is no template argument: the layers of a network then run the same code, which the SMs still hold from one
// launch to the next; 517 frames, six layers, 100.2 us, with a kernel per kind 101.6.)
template <bool SIGMOID>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(digit::THREADS, 1)
signw_digit_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ dense::Work w, const __grid_constant__ Args g,
                   TcStatus status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + dense::RING_BYTES;
    dense::Bars* bars = reinterpret_cast<dense::Bars*>(staging + digit::EPI_WARPS * STAGING);
    volatile int* abort_flag = &bars->wait.abort;
    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const bool digits_out = g.img_out && g.img_out_kind == 0;
    const uint32_t ring = smem_u32(smem);
    const uint32_t tmem = dense::set_up(bars, status, warp);

    if (warp >= digit::PROD_WARP0) {
        dense::widen_bits<false>(w, g.Wp, g.ldwp, bars, tmem, rank, warp, lane);
    } else if (warp == digit::COPY_WARP) {
        // the image is the output of the kernel before this one in the stream: wait until that kernel has
        // completed and its writes are visible (the weights do not depend on it)
        pdl_wait();
        if (lane == 0) dense::copy_digits(w, &map, ring, bars, rank);
    } else if (warp == BOUNDS_WARP) {
        if (digits_out && blockIdx.x == 0) {
            const UnitBounds b(g.next, lane, 32);
            if (lane == 0) b.store(g.img_out);
        }
    } else if (warp >= digit::EPI_WARPS) {
        if (rank == 0 && warp <= digit::MMA_WARP2) dense::issue(w, ring, bars, tmem, warp - digit::MMA_WARP);
    } else {
        // ---------------- epilogue: thread = one unit (tensor-memory lane); of a tile's frames warps 0-3 take the
        // first half, warps 4-7 the second
        pdl_wait();
        const int M = w.b_rows, N = w.a_rows;
        const int grans = w.n / (3 * digit::GRAN), per = (grans + 1) >> 1;
        const int g0 = (warp >> 2) * per, ng = grans - g0 < per ? grans - g0 : per;
        const int nb = w.nb();
        uint8_t* mine = staging + warp * STAGING;
        float* rs = reinterpret_cast<float*>(mine);      // frame scales of the input (2^-e) ...
        float* os = rs + 32;                             // ... and of the digits handed on (2^e)
        int* squares = reinterpret_cast<int*>(os + 32);  // of the high digits handed on: eight parts per frame
        const Image im(M, N, true);                      // of the digits handed on
        const UnitBounds bounds = digits_out ? UnitBounds(g.img) : UnitBounds{0u, 0u, 0u};
        const int half_off = ((lane & 15) >> 2) * 16 + (lane & 3) * 4 + (lane >> 4) * 2;     // of this unit in the fp16 image
        // byte transpose between the lanes l, l + 8, l + 16, l + 24: selectors of the two exchanges
        const uint32_t sel16 = lane & 16 ? 0x3276u : 0x5410u, sel8 = lane & 8 ? 0x3715u : 0x6240u;
        int tl = 0;
        for (digit::Tiles t(w); t.left > 0; t.next(), ++tl) {
            const int n0 = t.a * (2 * digit::ROWS) + rank * digit::ROWS + (warp & 3) * 32, n = n0 + lane;
            const int f0 = t.b * nb + g0 * digit::GRAN;
            const bool unit = n < N;
            const float sc = (g.scale && unit) ? __ldg(g.scale + n) : 1.0f;
            const float sh = (g.shift && unit) ? __ldg(g.shift + n) : 0.0f;
            __syncwarp();
            // sc and the scale of the first frame, the scale of its digits; these serve all frames of this warp when they have the
            // same scales, as they have in a chain whose outputs are not all small
            float scr, o0;
            bool same_in, same_out;
            {
                const int f = f0 + lane;
                const bool one = n0 == 0 && f < M && lane < ng * digit::GRAN;     // of all warps that work on a frame
                float r = f < M ? __ldcg(g.in_scales + f) : 0.f, o = 0.f;
                const uint32_t word = g.in_sums && f < M ? __ldcg(g.in_sums + f) : 0u;
                if (word & kNaNOutput) r = __int_as_float(0x7FC00000);
                rs[lane] = r;
                if (digits_out) {
                    const int e = bounds.exponent(magnitude_bound(r, word & ~kNaNOutput, g.K), SIGMOID);
                    o = dense::power_of_two(e);
                    os[lane] = o;
                    if (one) {
                        reinterpret_cast<float*>(g.img_out + im.scales)[f] = dense::power_of_two(-e);
                        g.spare_sums[f] = 0u;
                    }
                }
                const float r0 = __shfl_sync(0xFFFFFFFFu, r, 0);
                o0 = __shfl_sync(0xFFFFFFFFu, o, 0);
                scr = sc * r0;                           // fma(sc, S r, sh) = fma(sc r, S, sh) as long as sc r is exact
                const bool exact = sc == 0.f || (fabsf(scr) >= FLT_MIN && fabsf(scr) <= FLT_MAX);
                const bool none = f >= M || lane >= ng * digit::GRAN;
                same_in = __all_sync(0xFFFFFFFFu, exact && (none || r == r0));
                same_out = __all_sync(0xFFFFFFFFu, none || o == o0);
            }
            __syncwarp();
            const int b = tl & 1;
            if (!warp_wait_relaxed(smem_u32(&bars->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane)) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * w.n + g0 * 3 * digit::GRAN);
            const bool any = f0 < M && n0 < N;                      // uniform over the warp
            if (any) {
                uint32_t d[4][8];
                digit::load_granule(taddr, 3, d);
#pragma unroll 1
                for (int gi = 0; gi < ng; ++gi) {
                    tmem_ld_wait();
                    float S[8], y[8];
#pragma unroll
                    for (int i = 0; i < 8; ++i) S[i] = fmaf(digit::high_part((int)d[2][i]), 65536.0f, digit::low_part((int)d[0][i], (int)d[1][i]));
                    if (gi + 1 < ng) digit::load_granule(taddr + (uint32_t)(gi + 1) * 24, 3, d);
                    if (same_in) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = fmaf(scr, S[i], sh);
                    } else {
                        const float4 ra = reinterpret_cast<const float4*>(rs)[2 * gi], rb = reinterpret_cast<const float4*>(rs)[2 * gi + 1];
                        const float r[8] = {ra.x, ra.y, ra.z, ra.w, rb.x, rb.y, rb.z, rb.w};
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = fmaf(sc, S[i] * r[i], sh);
                    }
                    if (SIGMOID) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = 1.0f / (1.0f + expf(-y[i]));
                    } else if (g.hardtanh) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) y[i] = fminf(fmaxf(y[i], -1.0f), 1.0f);
                    }
                    const int f = f0 + gi * digit::GRAN;
                    if (g.Y && unit) {
                        float* dst = g.Y + (size_t)f * g.ldy + n;
#pragma unroll
                        for (int i = 0; i < 8; ++i, dst += g.ldy)
                            if (f + i < M) *dst = y[i];
                    }
                    if (digits_out && f < M) {
                        // digits of the 8 frames, byte q of word i; four frames at a time: bytes gathered per digit,
                        // transposed over the four lanes whose units are neighbours in the image, stored as words
                        uint32_t v[8];
                        if (same_out) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) y[i] *= o0;
                        } else {
                            const float4 oa = reinterpret_cast<const float4*>(os)[2 * gi], ob = reinterpret_cast<const float4*>(os)[2 * gi + 1];
                            const float o[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
#pragma unroll
                            for (int i = 0; i < 8; ++i) y[i] *= o[i];
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            if (SIGMOID) y[i] = fmaxf(y[i], kNaNDigits);      // (a hardtanh unit gives -1 for a NaN)
                            v[i] = unit ? digit::digits3(__float2int_rn(y[i])) : 0u;
                        }
                        uint8_t* dst = g.img_out + im.digits + ((size_t)(2 * (n0 >> 5) + ((lane >> 2) & 1)) * im.rows + (size_t)(f / digit::GRAN) * 24 + (lane >> 3)) * 16 + (lane & 3) * 4;
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
                                if (q == 2) squares[gi * 64 + h * 32 + lane] = SIGMOID && (x & 0x80808080u) ? kNaNSquare : __dp4a((int)x, (int)x, 0);     // frame 4 h + lane / 8
                            }
                    } else if (g.img_out && !digits_out) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            const float v = unit ? y[i] : 0.f;
                            const __half hi = __float2half_rn(v), lo = __float2half_rn(v - __half2float(hi));
                            uint8_t* p = mine + 128 + (gi * digit::GRAN + i) * 64 + half_off;
                            *reinterpret_cast<__half*>(p) = hi;
                            *reinterpret_cast<__half*>(p + 2048) = lo;
                        }
                    }
                }
            }
            digit::release_acc(bars, b, lane);
            if (digits_out && any) {
                // of the eight parts of a frame's sum
                __syncwarp();
                const int4 a = reinterpret_cast<const int4*>(squares)[2 * lane], c = reinterpret_cast<const int4*>(squares)[2 * lane + 1];
                const int sum = (a.x + a.y) + (a.z + a.w) + (c.x + c.y) + (c.z + c.w);
                if (lane < ng * digit::GRAN && f0 + lane < M) {
                    if (sum >= kNaNSquare) atomicOr(g.out_sums + f0 + lane, kNaNOutput);
                    else atomicAdd(g.out_sums + f0 + lane, (uint32_t)sum);
                }
            }
            if (any && g.img_out && !digits_out) {
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
    const Image im(M, K, false);
    return im.scales + (size_t)(im.rows / 3) * sizeof(float);
}

// Layer `pos` of a chain reads image pos (in the place of pos % 2) and writes image pos + 1.  The sums of image i are in array
// (i / 2) % 2 of its place; they are zero when it is written because the reader of image i - 2 cleared them -- or, for the
// first image that a layer writes, the kernel that wrote the chain's input.
int launch_signw_digit(const RealGemmArgs& r, void* workspace, bool image_ready, void* out_image, int out_kind, int pos, int* clear,
                       int clear_words, cudaStream_t st) {
    const bool digits_out = out_image && out_kind == 0;
    auto kern = r.act == BNN_ACT_SIGMOID ? signw_digit_kernel<true> : signw_digit_kernel<false>;
    const int sms = device_sm_count();
    if (sms < 2 || !ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM_BYTES)) return BNN_ERR_CUDA;
    const TcStatus status = tc_status();
    if (!status.word) return BNN_ERR_CUDA;
    uint8_t* img = static_cast<uint8_t*>(workspace);
    uint8_t* out = static_cast<uint8_t*>(out_image);
    const Image im(r.M, r.K, image_ready || digits_out);
    auto sums = [&](uint8_t* base, int which) { return reinterpret_cast<uint32_t*>(base + im.sums(which)); };
    // (when the kernel before this one in the stream already wrote the image -- the layer that produced
    // these activations -- there is nothing to convert)
    if (!image_ready) {
        const bool vec = (r.lda % 4 == 0) && aligned16(r.Af) && (r.splice_dim % 4 == 0);
        const Frames x{r.Af, r.lda, r.M, r.K, r.splice_dim, r.splice_left, vec};
        const size_t staged = (size_t)digit::GRAN * staged_pitch(r.K) * sizeof(float);
        const int blocks = ceil_div(r.M, digit::GRAN) + (digits_out ? 1 : 0);
        const Affine units{r.scale, r.shift, r.N};
        uint32_t *first = digits_out ? sums(img, 0) : nullptr, *next = digits_out ? sums(out, 0) : nullptr;
        if (staged <= STAGED_MAX) x_digits_kernel<true><<<blocks, 256, staged, st>>>(x, img, first, next, units, clear, clear ? clear_words : 0);
        else x_digits_kernel<false><<<blocks, 256, 0, st>>>(x, img, first, next, units, clear, clear ? clear_words : 0);
    }
    const int steps = ceil_div(r.K, 32), pairs = sms / 2;
    const dense::Work w{r.N, r.M, dense::tile_rows(r.N, r.M, steps, pairs), 3, steps, 0};
    const Args a{r.Bb, r.ldb, img, reinterpret_cast<const float*>(img + im.scales), image_ready || digits_out ? sums(img, pos / 2) : nullptr,
                 digits_out ? sums(img, pos / 2 + 1) : nullptr, r.scale, r.shift,
                 Affine{r.next_scale, r.next_shift, r.next_N}, r.act == BNN_ACT_HARDTANH, r.K, r.Y, r.ldy, out, out_kind, digits_out ? sums(out, (pos + 1) / 2) : nullptr};
    CUtensorMap map;
    if (!encode_digit_map(&map, img + im.digits, im.rows, im.chunks, w.n / 2, digit::KB / 16)) return BNN_ERR_CUDA;
    const long long tiles = dense::tile_count(r.N, r.M, w.n);
    if (launch_pdl(kern, dim3(2 * (int)(tiles < pairs ? tiles : pairs)), dim3(digit::THREADS), SMEM_BYTES, st, map, w, a, status) != cudaSuccess)
        return BNN_ERR_CUDA;
    return launch_status();
}

}  // namespace bnn
