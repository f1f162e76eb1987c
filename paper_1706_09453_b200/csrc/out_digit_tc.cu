// Real-valued top layer on +-1 (or 0/1) activations, on the tensor cores with exact integer sums:
//   z[m][c] = sum_h Wout[c][h] * a[m][h] + b[c].
//
// The weights are static, so they are prepared once (bnn_output_prepare_digits): as fixed-point numbers of a scale of each class's
// own, written as byte digits in the order the tensor core reads shared memory.  Four forms, of which the device chooses one for the whole matrix
// (out_range_kernel) and the GEMM reads the choice from the image:
//   pairs   sums and differences of pairs of weights in three digits (digit_gemm.cuh): half the tensor-core time of the others, for matrices of which it is as precise;
//   three   every weight in three digits (digit_dense.cuh), about 23 bits relative to the class's largest weight;
//   four    every weight in four digits (31 bits), where some class's largest weight is more than 16 times its mean magnitude.  Up to that,
//           even if all H roundings of three digits, each at most 1.01 * 2^-24 of the largest weight, add up, a logit is within 1.01 * 2^-20 of sum |w|;
//   pairs, four   the same on pairs, for 2000 and more units, where the tensor core counts: single weights -> pairs, us, 16384 x 4000 x 3072 517 -> 431, 8192 x 3400 x 2048
//           138 -> 120; but 8336 x 1370 x 416 33 -> 36, 4844 x 678 x 492 14 -> 18.
//
// The GEMM runs on CTA pairs, frames on the M side (tensor-memory lane = frame), class digits on the N side: a tile
// is 256 frames x 128 (64, 32) classes on pairs, x 64 or 32 (48, 24) else.  The epilogue transposes through shared memory so that a store covers
// 32 consecutive classes of a frame.  With (0,1) activations, h = (1 + sigma) / 2: the sum over all pairs of a class,
// prepared with the image, is added.
//
// Bound by what L2 delivers (at the full rate of the sparse MMAs a CTA would take 64 bytes of digits per clock; 8192 x 3400 x 2048 takes 740 MB,
// 35 bytes per clock and SM) and by the epilogue's reads of the accumulators.  Measured on B200, single weights in three digits -> pairs, 3400 classes x 2048 units:
// 8192 frames 109 -> 73 us (the MMAs take 40), in (0,1) 102 -> 76, 20 frames 9.2 -> 7.7; 3401 classes 110 -> 86; 731 frames x 3307 19 -> 16.4;
// 16384 x 4000 x 3072 360 -> 250.
#include "bnn_common.cuh"
#include "digit_dense.cuh"
#include "digit_gemm.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

using namespace tc;
namespace dense = digit::dense;

enum Form { kPairs = 0, kFour = 1, kThree = 2, kPairsFour = 3 };
constexpr int kPairsFourMin = 2000;      // units
__host__ __device__ constexpr bool in_pairs(int form) { return form == kPairs || form == kPairsFour; }
__host__ __device__ constexpr int digits_of(int form) { return form == kFour || form == kPairsFour ? 4 : 3; }

// The image: [Header, 256 bytes][largest magnitude per class][half of the largest |w1| + |w2| per class][scale per class][sum over all pairs per class][digits].
struct Header {
    int form;                         // what GEMM and log-softmax go by
    int outlier;                      // out_range_kernel's findings
    long long balance;
};
struct DigitImage {
    size_t mx, top, scales, totals, digits, bytes;   // offsets; total size
    int cpad;
    int rows;                         // digit rows per chunk of 16 positions: room for four digits
    int chunks;
};
DigitImage digit_image(int C, int H) {
    DigitImage d;
    d.cpad = ceil_div(C, digit::GRAN) * digit::GRAN;
    d.mx = 256;
    d.top = d.mx + (size_t)d.cpad * sizeof(float);
    d.scales = d.top + (size_t)d.cpad * sizeof(float);
    d.totals = (d.scales + (size_t)d.cpad * sizeof(float) + 255) & ~size_t(255);
    d.digits = (d.totals + (size_t)d.cpad * sizeof(long long) + 255) & ~size_t(255);
    d.rows = 4 * d.cpad;
    d.chunks = 2 * ceil_div(H, 32);
    d.bytes = d.digits + (size_t)d.chunks * d.rows * 16;
    return d;
}

constexpr int STAGING_PITCH = 33;
// Staging of the epilogue warps: 32 x 33 logits of each, or a block of 32 x 32 of each (1 KB aligned); then of each the scales and biases of its 32 classes and, for activations in (0,1),
// the high and low parts of their sums over all pairs.
constexpr int BLOCK = 32 * 32 * 4, ROWS_BYTES = 32 * STAGING_PITCH * 4, CONSTS = 4 * 32 * 4;
constexpr int STAGING = digit::EPI_WARPS * (ROWS_BYTES + CONSTS);
static_assert(dense::RING_BYTES == digit::RING_BYTES, "either ring fits");
constexpr int SMEM_BYTES = digit::RING_BYTES + STAGING + (int)sizeof(digit::Bars) + (int)sizeof(dense::Bars) + 1024;
constexpr int kFollowGroupMin = 2 * digit::ROWS;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

// ---- one-time preparation of the weights -------------------------------------------------
constexpr double kTop = 8355711.0;       // 0x7F7F7F, the largest balanced number of three digits
// What a unit of a class's fixed-point numbers stands for.  With three digits any fp32 number will do, because the numbers are prepared in
// double precision, and the smallest that keeps the largest within range is the most precise.  (Pairs: the margin is that of the
// rounding of `half`.)  With four, where the rounding of the result is all that counts, a power of two, which costs none.
__device__ __forceinline__ float class_scale(int form, float mx, float half) {
    const double top = in_pairs(form) ? 2.0 * (double)half : (double)mx;
    if (!(top > 0.0)) return (float)(top == 0.0 ? 1.0 : top);         // no weights; a NaN
    if (digits_of(form) == 3) return __double2float_ru(top / (form == kPairs ? kTop - 11.0 : kTop));
    int e;
    frexp(top / 2e9, &e);
    return (float)ldexp(1.0, e > -149 ? e : -149);
}

// One warp per class: mx[c] = its largest magnitude and tops[c] = half of the largest |W[c][k]| + |W[c][k + 16]| of its pairs, NaNs for a row with an infinity or a NaN;
// outlier is set when some class needs four digits.  balance comes out above zero when pairs are less precise than single weights rounded to multiples of the power of two
// at which the row's largest fits: a class's mean square of the
// error of a sum, over that, is half the squared ratio of the units (half as many
// roundings), between 1/8 and 2, and the fourth powers of these, so that classes above 1 count for more than those below, are compared with 1 on the mean.
// Pairs win on rows of N(0, 1) numbers (rms 0.74 - 0.80), whose largest pair is some 1.4 times the largest number; on rows that fill their range evenly it is
// twice that, and they lose where the largest number is just below a power of two (uniform in +-0.99: 1.2).
__global__ void out_range_kernel(const float* __restrict__ W, int ldw, int C, int H, float* __restrict__ mx, float* __restrict__ tops, Header* __restrict__ head) {
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= C) return;
    float sum = 0.f, half = 0.f;
    uint32_t top = 0u;   // largest magnitude as bits: orders NaN above infinity above every number
    for (int h0 = 0; h0 < H; h0 += 32) {
        const int h = h0 + lane;
        const float a = h < H ? fabsf(W[(size_t)c * ldw + h]) : 0.f;
        sum += a;
        top = max(top, __float_as_uint(a));
        half = fmaxf(half, digit::half_sum(a, __shfl_xor_sync(0xFFFFFFFFu, a, 16)));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        half = fmaxf(half, __shfl_xor_sync(0xFFFFFFFFu, half, o));
        top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
    }
    if (lane == 0) {
        const float m = __uint_as_float(top);
        const bool finite = top < 0x7F800000u;
        mx[c] = finite ? m : __int_as_float(0x7FC00000);
        tops[c] = finite ? half : __int_as_float(0x7FC00000);
        if ((float)H * m > 16.0f * sum) atomicOr(&head->outlier, 1);
        if (finite && half > 0.f) {
            const int pairs = (H >> 5) * 16 + ((H & 31) < 16 ? H & 31 : 16);
            const double units = ldexp((double)class_scale(kPairs, m, half), digit::scale_exponent(m));
            double r = 0.999 * units * units * pairs / H;       // (the margins of the two scales differ)
            r *= r;
            atomicAdd(reinterpret_cast<unsigned long long*>(&head->balance), (unsigned long long)__double2ll_rn((r * r - 1.0) * 1048576.0));
        }
    }
}

// One thread writes the digits of 16 positions (one chunk of each digit row) of a class: eight pairs, their sums and differences, or 16 weights.
__global__ void out_digits_kernel(const float* __restrict__ W, int ldw, int C, int H, int Cpad8, int rows, int chunks,
                                  const float* __restrict__ mx, const float* __restrict__ tops, Header* head, float* __restrict__ scales,
                                  unsigned long long* __restrict__ totals, uint8_t* __restrict__ img) {
    const int form = head->outlier ? (H >= kPairsFourMin ? kPairsFour : kFour) : head->balance > 0 ? kThree : kPairs, nd = digits_of(form);
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)chunks * Cpad8) return;
    if (i == 0) head->form = form;
    const int c = (int)(i % Cpad8), ch = (int)(i / Cpad8);
    const float scale = c < C ? class_scale(form, mx[c], tops[c]) : 0.f;
    const bool some = scale > 0.f;               // (not for a NaN)
    if (ch == 0) scales[c] = scale;
    auto weight = [&](int k) { return some && k < H ? (double)W[(size_t)c * ldw + k] : 0.0; };
    auto digits = [&](double x) {
        const int v = some ? __double2int_rn(x / (double)scale) : 0;
        return nd == 4 ? digit::digits4(v) : digit::digits3(v);
    };
    long long total = 0;                         // of the sums of pairs
    uint32_t d[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {                // word x of the chunk
        uint32_t v[4];
        if (in_pairs(form)) {                    // two pairs
#pragma unroll
            for (int y = 0; y < 2; ++y) {
                // the t, w and q = y of digit::image_byte(half, w, t, q) = 16 (ch % 4) + 4 x + 2 y
                const bool half = (ch & ~3) + 2 == chunks;
                const int t = half ? 4 * (x & 1) + 2 * (ch & 1) + (x >> 1) : 4 * (ch & 1) + 2 * (x >> 1) + ((ch >> 1) & 1);
                const int k = (ch >> 2) * 64 + (half ? 0 : 32 * (x & 1)) + 8 * y + t;
                const double w1 = weight(k), w2 = weight(k + 16);
                v[2 * y] = digits(w1 + w2);
                v[2 * y + 1] = digits(w1 - w2);
                if (some) total += __double2int_rn((w1 + w2) / (double)scale);
            }
        } else {                                 // byte 4 x + j, see digit_dense.cuh
#pragma unroll
            for (int j = 0; j < 4; ++j) v[j] = digits(weight((ch >> 1) * 32 + (ch & 1) * 4 + x + 8 * j));
        }
        d[0][x] = digit::gather_bytes<0>(v[0], v[1], v[2], v[3]);
        d[1][x] = digit::gather_bytes<1>(v[0], v[1], v[2], v[3]);
        d[2][x] = digit::gather_bytes<2>(v[0], v[1], v[2], v[3]);
        d[3][x] = digit::gather_bytes<3>(v[0], v[1], v[2], v[3]);
    }
    uint8_t* dst = img + ((size_t)ch * rows + (size_t)(c / digit::GRAN) * digit::GRAN * nd + c % digit::GRAN) * 16;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < nd) *reinterpret_cast<uint4*>(dst + (size_t)q * digit::GRAN * 16) = make_uint4(d[q][0], d[q][1], d[q][2], d[q][3]);
    if (total != 0) atomicAdd(totals + c, (unsigned long long)total);
}

// ---- the GEMM ---------------------------------------------------------------------------
struct Logits {
    float* Z; int ldz;
    int M, C;
    const float* scales; const float* bias;
    const long long* totals;
    int* done;
};

// This warp's logits of a tile of 256 frames are stored: count it in for these (release).
__device__ __forceinline__ void count_in(int* done, int tile) {
    __threadfence();
    __syncwarp();
    if ((threadIdx.x & 31) == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(done + tile) : "memory");
}

// What a class's sums are multiplied by, and what is added.  PAIRS01: pairs on activations in (0,1), where the class's sum over all pairs comes in, as
// 65536 high + low: the high part is added to that of the products, which costs nothing; the low part goes with the bias.  (Four digits: 2^24 high + low, which is
// added to the low part.)
template <bool PAIRS01>
struct Class {
    float scale, bias;
    int high, low;
    __device__ __forceinline__ Class(const Logits& o, int c, bool some, int nd) : high(0), low(0) {
        some = some && c < o.C;
        scale = some ? __ldg(o.scales + c) * (PAIRS01 ? 0.5f : 1.0f) : 0.f;
        bias = o.bias && some ? __ldg(o.bias + c) : 0.f;
        if (PAIRS01) {
            const long long total = some ? __ldg(o.totals + c) : 0;
            const int bits = nd == 3 ? 16 : 24;
            high = (int)((total + (1ll << (bits - 1))) >> bits);
            low = (int)(total - ((long long)high << bits));
            if (nd == 3) bias = fmaf((float)low, scale, bias);
        }
    }
};
// Where a warp keeps that of its 32 classes, lane = class.
struct Classes {
    float* consts;
    uint32_t smem;
    __device__ __forceinline__ Classes(uint8_t* staging, int warp)
        : consts(reinterpret_cast<float*>(staging + digit::EPI_WARPS * ROWS_BYTES + warp * CONSTS)), smem(smem_u32(consts)) {}
    // `all`, or the sums only.
    template <bool PAIRS01>
    __device__ __forceinline__ void put(const Class<PAIRS01>& c, bool all) {
        const int lane = threadIdx.x & 31;
        __syncwarp();
        if (all) {
            consts[lane] = c.scale;
            consts[32 + lane] = c.bias;
        }
        if (PAIRS01) {
            reinterpret_cast<int*>(consts)[64 + lane] = c.high;
            reinterpret_cast<int*>(consts)[96 + lane] = c.low;
        }
        __syncwarp();
    }
    __device__ __forceinline__ static void get(uint32_t at, float (&v)[8]) {
        const uint4 a = lds128u(at), b = lds128u(at + 16);
        v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y); v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
        v[4] = __uint_as_float(b.x); v[5] = __uint_as_float(b.y); v[6] = __uint_as_float(b.z); v[7] = __uint_as_float(b.w);
    }
    // The sums of granule g, 65536 high + low, rounded once.
    template <bool PAIRS01>
    __device__ __forceinline__ void sums3(const uint32_t (&d)[4][8], int g, float (&z)[8]) const {
        float t[8] = {};
        if (PAIRS01) get(smem + 256 + g * 32, t);
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = fmaf(digit::high_part((int)d[2][i], __float_as_int(t[i])), 65536.0f, digit::low_part((int)d[0][i], (int)d[1][i]));
    }
    // The same with four digits.
    template <bool PAIRS01>
    __device__ __forceinline__ void sums4(const uint32_t (&d)[4][8], int g, float (&z)[8]) const {
        float t[8] = {}, u[8] = {};
        if (PAIRS01) {
            get(smem + 256 + g * 32, t);
            get(smem + 384 + g * 32, u);
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = digit::join4((int)d[0][i], (int)d[1][i], (int)d[2][i], (int)d[3][i], __float_as_int(t[i]), __float_as_int(u[i]));
    }
    // Its logits, scale * (65536 high + low) + bias, of which the low part and the bias are rounded first, and the sum once.
    template <bool PAIRS01>
    __device__ __forceinline__ void logits3(const uint32_t (&d)[4][8], int g, float (&z)[8]) const {
        float s[8], b[8], t[8] = {};
        get(smem + g * 32, s);
        get(smem + 128 + g * 32, b);
        if (PAIRS01) get(smem + 256 + g * 32, t);
#pragma unroll
        for (int i = 0; i < 8; ++i)
            z[i] = fmaf(digit::high_part((int)d[2][i], __float_as_int(t[i])), 65536.0f * s[i], fmaf(digit::low_part((int)d[0][i], (int)d[1][i]), s[i], b[i]));
    }
};

// A warp's share of an accumulator, n granules of 8 classes from class c0 on x 32 frames from f0 on (join: a granule's digit sums -> 8 of a frame's sums or, SCALED, logits),
// through shared memory (`mine`, 32 rows of STAGING_PITCH), so that a store covers consecutive classes.  `released` hands the accumulator back.
// Sums are rounded, and again when scale and bias (of the class that a lane stores) are applied here; logits, rounded once, take four more 16-byte loads per granule
// (3-5 % of the kernel).  They are for scales that are no powers of two where there are no biases: with a power of two the second rounding would not be there.
__device__ __forceinline__ int store_lane(int n) { return n > 2 ? threadIdx.x & 31 : threadIdx.x & 15; }     // a frame per store, or two
template <bool SCALED, typename F, typename Released>
__device__ __forceinline__ void store_rows(const Logits& o, float* mine, uint32_t taddr, int n, int nd, int f0, int c0, float scale, float bias, uint64_t pol, F join, Released released) {
    const int lane = threadIdx.x & 31;
    if (f0 < o.M && n > 0) {                            // uniform over the warp
        float* row = mine + lane * STAGING_PITCH;
        const uint32_t width = (uint32_t)(nd * digit::GRAN);
        uint32_t d[4][8];
        digit::load_granule(taddr, nd, d);
#pragma unroll 1
        for (int g = 0; g < n; ++g) {
            tmem_ld_wait();
            float z[8];
            join(d, g, z);
#pragma unroll
            for (int i = 0; i < 8; ++i) row[g * digit::GRAN + i] = z[i];
            if (g + 1 < n) digit::load_granule(taddr + (uint32_t)(g + 1) * width, nd, d);
        }
    }
    released();
    __syncwarp();
    const int cl = store_lane(n), fstep = n > 2 ? 1 : 2, fo = n > 2 ? 0 : lane >> 4;
    if (f0 < o.M && cl < n * digit::GRAN && c0 + cl < o.C) {
        // eight rows of the staging block at a time, so that their loads are in flight together
        float* dst = o.Z + (size_t)(f0 + fo) * o.ldz + c0 + cl;
        const size_t step = (size_t)fstep * o.ldz;
        const float* src = mine + fo * STAGING_PITCH + cl;
        const int left = (o.M - f0 - fo + fstep - 1) / fstep;    // rows of this lane that exist
#pragma unroll 1
        for (int j = 0; j < 32 / fstep; j += 8) {
            float v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                v[i] = src[(j + i) * fstep * STAGING_PITCH];
                if (!SCALED) v[i] = fmaf(v[i], scale, bias);
            }
#pragma unroll
            for (int i = 0; i < 8; ++i, dst += step)
                if (j + i < left) asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(dst), "f"(v[i]), "l"(pol));
        }
    }
    __syncwarp();
}

__device__ __forceinline__ uint64_t keep_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// Pairs, epilogue: thread = one frame (tensor-memory lane); of a tile's classes, or of either part's, warps 0-3 take
// the first half, warps 4-7 the second.  by_blocks (three digits): the logits leave by tile stores (out_map).
template <bool ZO>
__device__ __forceinline__ void pairs_epilogue(const digit::Work& w, const Logits& o, const CUtensorMap* out_map, bool by_blocks, uint8_t* staging,
                                               digit::Bars* bars, uint32_t tmem, int rank, int warp, int lane) {
    volatile int* abort_flag = &bars->wait.abort;
    const bool halved = w.halved();
    const int grans = w.grans(), per = halved ? (grans + 1) >> 1 : grans;
    const int g0 = halved ? (warp >> 2) * per : 0, g1 = g0 + per < grans ? g0 + per : grans;
    float* mine = reinterpret_cast<float*>(staging + warp * ROWS_BYTES);
    const uint32_t block_smem = smem_u32(staging) + warp * BLOCK;
    Classes classes(staging, warp);
    const uint64_t pol = keep_policy();
    uint32_t parities = 0u;                                 // to wait for, of the parts
    for (digit::Tiles t(w); t.left > 0; t.next()) {
        for (int part = halved ? 0 : warp >> 2; part < (halved ? digit::PARTS : (warp >> 2) + 1) && !w.beyond(t.b, part); ++part) {
            const int c0 = ((t.b * digit::PARTS + part) * grans + g0) * digit::GRAN;
            const int n = g1 - g0, cl = store_lane(n);
            // before the wait for the accumulator, which then is read without waiting for these
            const Class<ZO> y(o, c0 + lane, lane < n * digit::GRAN, w.nd);
            const bool scaled = by_blocks || (!o.bias && w.nd == 3);       // (with four digits the scale is a power of two)
            if (ZO || scaled) classes.put(y, scaled);
            const float scale = __shfl_sync(0xFFFFFFFFu, y.scale, cl), bias = __shfl_sync(0xFFFFFFFFu, y.bias, cl);
            const int f0 = t.a * (2 * digit::ROWS) + rank * digit::ROWS + (warp & 3) * 32;
            const bool ok = warp_wait_relaxed(smem_u32(&bars->acc_full[part]), (parities >> part) & 1u, abort_flag, lane);
            parities ^= 1u << part;
            if (!ok) return;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(part * w.n + g0 * digit::GRAN * w.nd);
            if (by_blocks) {
                // 32 frames x 32 classes: a tile store, which drops what lies outside
                uint32_t d[4][8];
                digit::load_granule(taddr, 3, d);
                if (lane == 0) bulk_wait_read<0>();             // the block before has left shared memory
                __syncwarp();
#pragma unroll
                for (int g = 0; g < 4; ++g) {
                    tmem_ld_wait();
                    float z[8];
                    classes.logits3<ZO>(d, g, z);
                    if (g < 3) digit::load_granule(taddr + (uint32_t)(g + 1) * 24, 3, d);
                    else digit::release_acc(bars, part, lane);
#pragma unroll
                    for (int h = 0; h < 2; ++h)
                        sts128(block_smem + lane * 128 + (((g * 2 + h) ^ (lane & 7)) << 4), __float_as_uint(z[4 * h]), __float_as_uint(z[4 * h + 1]),
                               __float_as_uint(z[4 * h + 2]), __float_as_uint(z[4 * h + 3]));
                }
                fence_proxy_async_smem();
                __syncwarp();
                if (lane == 0) {
                    if (f0 < o.M && c0 < o.C) tma_store_2d_hint(out_map, c0, f0, block_smem, pol);
                    bulk_commit();
                    if (o.done) {
                        // this warp's logits of the tile are stored: count it in for the tile's frames (release)
                        bulk_wait<0>();
                        __threadfence();
                        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(o.done + t.a) : "memory");
                    }
                }
            } else {
                auto released = [&] { digit::release_acc(bars, part, lane); };
                if (scaled) store_rows<true>(o, mine, taddr, n, 3, f0, c0, scale, bias, pol, [&](const uint32_t (&d)[4][8], int g, float (&z)[8]) { classes.logits3<ZO>(d, g, z); }, released);
                else if (w.nd == 3) store_rows<false>(o, mine, taddr, n, 3, f0, c0, scale, bias, pol, [&](const uint32_t (&d)[4][8], int g, float (&z)[8]) { classes.sums3<ZO>(d, g, z); }, released);
                else store_rows<false>(o, mine, taddr, n, 4, f0, c0, scale, bias, pol, [&](const uint32_t (&d)[4][8], int g, float (&z)[8]) { classes.sums4<ZO>(d, g, z); }, released);
                if (o.done) count_in(o.done, t.a);
            }
        }
    }
    if (by_blocks && lane == 0) bulk_wait<0>();
}

// Single weights, all roles of a CTA pair.
template <bool ZO>
__device__ __forceinline__ void single_weights(const dense::Work& w, const Logits& o, const CUtensorMap* map, const uint32_t* __restrict__ Hp, int ldhp, uint32_t ring, uint8_t* staging,
                                               dense::Bars* bars, uint32_t tmem, int rank, int warp, int lane) {
    if (warp >= digit::PROD_WARP0) {
        dense::widen_bits<ZO>(w, Hp, ldhp, bars, tmem, rank, warp, lane);
    } else if (warp == digit::COPY_WARP) {
        if (lane == 0) dense::copy_digits(w, map, ring, bars, rank);
    } else if (warp >= digit::EPI_WARPS) {
        if (rank == 0 && warp <= digit::MMA_WARP2) dense::issue(w, ring, bars, tmem, warp - digit::MMA_WARP);
    } else {
        // epilogue: thread = one frame; of a tile's classes warps 0-3 take the first half, warps 4-7 the second
        volatile int* abort_flag = &bars->wait.abort;
        const int grans = w.grans(), per = (grans + 1) >> 1, g0 = (warp >> 2) * per, g1 = g0 + per < grans ? g0 + per : grans;
        float* mine = reinterpret_cast<float*>(staging + warp * ROWS_BYTES);
        Classes classes(staging, warp);
        const uint64_t pol = keep_policy();
        int tl = 0;
        for (digit::Tiles t(w); t.left > 0; t.next(), ++tl) {
            const int c0 = t.b * w.nb() + g0 * digit::GRAN, b = tl & 1;
            const int n = g1 - g0, cl = store_lane(n);
            const Class<false> y(o, c0 + lane, lane < n * digit::GRAN, w.nd);
            const bool scaled = !o.bias && w.nd == 3;        // as above
            if (scaled) classes.put(y, true);
            const float scale = __shfl_sync(0xFFFFFFFFu, y.scale, cl), bias = __shfl_sync(0xFFFFFFFFu, y.bias, cl);
            const int f0 = t.a * (2 * digit::ROWS) + rank * digit::ROWS + (warp & 3) * 32;
            if (!warp_wait_relaxed(smem_u32(&bars->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane)) return;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * w.n + g0 * digit::GRAN * w.nd);
            auto released = [&] { digit::release_acc(bars, b, lane); };
            if (scaled) store_rows<true>(o, mine, taddr, n, 3, f0, c0, scale, bias, pol, [&](const uint32_t (&d)[4][8], int g, float (&z)[8]) { classes.logits3<false>(d, g, z); }, released);
            else if (w.nd == 3) store_rows<false>(o, mine, taddr, n, 3, f0, c0, scale, bias, pol, [&](const uint32_t (&d)[4][8], int g, float (&z)[8]) { classes.sums3<false>(d, g, z); }, released);
            else store_rows<false>(o, mine, taddr, n, 4, f0, c0, scale, bias, pol, [&](const uint32_t (&d)[4][8], int g, float (&z)[8]) { classes.sums4<false>(d, g, z); }, released);
            if (o.done) count_in(o.done, t.a);
        }
    }
}

// ZO: the activation bits stand for (0,1) instead of (-1,+1).
template <bool ZO>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(digit::REG_THREADS, 1)
out_digit_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap single_map, const __grid_constant__ CUtensorMap out_map, int by_blocks,
                 const uint32_t* __restrict__ Hp, int ldhp, const int* __restrict__ form, digit::Work w, dense::Work single, const __grid_constant__ Logits o,
                 TcStatus status) {
    extern __shared__ uint8_t smem_raw[];
    // A kernel launched behind this one with programmatic stream serialisation (the log-softmax that
    // follows the frame tiles as they complete) may move onto the SMs once every CTA has got this far.
    pdl_trigger();
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + digit::RING_BYTES;
    digit::Bars* bars = reinterpret_cast<digit::Bars*>(staging + STAGING);
    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const uint32_t ring = smem_u32(smem);
    dense::Bars* more = reinterpret_cast<dense::Bars*>(bars + 1);
    if (warp == 1) {                 // beside those of the pairs: which form it is stands in memory that the kernel before may be writing
        dense::init_bars(more, lane, 32);
        if (lane == 0) wait_state_init(&more->wait, status);
        mbar_init_fence();
    }
    const uint32_t tmem = digit::set_up(bars, status, warp, w.halved());
    pdl_wait();      // (returns at once in a plain launch) the set-up overlaps the end of the kernel before
                     // this one: 2 us of 35 on 256 frames of the small network
    const int f = __ldg(form);

    w.nd = single.nd = digits_of(f);
    if (!in_pairs(f)) {
        single_weights<ZO>(single, o, &single_map, Hp, ldhp, ring, staging, more, tmem, rank, warp, lane);
        if (more->wait.abort) bars->wait.abort = 1;
    } else if (warp >= digit::PROD_WARP0) {
        digit::widen_bits(w, Hp, ldhp, bars, tmem, rank, warp, lane);
    } else if (warp == digit::COPY_WARP) {
        if (lane == 0) digit::copy_digits(w, &map, ring, bars, rank);
    } else if (warp >= digit::EPI_WARPS) {
        if (rank == 0 && warp <= digit::MMA_WARP2) digit::issue(w, ring, bars, tmem, warp - digit::MMA_WARP);
    } else {
        pairs_epilogue<ZO>(w, o, &out_map, by_blocks && w.nd == 3, staging, bars, tmem, rank, warp, lane);
    }
    digit::tear_down(bars, status, warp, tmem);
}

int out_tile_rows(int M, int C, int H) {
    return digit::tile_rows(M, C, ceil_div(H, digit::GROUP), device_sm_count() / 2, C % 4 == 0);
}
int single_tile_rows(int M, int C, int H) {
    return dense::tile_rows(M, C, ceil_div(H, 32), device_sm_count() / 2);
}

}  // namespace

size_t out_digits_bytes(int C, int H) { return digit_image(C, H).bytes; }

int launch_out_prepare_digits(const float* W, int ldw, int C, int H, void* image, cudaStream_t st) {
    uint8_t* img = static_cast<uint8_t*>(image);
    const DigitImage d = digit_image(C, H);
    Header* head = reinterpret_cast<Header*>(img);
    float* mx = reinterpret_cast<float*>(img + d.mx);
    float* tops = reinterpret_cast<float*>(img + d.top);
    auto* totals = reinterpret_cast<unsigned long long*>(img + d.totals);
    if (cudaMemsetAsync(head, 0, sizeof(Header), st) != cudaSuccess) return BNN_ERR_CUDA;
    if (cudaMemsetAsync(totals, 0, (size_t)d.cpad * sizeof(long long), st) != cudaSuccess) return BNN_ERR_CUDA;
    out_range_kernel<<<ceil_div(C, 8), 256, 0, st>>>(W, ldw, C, H, mx, tops, head);
    const long long items = (long long)d.chunks * d.cpad;
    out_digits_kernel<<<(unsigned)((items + 255) / 256), 256, 0, st>>>(W, ldw, C, H, d.cpad, d.rows, d.chunks, mx, tops, head,
                                                                         reinterpret_cast<float*>(img + d.scales), totals, img + d.digits);
    return launch_status();
}

// With no more tiles than CTA pairs every tile ends at about the same time: nothing for a following kernel to
// overlap with (measured: 1-2 % slower than two launches in a row on 256 frames).
bool out_digit_can_be_followed(int M, int C, int H) {
    return M > kFollowGroupMin && digit::tile_count(M, C, out_tile_rows(M, C, H)) > device_sm_count() / 2;
}
FollowArgs out_digit_follow(const void* image, int M, int C, int H, int* done) {
    const int n = out_tile_rows(M, C, H);
    // the epilogue warps of every tile or part, by Form
    auto parts = [&](int rows, int nd) { return ceil_div(C, rows / (digit::GRAN * nd) * digit::GRAN) * digit::EPI_WARPS; };
    const int per = n == digit::MAX_N ? 2 : 1, s = single_tile_rows(M, C, H);
    return FollowArgs{done, {parts(n, 3) * per, parts(s, 4) * 2, parts(s, 3) * 2, parts(n, 4) * per},
                      &static_cast<const Header*>(image)->form, 2 * digit::ROWS};
}

int launch_out_digit(const uint32_t* Hp, int ldhp, const void* image, const float* bias,
                     int M, int C, int H, float* Z, int ldz, int zo, int* done, cudaStream_t st) {
    const int sms = device_sm_count();
    auto kern = zo ? out_digit_kernel<true> : out_digit_kernel<false>;
    if (sms < 2 || !ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM_BYTES)) return BNN_ERR_CUDA;
    const uint8_t* img = static_cast<const uint8_t*>(image);
    const DigitImage d = digit_image(C, H);
    const TcStatus status = tc_status();
    if (!status.word) return BNN_ERR_CUDA;
    const digit::Work w{M, C, out_tile_rows(M, C, H), 3, ceil_div(H, digit::GROUP), ceil_div(H, 32) & 1, 1};
    const dense::Work single{M, C, single_tile_rows(M, C, H), 3, ceil_div(H, 32), 1};
    CUtensorMap map, single_map;
    if (!encode_digit_map(&map, img + d.digits, d.rows, d.chunks, w.n / 2, digit::KB / 16) ||
        !encode_digit_map(&single_map, img + d.digits, d.rows, d.chunks, single.n / 2, digit::KB / 16)) return BNN_ERR_CUDA;
    // whole blocks of 32 classes per warp, in rows that a tile store can take
    const int by_blocks = w.n >= digit::MAX_N / 2 && C % 4 == 0 && ldz % 4 == 0 && aligned16(Z);
    CUtensorMap out_map = map;
    if (by_blocks && !encode_int32_map(&out_map, reinterpret_cast<int32_t*>(Z), ldz, M, C)) return BNN_ERR_CUDA;
    const long long some = digit::tile_count(M, C, w.n), more = dense::tile_count(M, C, single.n), tiles = some > more ? some : more;
    const int pairs = sms / 2;
    const dim3 grid(2 * (int)(tiles < pairs ? tiles : pairs)), block(digit::THREADS);
    const Logits o{Z, ldz, M, C, reinterpret_cast<const float*>(img + d.scales), bias, reinterpret_cast<const long long*>(img + d.totals), done};
    const int* form = &reinterpret_cast<const Header*>(img)->form;
    if (!done) {
        const cudaError_t e = launch_pdl(kern, grid, block, SMEM_BYTES, st, map, single_map, out_map, by_blocks, Hp, ldhp, form, w, single, o, status);
        return e == cudaSuccess ? launch_status() : BNN_ERR_CUDA;
    }
    // a kernel that follows this one's counters must not start before the kernels that clear them have ended
    kern<<<grid, block, SMEM_BYTES, st>>>(map, single_map, out_map, by_blocks, Hp, ldhp, form, w, single, o, status);
    return launch_status();
}

}  // namespace bnn
