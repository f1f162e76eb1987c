// Real-valued top layer on +-1 (or 0/1) activations, on the tensor cores with exact integer sums:
//   z[m][c] = sum_h Wout[c][h] * a[m][h] + b[c].
//
// The weights are static, so they are prepared once (bnn_output_prepare_digits): sums and differences of pairs of weights as
// fixed-point numbers of a scale of each class's own, written as byte digits in the order the tensor core reads shared memory
// (digit_gemm.cuh).  Three digits (about 23 bits relative to the class's largest weight) as long as every class's
// largest weight is at most 16 times its mean magnitude -- then even if all H / 2 roundings, each at most 1.01 * 2^-23 of
// the largest weight, add up, a logit is within 2^-20 of sum |w| -- and four digits (31 bits) for the whole
// matrix otherwise.  The choice is made on the device and read from the image by the GEMM.
//
// The GEMM runs on CTA pairs, frames on the M side (tensor-memory lane = frame), class digits on the N side: a tile
// is 256 frames x 128 (64, 32) classes.  The epilogue transposes through shared memory so that a store covers
// 32 consecutive classes of a frame.  With (0,1) activations, h = (1 + sigma) / 2: the digit sums of a class over all pairs,
// prepared with the image, are added to the sums before their digits are joined.
//
// Bound by what L2 delivers (at the full rate of the sparse MMAs a CTA would take 64 bytes of digits per clock; it gets about
// 39) and by the epilogue's reads of the accumulators.  Measured on B200 against dense MMAs on one digit per weight (256 frames x 64 classes per tile,
// two accumulators), 3400 classes x 2048 units: 8192 frames 109 -> 74 us (the MMAs take 40), 3000 frames 43 -> 32, 731
// frames (3307 classes) 18.4 -> 17.5, 128 frames 13 -> 11; 32768 frames x 4000 x 3072 688 -> 498 us.
#include "bnn_common.cuh"
#include "digit_gemm.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

using namespace tc;

// The image: [flag, 256 bytes][half of the largest |w1| + |w2| per class][scale per class][digit sums per class][digits].
struct DigitImage {
    size_t top, scales, totals, digits, bytes;   // offsets; total size
    int cpad;
    int rows;                         // digit rows per chunk of 16 positions: room for four digits
    int chunks;
};
DigitImage digit_image(int C, int H) {
    DigitImage d;
    d.cpad = ceil_div(C, digit::GRAN) * digit::GRAN;
    d.top = 256;
    d.scales = d.top + (size_t)d.cpad * sizeof(float);
    d.totals = (d.scales + (size_t)d.cpad * sizeof(float) + 255) & ~size_t(255);
    d.digits = (d.totals + (size_t)d.cpad * 4 * sizeof(int) + 255) & ~size_t(255);
    d.rows = 4 * d.cpad;
    d.chunks = 2 * ceil_div(H, 32);
    d.bytes = d.digits + (size_t)d.chunks * d.rows * 16;
    return d;
}

constexpr int STAGING_PITCH = 33;
// Staging of the epilogue warps: 32 x 33 sums of each; or a block of 32 x 32 logits of each (1 KB aligned), then 32 scales and biases of each.
constexpr int BLOCK = 32 * 32 * 4, CONSTS = 2 * 32 * 4;
constexpr int STAGING = digit::EPI_WARPS * (BLOCK + CONSTS);
static_assert(STAGING >= digit::EPI_WARPS * 32 * STAGING_PITCH * 4, "either use fits");
constexpr int TOTALS = 4 * 32 * 4;       // of each epilogue warp, behind the staging: the digit sums of its classes, for activations in (0,1)
constexpr int SMEM_BYTES = digit::RING_BYTES + STAGING + digit::EPI_WARPS * TOTALS + (int)sizeof(digit::Bars) + 1024;
constexpr int kFollowGroupMin = 2 * digit::ROWS;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

// ---- one-time preparation of the weights -------------------------------------------------
// One warp per class: tops[c] = half of the largest |W[c][k]| + |W[c][k + 16]| of its pairs, a NaN for a row with an infinity or a NaN;
// *flag is set when some class needs four digits.
__global__ void out_range_kernel(const float* __restrict__ W, int ldw, int C, int H, float* __restrict__ tops, int* __restrict__ flag) {
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
        tops[c] = top < 0x7F800000u ? half : __int_as_float(0x7FC00000);
        if ((float)H * __uint_as_float(top) > 16.0f * sum) atomicOr(flag, 1);
    }
}

constexpr float kTopValue = 8355700.0f;       // somewhat below 0x7F7F7F, the largest balanced number of three digits: room for roundings
// What a unit of a class's fixed-point numbers stands for.  With three digits any fp32 number will do, because the numbers are prepared in
// double precision, and the smallest that keeps the largest pair within range is the most precise.  (The margin is that of the
// rounding of `half`.)  With four, where the rounding of the result is all that counts, a power of two, which costs none.
__device__ __forceinline__ float class_scale(float half, int nd) {
    if (!(half > 0.f)) return half == 0.f ? 1.0f : half;      // no weights; a NaN
    if (nd == 3) return __double2float_ru(2.0 * (double)half / (double)kTopValue);
    int e;
    frexp(2.0 * (double)half / 2e9, &e);
    return (float)ldexp(1.0, e > -149 ? e : -149);
}

// One thread writes the digits of 16 positions (one chunk of each digit row) of a class: eight pairs, their sums and differences.
__global__ void out_digits_kernel(const float* __restrict__ W, int ldw, int C, int H, int Cpad8, int rows, int chunks,
                                  const float* __restrict__ tops, const int* __restrict__ flag, float* __restrict__ scales,
                                  int* __restrict__ totals, uint8_t* __restrict__ img) {
    const int nd = *flag ? 4 : 3;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)chunks * Cpad8) return;
    const int c = (int)(i % Cpad8), ch = (int)(i / Cpad8);
    const float scale = c < C ? class_scale(tops[c], nd) : 0.f;
    const bool some = scale > 0.f;               // (not for a NaN)
    if (ch == 0) scales[c] = scale;
    int sums[4] = {0, 0, 0, 0};                  // of the digits of the sums of pairs
    uint32_t d[4][4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {                // word x of the chunk: two pairs
        uint32_t v[4];
#pragma unroll
        for (int y = 0; y < 2; ++y) {
            // the t, w and q = y of digit::image_byte(half, w, t, q) = 16 (ch % 4) + 4 x + 2 y
            const bool half = (ch & ~3) + 2 == chunks;
            const int t = half ? 4 * (x & 1) + 2 * (ch & 1) + (x >> 1) : 4 * (ch & 1) + 2 * (x >> 1) + ((ch >> 1) & 1);
            const int k = (ch >> 2) * 64 + (half ? 0 : 32 * (x & 1)) + 8 * y + t;
            const double w1 = some && k < H ? (double)W[(size_t)c * ldw + k] : 0.0;
            const double w2 = some && k + 16 < H ? (double)W[(size_t)c * ldw + k + 16] : 0.0;
            const int s = some ? __double2int_rn((w1 + w2) / (double)scale) : 0, e = some ? __double2int_rn((w1 - w2) / (double)scale) : 0;
            v[2 * y] = nd == 4 ? digit::digits4(s) : digit::digits3(s);
            v[2 * y + 1] = nd == 4 ? digit::digits4(e) : digit::digits3(e);
#pragma unroll
            for (int q = 0; q < 4; ++q) sums[q] += (int)(int8_t)(v[2 * y] >> (8 * q));
        }
        d[0][x] = digit::gather_bytes<0>(v[0], v[1], v[2], v[3]);
        d[1][x] = digit::gather_bytes<1>(v[0], v[1], v[2], v[3]);
        d[2][x] = digit::gather_bytes<2>(v[0], v[1], v[2], v[3]);
        d[3][x] = digit::gather_bytes<3>(v[0], v[1], v[2], v[3]);
    }
    uint8_t* dst = img + ((size_t)ch * rows + (size_t)(c / digit::GRAN) * digit::GRAN * nd + c % digit::GRAN) * 16;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < nd) {
            *reinterpret_cast<uint4*>(dst + (size_t)q * digit::GRAN * 16) = make_uint4(d[q][0], d[q][1], d[q][2], d[q][3]);
            atomicAdd(totals + (c / digit::GRAN) * 4 * digit::GRAN + q * digit::GRAN + c % digit::GRAN, 64 * sums[q]);   // in the units of the products
        }
}

// ---- the GEMM ---------------------------------------------------------------------------
// The digit sums over all pairs of the 8 classes of granule g of this warp (shared-space address: [4 digits][32 classes]).
__device__ __forceinline__ void add_totals(uint32_t (&d)[4][8], uint32_t totals, int g) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint4 lo = lds128u(totals + q * 128 + g * 32), hi = lds128u(totals + q * 128 + g * 32 + 16);
        d[q][0] += lo.x; d[q][1] += lo.y; d[q][2] += lo.z; d[q][3] += lo.w;
        d[q][4] += hi.x; d[q][5] += hi.y; d[q][6] += hi.z; d[q][7] += hi.w;
    }
}

// ZO: the activation bits stand for (0,1) instead of (-1,+1).  by_blocks: the logits may leave by tile stores (out_map).
template <bool ZO>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(digit::REG_THREADS, 1)
out_digit_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap out_map, int by_blocks, const uint32_t* __restrict__ Hp, int ldhp,
              const int* __restrict__ flag, const float* __restrict__ scales, const int* __restrict__ totals, const float* __restrict__ bias,
              digit::Work w, float* __restrict__ Z, int ldz, int* __restrict__ done, TcStatus status) {
    extern __shared__ uint8_t smem_raw[];
    // A kernel launched behind this one with programmatic stream serialisation (the log-softmax that
    // follows the frame tiles as they complete) may move onto the SMs once every CTA has got this far.
    pdl_trigger();
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t* staging = smem + digit::RING_BYTES;
    digit::Bars* bars = reinterpret_cast<digit::Bars*>(staging + STAGING + digit::EPI_WARPS * TOTALS);
    volatile int* abort_flag = &bars->wait.abort;
    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const uint32_t ring = smem_u32(smem);
    const uint32_t tmem = digit::set_up(bars, status, warp, w.halved());
    pdl_wait();      // (returns at once in a plain launch) the set-up overlaps the end of the kernel before
                     // this one: 2 us of 35 on 256 frames of the small network
    w.nd = __ldg(flag) ? 4 : 3;

    if (warp >= digit::PROD_WARP0) {
        digit::widen_bits(w, Hp, ldhp, bars, tmem, rank, warp, lane);
    } else if (warp == digit::COPY_WARP) {
        if (lane == 0) digit::copy_digits(w, &map, ring, bars, rank);
    } else if (warp >= digit::EPI_WARPS) {
        if (rank == 0 && warp <= digit::MMA_WARP2) digit::issue(w, ring, bars, tmem, warp - digit::MMA_WARP);
    } else {
        // ---------------- epilogue: thread = one frame (tensor-memory lane); of a tile's classes, or of either part's, warps 0-3 take
        // the first half, warps 4-7 the second
        const int M = w.a_rows, C = w.b_rows;
        const bool halved = w.halved();
        const int grans = w.grans(), per = halved ? (grans + 1) >> 1 : grans;
        const int g0 = halved ? (warp >> 2) * per : 0, g1 = g0 + per < grans ? g0 + per : grans;
        const int ncls = (g1 - g0) * digit::GRAN;               // at most 32
        const int wide = ncls > 16;                             // one frame per store, else two
        const int cl = wide ? lane : lane & 15, fo = wide ? 0 : lane >> 4, fstep = wide ? 1 : 2;
        float* mine = reinterpret_cast<float*>(staging) + warp * 32 * STAGING_PITCH;
        float* row = mine + lane * STAGING_PITCH;
        uint64_t pol;
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
        by_blocks = by_blocks && w.nd == 3;
        const uint32_t block_smem = smem_u32(staging) + warp * BLOCK, consts = smem_u32(staging) + digit::EPI_WARPS * BLOCK + warp * CONSTS;
        const uint32_t tot_smem = smem_u32(staging) + STAGING + warp * TOTALS;
        uint32_t parities = 0u;                                 // to wait for, of the parts
        bool ok = true;
        for (digit::Tiles t(w); ok && t.left > 0; t.next()) {
            for (int part = halved ? 0 : warp >> 2; part < (halved ? digit::PARTS : (warp >> 2) + 1) && !w.beyond(t.b, part); ++part) {
                const int part_gran = (t.b * digit::PARTS + part) * grans, c = (part_gran + g0) * digit::GRAN + cl;
                const bool has = cl < ncls && c < C;
                const float rs = has ? __ldg(scales + c) * (ZO ? 0.5f : 1.0f) : 0.f;
                const float bia = (bias && has) ? __ldg(bias + c) : 0.f;
                if (ZO) {
                    // before the wait for the accumulator, which then is read without waiting for these (8192 x 3400 x 2048 on
                    // (0,1) activations 89 -> 80 us, 3401 classes 124 -> 100; dense digits took 101)
                    const int cls = (part_gran + g0) * digit::GRAN + lane;
                    const int* t0 = totals + (cls / digit::GRAN) * 4 * digit::GRAN + cls % digit::GRAN;
                    int* mine_totals = reinterpret_cast<int*>(staging + STAGING + warp * TOTALS);
                    __syncwarp();
#pragma unroll
                    for (int q = 0; q < 4; ++q) mine_totals[q * 32 + lane] = lane < ncls && cls < C ? __ldg(t0 + q * digit::GRAN) : 0;
                    __syncwarp();
                }
                if (by_blocks) {
                    float* mine_consts = reinterpret_cast<float*>(staging + digit::EPI_WARPS * BLOCK + warp * CONSTS);
                    mine_consts[lane] = rs;
                    mine_consts[32 + lane] = bia;
                    __syncwarp();
                }
                const int f0 = t.a * (2 * digit::ROWS) + rank * digit::ROWS + (warp & 3) * 32;
                ok = warp_wait_relaxed(smem_u32(&bars->acc_full[part]), (parities >> part) & 1u, abort_flag, lane);
                parities ^= 1u << part;
                if (!ok) break;
                tc_fence_after_sync();
                if (by_blocks) {
                    // 32 frames x 32 classes: a tile store, which drops what lies outside
                    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(part * w.n) + (uint32_t)g0 * 24;
                    uint32_t d[4][8];
                    digit::load_granule(taddr, 3, d);
                    if (lane == 0) bulk_wait_read<0>();             // the block before has left shared memory
                    __syncwarp();
#pragma unroll
                    for (int g = 0; g < 4; ++g) {
                        tmem_ld_wait();
                        if (ZO) add_totals(d, tot_smem, g);
                        float z[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) z[i] = fmaf(digit::high_part((int)d[2][i]), 65536.0f, digit::low_part((int)d[0][i], (int)d[1][i]));
                        if (g < 3) digit::load_granule(taddr + (uint32_t)(g + 1) * 24, 3, d);
                        else digit::release_acc(bars, part, lane);
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const uint4 s4 = lds128u(consts + (g * 8 + h * 4) * 4), b4 = lds128u(consts + 128 + (g * 8 + h * 4) * 4);
                            sts128(block_smem + lane * 128 + (((g * 2 + h) ^ (lane & 7)) << 4),
                                   __float_as_uint(fmaf(z[4 * h], __uint_as_float(s4.x), __uint_as_float(b4.x))),
                                   __float_as_uint(fmaf(z[4 * h + 1], __uint_as_float(s4.y), __uint_as_float(b4.y))),
                                   __float_as_uint(fmaf(z[4 * h + 2], __uint_as_float(s4.z), __uint_as_float(b4.z))),
                                   __float_as_uint(fmaf(z[4 * h + 3], __uint_as_float(s4.w), __uint_as_float(b4.w))));
                        }
                    }
                    fence_proxy_async_smem();
                    __syncwarp();
                    const int c0 = (part_gran + g0) * digit::GRAN;
                    if (lane == 0) {
                        if (f0 < M && c0 < C) tma_store_2d_hint(&out_map, c0, f0, block_smem, pol);
                        bulk_commit();
                        if (done) {
                            // this warp's logits of the tile are stored: count it in for the tile's frames (release)
                            bulk_wait<0>();
                            __threadfence();
                            asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(done + t.a) : "memory");
                        }
                    }
                    continue;
                }
                if (f0 < M && g0 < g1) {                            // uniform over the warp
                    const uint32_t width = (uint32_t)(w.nd * digit::GRAN);
                    const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(part * w.n) + (uint32_t)g0 * width;
                    uint32_t d[4][8];
                    digit::load_granule(taddr, w.nd, d);
#pragma unroll 1
                    for (int g = 0; g < g1 - g0; ++g) {
                        tmem_ld_wait();
                        if (ZO) add_totals(d, tot_smem, g);
                        float* dst = row + g * digit::GRAN;
                        if (w.nd == 4) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) dst[i] = digit::join4((int)d[0][i], (int)d[1][i], (int)d[2][i], (int)d[3][i]);
                        } else {
#pragma unroll
                            for (int i = 0; i < 8; ++i)
                                dst[i] = fmaf(digit::high_part((int)d[2][i]), 65536.0f, digit::low_part((int)d[0][i], (int)d[1][i]));
                        }
                        if (g + 1 < g1 - g0) digit::load_granule(taddr + (uint32_t)(g + 1) * width, w.nd, d);
                    }
                }
                digit::release_acc(bars, part, lane);
                if (f0 < M) {
                    // eight rows of the staging block at a time, so that their loads are in flight together
                    __syncwarp();
                    float* dst = Z + (size_t)(f0 + fo) * ldz + c;
                    const size_t step = (size_t)fstep * ldz;
                    const float* src = mine + fo * STAGING_PITCH + cl;
                    const int left = has ? (M - f0 - fo + fstep - 1) / fstep : 0;    // rows of this lane that exist
#pragma unroll 1
                    for (int j = 0; j < 32 / fstep; j += 8) {
                        float v[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) v[i] = fmaf(src[(j + i) * fstep * STAGING_PITCH], rs, bia);
#pragma unroll
                        for (int i = 0; i < 8; ++i, dst += step)
                            if (j + i < left) asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(dst), "f"(v[i]), "l"(pol));
                    }
                }
                __syncwarp();
                if (done) {
                    // this warp's logits of the tile are stored: count it in for the tile's frames (release)
                    __threadfence();
                    __syncwarp();
                    if (lane == 0)
                        asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(done + t.a) : "memory");
                }
            }
        }
    }
    if (by_blocks && warp < digit::EPI_WARPS && lane == 0) bulk_wait<0>();
    digit::tear_down(bars, status, warp, tmem);
}

int out_tile_rows(int M, int C, int H) {
    return digit::tile_rows(M, C, ceil_div(H, digit::GROUP), device_sm_count() / 2);
}

}  // namespace

size_t out_digits_bytes(int C, int H) { return digit_image(C, H).bytes; }

int launch_out_prepare_digits(const float* W, int ldw, int C, int H, void* image, cudaStream_t st) {
    uint8_t* img = static_cast<uint8_t*>(image);
    const DigitImage d = digit_image(C, H);
    int* flag = reinterpret_cast<int*>(img);
    float* tops = reinterpret_cast<float*>(img + d.top);
    int* totals = reinterpret_cast<int*>(img + d.totals);
    if (cudaMemsetAsync(flag, 0, sizeof(int), st) != cudaSuccess) return BNN_ERR_CUDA;
    if (cudaMemsetAsync(totals, 0, (size_t)d.cpad * 4 * sizeof(int), st) != cudaSuccess) return BNN_ERR_CUDA;
    out_range_kernel<<<ceil_div(C, 8), 256, 0, st>>>(W, ldw, C, H, tops, flag);
    const long long items = (long long)d.chunks * d.cpad;
    out_digits_kernel<<<(unsigned)((items + 255) / 256), 256, 0, st>>>(W, ldw, C, H, d.cpad, d.rows, d.chunks, tops, flag,
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
    auto need = [&](int nd) { return ceil_div(C, n / (digit::GRAN * nd) * digit::GRAN) * (n == digit::MAX_N ? 2 : 1) * digit::EPI_WARPS; };    // the epilogue warps of every part
    return FollowArgs{done, need(3), need(4), static_cast<const int*>(image), 2 * digit::ROWS};
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
    CUtensorMap map;
    if (!encode_digit_map(&map, img + d.digits, d.rows, d.chunks, w.n / 2, digit::KB / 16)) return BNN_ERR_CUDA;
    // whole blocks of 32 classes per warp, in rows that a tile store can take
    const int by_blocks = w.n >= digit::MAX_N / 2 && C % 4 == 0 && ldz % 4 == 0 && aligned16(Z);
    CUtensorMap out_map = map;
    if (by_blocks && !encode_int32_map(&out_map, reinterpret_cast<int32_t*>(Z), ldz, M, C)) return BNN_ERR_CUDA;
    const long long tiles = digit::tile_count(M, C, w.n);
    const int pairs = sms / 2;
    const dim3 grid(2 * (int)(tiles < pairs ? tiles : pairs)), block(digit::THREADS);
    const int* flag = reinterpret_cast<const int*>(img);
    const float* scales = reinterpret_cast<const float*>(img + d.scales);
    const int* totals = reinterpret_cast<const int*>(img + d.totals);
    if (!done) {
        const cudaError_t e = launch_pdl(kern, grid, block, SMEM_BYTES, st, map, out_map, by_blocks, Hp, ldhp, flag, scales, totals, bias, w, Z, ldz, done, status);
        return e == cudaSuccess ? launch_status() : BNN_ERR_CUDA;
    }
    // a kernel that follows this one's counters must not start before the kernels that clear them have ended
    kern<<<grid, block, SMEM_BYTES, st>>>(map, out_map, by_blocks, Hp, ldhp, flag, scales, totals, bias, w, Z, ldz, done, status);
    return launch_status();
}

}  // namespace bnn
