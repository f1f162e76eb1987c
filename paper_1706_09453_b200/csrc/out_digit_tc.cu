// Real-valued top layer on +-1 (or 0/1) activations, on the tensor cores with exact integer sums:
//   z[m][c] = sum_h Wout[c][h] * a[m][h] + b[c].
//
// The weights are static, so they are prepared once (bnn_output_prepare_digits): fixed-point numbers of a
// power-of-two scale of each class's own, written as byte digits in the order the tensor core reads shared memory
// (digit_gemm.cuh).  Three digits (about 23 bits relative to the class's largest weight) as long as every class's
// largest weight is at most 16 times its mean magnitude -- then even if all H roundings, each at most 1.01 * 2^-23 of
// the largest weight, add up, a logit is within 2^-19 of sum |w| -- and four digits (31 bits) for the whole
// matrix otherwise.  The choice is made on the device and read from the image by the GEMM.
//
// The GEMM runs on CTA pairs, frames on the M side (tensor-memory lane = frame), class digits on the N side: a tile
// is 256 frames x 64 (or 32) classes.  The epilogue transposes through shared memory so that a store covers
// 32 consecutive classes of a frame.
//
// Bound by the tensor pipe (three passes over the weights at the byte rate).  Measured on B200 against the kernel it
// replaced (two fp16 terms, fp32 sums, one CTA per tile of 128 classes x 512 frames), 3400 classes x 2048 units:
// 8192 frames 133 -> 108 us (1.06 PFLOP/s of algorithmic work; the bare MMAs take 84), 731 frames 54 -> 20 us, 20
// frames 42 -> 10 us; 65536 frames x 4000 x 3072 1.81 -> 1.36 ms.  Largest error of a logit (|z| up to 5) 1.9e-5 -> 1.1e-6.
#include "bnn_common.cuh"
#include "digit_gemm.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

using namespace tc;

// The image: [flag, 256 bytes][largest magnitude per class][2^-e per class][digits].
struct DigitImage {
    size_t mx, scales, digits, bytes;   // offsets; total size
    int cpad;
    int rows;                         // digit rows per chunk of 16 positions: room for four digits
    int chunks;
};
DigitImage digit_image(int C, int H) {
    DigitImage d;
    d.cpad = ceil_div(C, digit::GRAN) * digit::GRAN;
    d.mx = 256;
    d.scales = d.mx + (size_t)d.cpad * sizeof(float);
    d.digits = (d.scales + (size_t)d.cpad * sizeof(float) + 255) & ~size_t(255);
    d.rows = 4 * d.cpad;
    d.chunks = 2 * ceil_div(H, 32);
    d.bytes = d.digits + (size_t)d.chunks * d.rows * 16;
    return d;
}

constexpr int STAGING_PITCH = 33;
constexpr int SMEM_BYTES = digit::RING_BYTES + digit::EPI_WARPS * 32 * STAGING_PITCH * 4 + (int)sizeof(digit::Bars) + 1024;
constexpr int kFollowGroupMin = 2 * digit::ROWS;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

// ---- one-time preparation of the weights -------------------------------------------------
// One warp per class: mx[c] = max_h |W[c][h]|; *flag is set when some class needs four digits.
__global__ void out_range_kernel(const float* __restrict__ W, int ldw, int C, int H, float* __restrict__ mxs, int* __restrict__ flag) {
    const int c = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (c >= C) return;
    float sum = 0.f;
    uint32_t top = 0u;   // largest magnitude as bits: orders NaN above infinity above every number
    for (int h = lane; h < H; h += 32) {
        const float a = fabsf(W[(size_t)c * ldw + h]);
        sum += a;
        top = max(top, __float_as_uint(a));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
        top = max(top, __shfl_xor_sync(0xFFFFFFFFu, top, o));
    }
    if (lane == 0) {
        mxs[c] = __uint_as_float(top);
        if ((float)H * __uint_as_float(top) > 16.0f * sum) atomicOr(flag, 1);
    }
}

// One thread writes the digits of 16 positions of a class (one chunk of each digit row).
__global__ void out_digits_kernel(const float* __restrict__ W, int ldw, int C, int H, int Cpad8, int rows, int chunks,
                                  const float* __restrict__ mxs, const int* __restrict__ flag, float* __restrict__ scales,
                                  uint8_t* __restrict__ img) {
    const int nd = *flag ? 4 : 3;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (long long)chunks * Cpad8) return;
    const int c = (int)(i % Cpad8), ch = (int)(i / Cpad8);
    const digit::Scale scale(c < C ? digit::scale_exponent(mxs[c], nd) : 0);
    if (ch == 0) scales[c] = c < C ? digit::inverse_scale(mxs[c], nd) : 0.f;
    uint32_t d[4][4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        uint32_t v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {          // byte 4 t + j of the chunk
            const int k = (ch >> 1) * 32 + (ch & 1) * 4 + t + 8 * j;
            const int n = (c < C && k < H) ? scale.fixed_point(W[(size_t)c * ldw + k]) : 0;
            v[j] = nd == 4 ? digit::digits4(n) : digit::digits3(n);
        }
        d[0][t] = digit::gather_bytes<0>(v[0], v[1], v[2], v[3]);
        d[1][t] = digit::gather_bytes<1>(v[0], v[1], v[2], v[3]);
        d[2][t] = digit::gather_bytes<2>(v[0], v[1], v[2], v[3]);
        d[3][t] = digit::gather_bytes<3>(v[0], v[1], v[2], v[3]);
    }
    uint8_t* dst = img + ((size_t)ch * rows + (size_t)(c / digit::GRAN) * digit::GRAN * nd + c % digit::GRAN) * 16;
#pragma unroll
    for (int q = 0; q < 4; ++q)
        if (q < nd) *reinterpret_cast<uint4*>(dst + (size_t)q * digit::GRAN * 16) = make_uint4(d[q][0], d[q][1], d[q][2], d[q][3]);
}

// ---- the GEMM ---------------------------------------------------------------------------
// ZO: the activation bits stand for (0,1) instead of (-1,+1).
template <bool ZO>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(digit::REG_THREADS, 1)
out_digit_kernel(const __grid_constant__ CUtensorMap map, const uint32_t* __restrict__ Hp, int ldhp,
              const int* __restrict__ flag, const float* __restrict__ scales, const float* __restrict__ bias,
              digit::Work w, float* __restrict__ Z, int ldz, int* __restrict__ done, TcStatus status) {
    extern __shared__ uint8_t smem_raw[];
    // A kernel launched behind this one with programmatic stream serialisation (the log-softmax that
    // follows the frame tiles as they complete) may move onto the SMs once every CTA has got this far.
    pdl_trigger();
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    float* staging = reinterpret_cast<float*>(smem + digit::RING_BYTES);
    digit::Bars* bars = reinterpret_cast<digit::Bars*>(staging + digit::EPI_WARPS * 32 * STAGING_PITCH);
    volatile int* abort_flag = &bars->wait.abort;
    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const uint32_t ring = smem_u32(smem);
    const uint32_t tmem = digit::set_up(bars, status, warp);
    pdl_wait();      // (returns at once in a plain launch) the set-up overlaps the end of the kernel before
                     // this one: 2 us of 35 on 256 frames of the small network
    w.nd = __ldg(flag) ? 4 : 3;

    if (warp >= digit::PROD_WARP0) {
        digit::widen_bits<ZO>(w, Hp, ldhp, bars, tmem, rank, warp, lane);
    } else if (warp == digit::COPY_WARP) {
        if (lane == 0) digit::copy_digits(w, &map, ring, bars, rank);
    } else if (warp >= digit::EPI_WARPS) {
        if (rank == 0 && warp <= digit::MMA_WARP2) digit::issue(w, ring, bars, tmem, warp - digit::MMA_WARP);
    } else {
        // ---------------- epilogue: thread = one frame (tensor-memory lane); of a tile's classes warps 0-3 take the
        // first half, warps 4-7 the second
        const int M = w.a_rows, C = w.b_rows;
        const int grans = w.n / (digit::GRAN * w.nd), per = (grans + 1) >> 1;
        const int g0 = (warp >> 2) * per, g1 = g0 + per < grans ? g0 + per : grans;
        const int ncls = (g1 - g0) * digit::GRAN;               // at most 32
        const int wide = ncls > 16;                             // one frame per store, else two
        const int cl = wide ? lane : lane & 15, fo = wide ? 0 : lane >> 4, fstep = wide ? 1 : 2;
        float* mine = staging + warp * 32 * STAGING_PITCH;
        uint64_t pol;
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
        int tl = 0;
        const int nb = w.nb();
        for (digit::Tiles t(w); t.left > 0; t.next(), ++tl) {
            const int c = t.b * nb + g0 * digit::GRAN + cl;
            const int f0 = t.a * (2 * digit::ROWS) + rank * digit::ROWS + (warp & 3) * 32;
            const bool has = cl < ncls && c < C;
            const float rs = has ? __ldg(scales + c) : 0.f;
            const float bia = (bias && has) ? __ldg(bias + c) : 0.f;
            const int b = tl & 1;
            if (!warp_wait_relaxed(smem_u32(&bars->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane)) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * w.n);
            if (f0 < M) {                                       // uniform over the warp
                float* row = mine + lane * STAGING_PITCH;
                digit::granules(taddr + (uint32_t)(g0 * digit::GRAN * w.nd), g1 - g0, w.nd, [&](int g, const float (&S)[8]) {
#pragma unroll
                    for (int i = 0; i < 8; ++i) row[g * digit::GRAN + i] = S[i];
                });
            }
            digit::release_acc(bars, b, lane);
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
    digit::tear_down(bars, status, warp, tmem);
}

int out_tile_rows(int M, int C, int H) {
    return digit::tile_rows(M, C, ceil_div(H, 32), device_sm_count() / 2);
}

}  // namespace

size_t out_digits_bytes(int C, int H) { return digit_image(C, H).bytes; }

int launch_out_prepare_digits(const float* W, int ldw, int C, int H, void* image, cudaStream_t st) {
    uint8_t* img = static_cast<uint8_t*>(image);
    const DigitImage d = digit_image(C, H);
    int* flag = reinterpret_cast<int*>(img);
    float* mxs = reinterpret_cast<float*>(img + d.mx);
    if (cudaMemsetAsync(flag, 0, sizeof(int), st) != cudaSuccess) return BNN_ERR_CUDA;
    out_range_kernel<<<ceil_div(C, 8), 256, 0, st>>>(W, ldw, C, H, mxs, flag);
    const long long items = (long long)d.chunks * d.cpad;
    out_digits_kernel<<<(unsigned)((items + 255) / 256), 256, 0, st>>>(W, ldw, C, H, d.cpad, d.rows, d.chunks, mxs, flag,
                                                                         reinterpret_cast<float*>(img + d.scales), img + d.digits);
    return launch_status();
}

// With no more tiles than CTA pairs every tile ends at about the same time: nothing for a following kernel to
// overlap with (measured: 1-2 % slower than two launches in a row on 256 frames).
bool out_digit_can_be_followed(int M, int C, int H) {
    return M > kFollowGroupMin &&
           ceil_div(M, 2 * digit::ROWS) * ceil_div(C, out_tile_rows(M, C, H) / 3) > device_sm_count() / 2;
}
FollowArgs out_digit_follow(const void* image, int M, int C, int H, int* done) {
    const int n = out_tile_rows(M, C, H);
    auto need = [&](int nd) { return ceil_div(C, n / nd) * 2 * digit::EPI_WARPS; };
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
    const digit::Work w{M, C, out_tile_rows(M, C, H), 3, ceil_div(H, 32), 1};
    CUtensorMap map;
    if (!encode_digit_map(&map, img + d.digits, d.rows, d.chunks, w.n / 2, digit::KB / 16)) return BNN_ERR_CUDA;
    const long long tiles = (long long)ceil_div(M, 2 * digit::ROWS) * ceil_div(C, w.n / 3);
    const int pairs = sms / 2;
    const dim3 grid(2 * (int)(tiles < pairs ? tiles : pairs)), block(digit::THREADS);
    const int* flag = reinterpret_cast<const int*>(img);
    const float* scales = reinterpret_cast<const float*>(img + d.scales);
    if (!done) {
        const cudaError_t e = launch_pdl(kern, grid, block, SMEM_BYTES, st, map, Hp, ldhp, flag, scales, bias, w, Z, ldz, done, status);
        return e == cudaSuccess ? launch_status() : BNN_ERR_CUDA;
    }
    // a kernel that follows this one's counters must not start before the kernels that clear them have ended
    kern<<<grid, block, SMEM_BYTES, st>>>(map, Hp, ldhp, flag, scales, bias, w, Z, ldz, done, status);
    return launch_status();
}

}  // namespace bnn
