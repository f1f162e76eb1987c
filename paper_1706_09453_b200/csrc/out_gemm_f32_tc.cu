// Real-valued layer on real-valued activations, on the tensor cores: the top layer of the
// binary-weights-only networks of Algorithm 1 (whose last hidden layer hands on fp32 values) and
// the real-valued hidden layers of the paper's mixed networks (Table 2), with an optional
// activation f (Sigmoid, clamp):
//   z[m][c] = f( sum_h Wout[c][h] * a[m][h] + b[c] ).
//
// Both operands are split into two fp16 terms.  The weights use the image bnn_output_prepare
// builds (per-row power-of-two scaling, w * 2^e = w1 + w2, about 22 significant bits).  The
// activations are split once per call into a scratch image, a = a1 + a2 with
// |a - a1 - a2| <= max(2^-22 |a|, 2^-25), in the order the MMA reads shared memory
// (h_split_kernel, a memory-bound pass).  Three MMAs per K step, a1 w1 + a1 w2 + a2 w1,
// accumulate in fp32 in tensor memory; the term a2 w2 (<= 2^-22 |a w|) is dropped, so
//   |z - exact| <= ~3 * 2^-22 * sum_h |a[m][h]| |Wout[c][h]|  + fp32 accumulation rounding.
// Activations must be finite fp16-range numbers (|a| < 65504; the outputs of hardtanh are
// within [-1, 1]).
//
// Orientation as in out_gemm_tc.cu: classes on the M side (TMEM lanes), frames on the N side;
// a CTA tile is 128 classes x 256, 128 or 64 frames with two accumulators, so the epilogue of one tile
// overlaps the MMAs of the next.  A pipeline stage (32 positions of K) is bulk copies of 16 KB of the weight
// image and 128 bytes per frame of the activation image; nothing is widened on chip.  Where the tiles of a few frames
// would leave SMs idle, a cluster of 2 or 4 CTAs shares a tile (SPLIT): each takes a part of K, leaves its sums in its
// shared memory, and adds up and finishes its part of the frames from all of them.
//   warp 17      issues the bulk copies
//   warp 16      issues the MMAs (6 per stage, from one elected lane) and the commits
//   warps 0-15   epilogue: f(acc * 2^-e + b), 32 consecutive classes of a frame per warp store; warp w takes the
//                lanes of quarter w % 4 and every fourth group of 32 frames.  (A Sigmoid is about 40 instructions, so a layer
//                of short rows is bound by the epilogue: 8192 x 440 -> 2048 with Sigmoid 114 us with four warps, 44 us with
//                sixteen; 8192 x 2048 -> 3400 without, 198 us, is bound by the MMAs: three passes at half-precision rate.)
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles fall
// through to the common teardown and the device status word is set.
#include <cuda_fp16.h>

#include "bnn_common.cuh"
#include "tcgen05.cuh"

namespace bnn {

namespace {

using namespace tc;

constexpr int BC = 128;           // classes per tile (as the prepared weight image)
constexpr int IMG = 256;          // frames per block of the activation image
constexpr int BK = 32;            // k per stage
constexpr int A_PLANE = BC * BK * 2;        // 8 KB per weight term
constexpr int A_BYTES = 2 * A_PLANE;
constexpr int IMG_PLANE = IMG * BK * 2;     // 16 KB per activation term and block
constexpr int IMG_BYTES = 2 * IMG_PLANE;
// FN: frames per tile
template <int FN> struct Cfg {
    static constexpr int B_PLANE = FN * BK * 2, B_BYTES = 2 * B_PLANE;
    static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int STAGES = FN == 256 ? 4 : FN == 128 ? 6 : 8;
};
constexpr int MAX_STAGES = 8;
constexpr int EPI_WARPS = 16, MMA_WARP = EPI_WARPS, TMA_WARP = MMA_WARP + 1;
constexpr int THREADS = (TMA_WARP + 1) * 32;
constexpr uint32_t TMEM_COLS = 512;

struct Control {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES], acc_full[2], acc_empty[2];
    uint32_t tmem_base;
    WaitState wait;
};
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// ---- split: thread = one 16-byte chunk of a frame row ---------------------------------------
// Block (ft, ks) of the image: [term 0..1][chunk c = 2 j + cc][row 0..255][16 bytes], where
// chunk (j, cc) holds, in element e, position k = 32 ks + 8 j + (pos >> 1) + 16 (pos & 1),
// pos = 8 cc + e: the order of the prepared weight image, so both operands agree on k.  In other words element
// e of chunk c is position 4 c + (e >> 1) + 16 (e & 1): a chunk is two groups of four consecutive positions.
// Four lanes cover the 128 bytes of a row, a warp eight rows.  (Measured on B200, a thread with the 32 positions of a
// row before: 8192 x 2048 of int32 with Sigmoid 48 -> 37 us,
// of which the Sigmoids are most.)
// FROM_I32: the activations are Sigmoid(fma(scale[h], d, shift[h])) of integer dot products d (a binary
// layer with Sigmoid units, Section 3.2 / Table 2), evaluated here instead of in a pass of their own.
// p[k0 .. k0 + 3] and p[k0 + 16 .. k0 + 19]; `other` beyond H or without p.
__device__ __forceinline__ void load8(const float* __restrict__ p, int k0, int H, float other, float (&o)[8]) {
    if (p && (reinterpret_cast<uintptr_t>(p) & 15) == 0 && k0 + 20 <= H) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(p + k0)), b = __ldg(reinterpret_cast<const float4*>(p + k0 + 16));
        o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w; o[4] = b.x; o[5] = b.y; o[6] = b.z; o[7] = b.w;
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = k0 + (i & 3) + (i >> 2) * 16;
            o[i] = p && k < H ? __ldg(p + k) : other;
        }
    }
}
constexpr int SPLIT_THREADS = 256, SPLIT_ROWS = SPLIT_THREADS / 4;
template <bool FROM_I32>
__global__ void __launch_bounds__(SPLIT_THREADS)
h_split_kernel(const void* __restrict__ src, int ldh, int M, int H, int nks, uint8_t* __restrict__ img,
               const float* __restrict__ scale, const float* __restrict__ shift) {
    pdl_trigger();
    pdl_wait();
    const int ks = (int)blockIdx.x % nks, rb = (int)blockIdx.x / nks;      // rb: block of SPLIT_ROWS rows
    const int c = threadIdx.x & 3, m = rb * SPLIT_ROWS + ((int)threadIdx.x >> 2);
    const int ft = m / IMG, row = m % IMG, k0 = ks * BK + 4 * c;
    float v[8];              // positions k0 .. k0 + 3, k0 + 16 .. k0 + 19
    const uint32_t* p = static_cast<const uint32_t*>(src) + (size_t)m * ldh + k0;
    const bool vec = (ldh % 4 == 0) && ((reinterpret_cast<uintptr_t>(src) & 15) == 0) && k0 + 20 <= H;
    if (m < M && vec) {
        const uint4 a = __ldg(reinterpret_cast<const uint4*>(p)), b = __ldg(reinterpret_cast<const uint4*>(p + 16));
        v[0] = __uint_as_float(a.x); v[1] = __uint_as_float(a.y); v[2] = __uint_as_float(a.z); v[3] = __uint_as_float(a.w);
        v[4] = __uint_as_float(b.x); v[5] = __uint_as_float(b.y); v[6] = __uint_as_float(b.z); v[7] = __uint_as_float(b.w);
    } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const int k = (i & 3) + (i >> 2) * 16;
            v[i] = (m < M && k0 + k < H) ? __uint_as_float(__ldg(p + k)) : 0.f;
        }
    }
    if (FROM_I32) {
        float sc[8], sh[8];
        load8(scale, k0, H, 1.0f, sc);
        load8(shift, k0, H, 0.0f, sh);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const float d = (float)__float_as_int(v[i]);
            const float y = fmaf(sc[i], d, sh[i]);
            v[i] = (m < M && k0 + (i & 3) + (i >> 2) * 16 < H) ? 1.0f / (1.0f + expf(-y)) : 0.f;
        }
    }
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {      // elements 2 i and 2 i + 1
        const __half2 h1 = __floats2half2_rn(v[i], v[i + 4]);
        const float2 f1 = __half22float2(h1);
        const __half2 h2 = __floats2half2_rn(v[i] - f1.x, v[i + 4] - f1.y);
        hi[i] = *reinterpret_cast<const uint32_t*>(&h1);
        lo[i] = *reinterpret_cast<const uint32_t*>(&h2);
    }
    uint8_t* dst = img + ((size_t)ft * nks + ks) * IMG_BYTES + (size_t)(c * IMG + row) * 16;
    *reinterpret_cast<uint4*>(dst) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dst + IMG_PLANE) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

// ---- the GEMM ---------------------------------------------------------------------------
__device__ __forceinline__ float lds_cluster(uint32_t cluster_addr) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_addr) : "memory");
    return v;
}
__device__ __forceinline__ float finish(float acc, float scl, float bia, int act) {
    float v = fmaf(acc, scl, bia);
    if (act == BNN_ACT_SIGMOID) v = 1.0f / (1.0f + expf(-v));
    else if (act == BNN_ACT_HARDTANH) v = fminf(fmaxf(v, -1.0f), 1.0f);
    return v;
}

// SPLIT > 1: clusters of SPLIT CTAs, one tile per cluster.
template <int FN, int SPLIT>
__global__ void __launch_bounds__(THREADS, 1)
outf_tc_kernel(const uint8_t* __restrict__ himg, const uint8_t* __restrict__ wimg,
               const float* __restrict__ rs, const float* __restrict__ bias,
               int M, int C, int H, float* __restrict__ Z, int ldz, int act, TcStatus status) {
    constexpr int B_PLANE = Cfg<FN>::B_PLANE, STAGE_BYTES = Cfg<FN>::STAGE_BYTES, STAGES = Cfg<FN>::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
    Control* ctl = reinterpret_cast<Control*>(smem + STAGES * STAGE_BYTES);
    volatile int* abort_flag = &ctl->wait.abort;

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int nks = ceil_div(H, BK);
    const int rank = SPLIT > 1 ? (int)cluster_rank() : 0, group = (int)blockIdx.x / SPLIT, groups = (int)gridDim.x / SPLIT;
    const int k0 = rank * nks / SPLIT, k1 = (rank + 1) * nks / SPLIT;      // this CTA's stages
    const int c_tiles = ceil_div(C, BC), f_tiles = ceil_div(M, FN);
    const int tiles = c_tiles * f_tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 1);    // the copying warp (+ bytes)
            mbar_init(smem_u32(&ctl->empty[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), EPI_WARPS);
        }
        wait_state_init(&ctl->wait, status);
        mbar_init_fence();
    }
    if (warp == MMA_WARP) {
        tmem_alloc(smem_u32(&ctl->tmem_base), TMEM_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = ctl->tmem_base;
    pdl_trigger();
    pdl_wait();      // the set-up above overlaps the end of the kernel before this one

    if (warp == TMA_WARP) {
        // ---------------- a warp streams both images, a lane per copy (one thread takes about 100 clocks for each); class
        // tiles vary fastest so that consecutive CTAs share a tile of frames in L2
        int s = 0;
        uint32_t ph = 1;     // parity to wait for on `empty`: a fresh barrier passes parity 1
        bool ok = true;
        for (int tile = group; tile < tiles && ok; tile += groups) {
            const uint8_t* wsrc = wimg + (size_t)(tile % c_tiles) * nks * A_BYTES;
            const int f0 = (tile / c_tiles) * FN;
            const uint8_t* hsrc = himg + (size_t)(f0 / IMG) * nks * IMG_BYTES + (f0 % IMG) * 16;
            // this lane's copy of every stage: its term and chunk, the whole block where the tile is one, or the weights
            const uint8_t* src = nullptr;
            uint32_t to = 0, bytes = 0, step = IMG_BYTES;
            if (lane == 8) { src = wsrc; bytes = A_BYTES; step = A_BYTES; }
            else if (FN == IMG) { if (lane == 0) { src = hsrc; to = A_BYTES; bytes = IMG_BYTES; } }
            else if (lane < 8) { src = hsrc + lane * (IMG * 16); to = A_BYTES + lane * (FN * 16); bytes = FN * 16; }
            src += (size_t)k0 * step;
            for (int ks = k0; ks < k1; ++ks) {
                ok = warp_wait(smem_u32(&ctl->empty[s]), ph, abort_flag, lane);
                if (!ok) break;
                const uint32_t bar = smem_u32(&ctl->full[s]);
                if (lane == 0) mbar_arrive_expect_tx(bar, STAGE_BYTES);
                __syncwarp();
                if (bytes) bulk_g2s(smem_u32(smem) + s * STAGE_BYTES + to, src, bytes, bar);
                src += step;
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
        }
        __syncwarp();
    } else if (warp == MMA_WARP) {
        constexpr uint32_t idesc = instr_desc(kAccF32, kFmtF16, kFmtF16, BC, FN);
        const uint64_t w0 = smem_desc_kmajor(smem_u32(smem), BC * 16, 128), h0 = smem_desc_kmajor(smem_u32(smem) + A_BYTES, FN * 16, 128);
        int s = 0, tl = 0;
        uint32_t ph = 0;
        bool ok = true;
        for (int tile = group; tile < tiles && ok; tile += groups, ++tl) {
            const int b = tl & 1;
            ok = warp_wait(smem_u32(&ctl->acc_empty[b]), (uint32_t)(((tl >> 1) & 1) ^ 1), abort_flag, lane);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t d = tmem + (uint32_t)(b * IMG);
            for (int ks = k0; ks < k1; ++ks) {
                ok = warp_wait(smem_u32(&ctl->full[s]), ph, abort_flag, lane);
                if (!ok) break;
                tc_fence_after_sync();
                // the address field (16-byte units) is advanced by plain additions: the ring lies below 2^14 * 16 bytes
                const uint64_t at = (uint64_t)(s * (STAGE_BYTES >> 4));
                if (elect_one()) {
#pragma unroll
                    for (int j = 0; j < 2; ++j) {   // K step of 16 = two 16-byte chunks
                        const uint64_t w1 = w0 + at + (uint64_t)((2 * j * (BC * 16)) >> 4), w2 = w1 + (uint64_t)(A_PLANE >> 4);
                        const uint64_t h1 = h0 + at + (uint64_t)((2 * j * (FN * 16)) >> 4), h2 = h1 + (uint64_t)(B_PLANE >> 4);
                        mma_f16(d, w1, h1, idesc, ks != k0 || j != 0);
                        mma_f16(d, w2, h1, idesc, 1u);
                        mma_f16(d, w1, h2, idesc, 1u);
                    }
                    mma_commit(smem_u32(&ctl->empty[s]));
                }
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            if (ok && elect_one()) mma_commit(smem_u32(&ctl->acc_full[b]));
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: thread = one class (TMEM lane), columns = frames
        const int row_in_tile = (warp & 3) * 32 + lane;
        int tl = 0;
        bool ok = true;
        for (int tile = group; tile < tiles && ok; tile += groups, ++tl) {
            const int c = (tile % c_tiles) * BC + row_in_tile;
            const int f0 = (tile / c_tiles) * FN;
            const float scl = rs[c];                       // rs is padded to whole tiles
            const float bia = (bias && c < C) ? bias[c] : 0.f;
            const int b = tl & 1;
            ok = warp_wait_relaxed(smem_u32(&ctl->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * IMG);
#pragma unroll 1
            for (int gi = warp >> 2; gi < FN / 32; gi += EPI_WARPS / 4) {
                if (f0 + gi * 32 >= M) break;              // uniform over the warp
                uint32_t acc[32];
                tmem_ld32(taddr + gi * 32, acc);
                tmem_ld_wait();
                if (SPLIT > 1) {                           // the ring is free: every stage has been multiplied
                    float* sums = reinterpret_cast<float*>(smem) + gi * 32 * BC + row_in_tile;      // [frame][class]
#pragma unroll
                    for (int j = 0; j < 32; ++j) sums[j * BC] = __uint_as_float(acc[j]);
                } else if (c < C) {
                    float* dst = Z + (size_t)(f0 + gi * 32) * ldz + c;
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (f0 + gi * 32 + j < M) dst[(size_t)j * ldz] = finish(__uint_as_float(acc[j]), scl, bia, act);
                }
            }
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
        }
    }

    if (SPLIT > 1) {
        __syncwarp();
        cluster_sync();                                    // the sums of all CTAs are in place
        if (warp < EPI_WARPS) {
            const int row_in_tile = (warp & 3) * 32 + lane, c = (group % c_tiles) * BC + row_in_tile, f0 = (group / c_tiles) * FN;
            const float scl = rs[c], bia = (bias && c < C) ? bias[c] : 0.f;
            uint32_t from[SPLIT];
#pragma unroll
            for (int r = 0; r < SPLIT; ++r) from[r] = peer_addr(smem_u32(smem) + row_in_tile * 4, r);
#pragma unroll 4
            for (int f = rank * (FN / SPLIT) + (warp >> 2); f < (rank + 1) * (FN / SPLIT) && f0 + f < M; f += EPI_WARPS / 4) {
                float v = lds_cluster(from[0] + f * (BC * 4));
#pragma unroll
                for (int r = 1; r < SPLIT; ++r) v += lds_cluster(from[r] + f * (BC * 4));
                if (c < C) Z[(size_t)(f0 + f) * ldz + c] = finish(v, scl, bia, act);
            }
        }
        __syncwarp();
        cluster_sync();                                    // nobody reads this CTA's shared memory any more
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && ctl->wait.abort) atomicExch(status.word, 1);
}

}  // namespace

size_t outf_image_bytes(int M, int H) {
    return (size_t)ceil_div(M, IMG) * ceil_div(H, BK) * IMG_BYTES;
}

// Frames per tile and CTAs per tile: the least clocks of the busiest CTA.  What a stage takes is as measured; it is bound by
// the copies (an SM receives 30 to 50 bytes per clock from L2), so that 64 frames take little less than 128.  Measured on
// B200, 2048 -> 3307, us, one CTA to a tile of 256 frames before: 3 frames 31 -> 11, 200 33 -> 17, 400 35 -> 28; from 731
// frames on as before (36; tiles of 128 would take 52).  Sums
// of a layer with an activation are not split: a Sign layer may come behind, whose decisions follow their rounding.
struct Tiling { int frames, split; };
static Tiling tiling(int M, int C, int nks, int act, int sms) {
    struct Candidate { int frames, stage; };
    const Candidate all[] = {{256, 950}, {128, 740}, {64, 670}};
    Tiling best{256, 1};
    long long best_cost = 0;
    for (const Candidate& c : all)
        for (const int split : {1, 2, 4}) {
            const int tiles = ceil_div(C, BC) * ceil_div(M, c.frames);
            if (split > 1 && (tiles * split > sms || nks < 4 * split || act != BNN_ACT_NONE)) continue;
            const long long cost = (long long)ceil_div(tiles * split, sms) * ceil_div(nks, split) * c.stage + (split > 1 ? 3000 : 0);
            if (best_cost == 0 || cost < best_cost) { best = Tiling{c.frames, split}; best_cost = cost; }
        }
    return best;
}

template <int FN, int SPLIT>
static int launch_gemm(const uint8_t* himg, const uint8_t* wimg, const float* rs, const float* bias, int M, int C, int H,
                       float* Z, int ldz, int act, int sms, cudaStream_t st) {
    constexpr int SMEM = Cfg<FN>::STAGES * Cfg<FN>::STAGE_BYTES + (int)sizeof(Control) + 128;
    static_assert(SMEM <= 232448, "shared memory of one CTA");
    static_assert(SPLIT == 1 || FN * BC * 4 <= Cfg<FN>::STAGES * Cfg<FN>::STAGE_BYTES, "the sums of a tile fit the ring");
    auto kern = outf_tc_kernel<FN, SPLIT>;
    if (!ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM)) return BNN_ERR_CUDA;
    const TcStatus status = tc_status();
    if (!status.word) return BNN_ERR_CUDA;
    const int tiles = ceil_div(C, BC) * ceil_div(M, FN);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SPLIT > 1 ? tiles * SPLIT : (tiles < sms ? tiles : sms));
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = SPLIT;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = SPLIT > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, kern, himg, wimg, rs, bias, M, C, H, Z, ldz, act, status) != cudaSuccess) return BNN_ERR_CUDA;
    return launch_status();
}
template <int FN>
static int launch_split(int split, const uint8_t* himg, const uint8_t* wimg, const float* rs, const float* bias, int M, int C, int H,
                        float* Z, int ldz, int act, int sms, cudaStream_t st) {
    if (split == 4) return launch_gemm<FN, 4>(himg, wimg, rs, bias, M, C, H, Z, ldz, act, sms, st);
    if (split == 2) return launch_gemm<FN, 2>(himg, wimg, rs, bias, M, C, H, Z, ldz, act, sms, st);
    return launch_gemm<FN, 1>(himg, wimg, rs, bias, M, C, H, Z, ldz, act, sms, st);
}

int launch_outf_tc(const float* Hf, int ldhf, const void* prepared, const float* bias,
                   int M, int C, int H, float* Z, int ldz, int act, void* workspace, bool image_ready, cudaStream_t st) {
    const int sms = device_sm_count();
    if (sms <= 0) return BNN_ERR_CUDA;
    const int ct = ceil_div(C, BC), hs = ceil_div(H, BK);
    // the prepared weight image: ct * hs blocks of both terms, then the per-class factors 2^-e
    const uint8_t* wimg = static_cast<const uint8_t*>(prepared);
    const float* rs = reinterpret_cast<const float*>(wimg + (size_t)ct * hs * A_BYTES);
    uint8_t* himg = static_cast<uint8_t*>(workspace);
    if (!image_ready)   // (else the layer that produced the activations wrote the image itself)
        if (launch_pdl(h_split_kernel<false>, dim3(ceil_div(M, IMG) * hs * (IMG / SPLIT_ROWS)), dim3(SPLIT_THREADS), 0, st, Hf, ldhf, M, H, hs, himg,
                       nullptr, nullptr) != cudaSuccess)
            return BNN_ERR_CUDA;
    const Tiling t = tiling(M, C, hs, act, sms);
    if (t.frames == 64) return launch_split<64>(t.split, himg, wimg, rs, bias, M, C, H, Z, ldz, act, sms, st);
    if (t.frames == 128) return launch_split<128>(t.split, himg, wimg, rs, bias, M, C, H, Z, ldz, act, sms, st);
    return launch_split<256>(t.split, himg, wimg, rs, bias, M, C, H, Z, ldz, act, sms, st);
}


int launch_outf_image_from_i32(const int32_t* D, int ldd, const float* scale, const float* shift, int M, int H,
                               void* image, cudaStream_t st) {
    const int hs = ceil_div(H, BK), ft = ceil_div(M, IMG);
    const dim3 grid(ft * hs * (IMG / SPLIT_ROWS)), block(SPLIT_THREADS);
    uint8_t* img = static_cast<uint8_t*>(image);
    // On a large batch the CTAs of this pass would wait beside the binary product's for most of its time (mixed network, 8192
    // frames: 513 us against 504); on a small one the early start is worth 1 to 2 us.
    if (M > 2048) h_split_kernel<true><<<grid, block, 0, st>>>(D, ldd, M, H, hs, img, scale, shift);
    else if (launch_pdl(h_split_kernel<true>, grid, block, 0, st, D, ldd, M, H, hs, img, scale, shift) != cudaSuccess) return BNN_ERR_CUDA;
    return launch_status();
}

}  // namespace bnn
