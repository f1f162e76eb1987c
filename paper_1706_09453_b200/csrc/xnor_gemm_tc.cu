// XNOR GEMM on the 5th-generation tensor cores as a 4-bit floating-point contraction.
//
//   dot[m][n] = sum_k a[m][k] * w[n][k],  a, w in {-1, +1}  ( = K - 2 popc(a xor w) )
//
// The tensor cores have no 1-bit mode, so every bit is widened on the fly, in the SM, to the
// narrowest type they multiply: the 4-bit float e2m1, in which +1 is the nibble 0x2 and -1 the
// nibble 0xA (kind::mxf4; its per-32-element block scales are all set to 2^0).  The products are
// +-1 and the fp32 accumulator holds their integer sums exactly for K <= 2^22, so the result is
// the signed dot product itself: no popcount correction terms, no bias.  Padding (K rounded up
// to the stage size) is the nibble 0, i.e. +0.
//
// Widening costs 4 bits of shared memory per bit of input, half of what an 8-bit integer
// contraction needs, and the 4-bit MMA has twice its rate; both matter because this kernel
// is bound by the shared-memory pipe (stores of the widened operands + the tensor core's
// reads of them), not by HBM: the packed operands are tiny.
//
// K may be visited in any order as long as both operands use the same one.  The order here
// makes widening two instructions per 32-bit output word: output word t (0..3) of input word
// w holds, in nibble i, bit 4i + t of w:   ((w << (3 - t)) & 0x88888888) ^ 0xAAAAAAAA
// (sign bit = NOT the input bit, exponent field = 01).
//
// A pair of CTAs (cluster of two, one per SM of a TPC) works on a tile of 256 frames x two parts of 128 units (64 where that fills more SMs, launch_xnor_tc): each CTA widens
// its own 128 frames and half of the units, where a CTA by itself (xnor_gemm_cta.cu) widens all of them.  Roles in a CTA of 27 warps, with parts of 64 units 23
// (persistent, one CTA per SM):
//   the last     one thread issues 2-D TMA tile loads of the packed rows (64 bytes per row =
//                two stages) into a staging ring (64-byte swizzle, no multicast)
//   warps 10-17  two teams widen the frame rows, thread = one row, 32 bytes -> 128 bytes per stage,
//                written to tensor memory (the MMA reads its A operand from there); they take alternate stages
//   warps 18-25  (18-21) two teams widen the unit rows the same way into shared memory
//   warps 8, 9   rank 0: issue the MMAs (4 per stage and part, K = 64 each) and the commits, which arrive in both CTAs; a warp has a part
//                with its accumulator.  The epilogue reads one accumulator after the other, so one part runs ahead (by
//                up to the ring's six stages) and its epilogue is hidden behind the other's MMAs.
//   warps 0-7    epilogue: accumulator -> Sign/threshold -> repacked bits (or int32 output), two warps per tensor-memory lane quarter
// A stage of both operands is one barrier of rank 0, on which the widening warps of both CTAs arrive.
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles of both CTAs fall
// through to the common teardown and the device status word is set.
//
// What bounds it, measured on B200: the widening (about 600 clocks per stage of 256 x 256 outputs against 512 of MMA).  A CTA that
// widened 128 frames and 192 units by itself took 720 clocks per stage of 128 x 192 outputs (384 of MMA).  65536 x 4096 x 4096, int32 out,
// 483 -> 394 us; 4096 x 2048 x 4096 24.0 -> 22.2 us (its tiles have 8 stages, so the int32 epilogue counts there, and 256
// tiles are 3.5 turns of 74 pairs).
#include "bnn_common.cuh"
#include "tcgen05.cuh"
#include "xnor_both.cuh"

namespace bnn {

namespace {

using namespace tc;

constexpr int BM = 128;                                   // frames per CTA
constexpr int PARTS = 2;
constexpr int BK = 256;                                   // bits of K per stage = nibbles per widened row
constexpr int ROW_BYTES = BK / 2;                         // widened bytes per row and stage (128)
constexpr int STAGES = 6;                                 // even: a stage always belongs to the same team of producers
constexpr int EPI_WARPS = 8, MMA_WARP = 8, PROD_WARP0 = 10, TEAMS = 2, A_WARPS = BM / 32;
constexpr int GROUPS = 3;                                 // staging ring: groups of two stages (an odd last stage has an empty partner)
constexpr int GA_BYTES = BM * 64;
constexpr uint32_t A_COLS = ROW_BYTES / 4;                // 32-bit columns per A stage
constexpr uint32_t SF_COLS = 32, TMEM_COLS = 512;

// PN: units per part, 128 or 64.
template <int PN> struct Tile {
    static constexpr int BN = PARTS * PN, BR = BN / 2, B_WARPS = BR / 32;              // units per tile; unit rows per CTA: half of each part
    static constexpr int PART_BYTES = PN / 2 * ROW_BYTES, STAGE_BYTES = PARTS * PART_BYTES;   // only the unit operand lives in shared memory
    static constexpr int TMA_WARP = PROD_WARP0 + TEAMS * (A_WARPS + B_WARPS), THREADS = (TMA_WARP + 1) * 32;
    static constexpr int GB_BYTES = BR * 64, GROUP_BYTES = GA_BYTES + GB_BYTES;
    static constexpr uint32_t TMEM_A_COL = BN;                                          // A stages start after the two accumulators
    static constexpr uint32_t TMEM_SF_COL = TMEM_A_COL + STAGES * A_COLS;               // block scales: 16 columns per operand
    static_assert(TMEM_SF_COL + SF_COLS <= TMEM_COLS, "tensor memory columns");
};

// With int32 output each epilogue warp needs two staging blocks of 32 rows x 128 bytes (1024-byte aligned).
template <bool STORE_C> struct Cfg {
    static constexpr int CSTAGE_BYTES = STORE_C ? EPI_WARPS * 2 * 32 * 128 : 0;
};

struct Control {
    int T[EPI_WARPS][64];            // per epilogue warp: threshold + kMagicBits of its units (Sign epilogue only)
    uint64_t full[STAGES], empty[STAGES], acc_full[PARTS], acc_empty[PARTS];
    uint64_t group_full[GROUPS], group_empty[GROUPS];
    uint32_t tmem_base;
    WaitState wait;
};
template <bool STORE_C, int PN> constexpr int smem_bytes() {
    return STAGES * Tile<PN>::STAGE_BYTES + GROUPS * Tile<PN>::GROUP_BYTES + (int)sizeof(Control) + Cfg<STORE_C>::CSTAGE_BYTES + 1024;
}
static_assert(smem_bytes<false, 128>() <= 232448 && smem_bytes<true, 128>() <= 232448, "shared memory of one CTA");

struct ProducerArgs {
    uint32_t smem;        // shared-space address of stage 0
    uint32_t tmem;        // base of the tensor-memory allocation
    Control* ctl;
    volatile int* abort_flag;
    int total;            // stages of all tiles of this pair
    both::Rows rows;
    int rank, lane;
};

// Producer of an operand: thread = row `r` of every tile of this CTA's half; team `team` takes one of the two stages of every
// staging group.  FRAMES: widened rows go to tensor memory, else (unit rows) to shared memory.
// Template arguments say what the loops of the producers have to deal with: code that is there for another case costs this
// one, though it is not executed.
template <int PN, bool FRAMES, bool ZO, bool RAGGED>
__device__ __forceinline__ void produce(const ProducerArgs& a, int r, int team) {
    using T = Tile<PN>;
    constexpr int STAGE_BYTES = T::STAGE_BYTES, PART_BYTES = T::PART_BYTES, GROUP_BYTES = T::GROUP_BYTES;
    constexpr uint32_t TMEM_A_COL = T::TMEM_A_COL;
    Control* ctl = a.ctl;
    // TMEM lane of this thread's frame row: a warp may only touch lanes 32*(warp%4)..+31
    const uint32_t tdst0 = a.tmem + ((uint32_t)(r & ~31) << 16) + TMEM_A_COL;
    // rows of a part in shared memory: K-major core matrices, chunk c of 16 bytes PN / 2 rows apart
    const uint32_t bdst0 = a.smem + (r / (PN / 2)) * PART_BYTES + (r % (PN / 2)) * 16;
    // this row inside a staging group: 64 bytes per row, 16-byte chunk c stored at c ^ ((r/2)%4)
    const uint32_t sw = (uint32_t)(r >> 1) & 3u;
    const uint32_t stg0 = a.smem + STAGES * STAGE_BYTES + (FRAMES ? 0 : GA_BYTES) + r * 64 + (((2u * team) ^ (sw & 2u)) << 4);
    const uint32_t lo = (sw & 1u) << 4;
    const uint32_t full0 = a.rank == 0 ? smem_u32(&ctl->full[0]) : peer_addr(smem_u32(&ctl->full[0]), 0);
    int ks = team, gslot = 0, s = team;
    uint32_t gph = 0, ph = 1;                  // parities to wait for (a fresh barrier passes 1)
    for (int it = team; it < a.total; it += TEAMS) {
        if (!warp_wait(smem_u32(&ctl->group_full[gslot]), gph, a.abort_flag, a.lane)) return;
        const uint32_t src = stg0 + gslot * GROUP_BYTES;
        const uint4 v0 = lds128u(src + lo), v1 = lds128u(src + (lo ^ 16u));
        uint4 o[8];
        both::widen_stage<ZO, RAGGED>(a.rows, ks, v0, v1, o);
        if (!warp_wait(smem_u32(&ctl->empty[s]), ph, a.abort_flag, a.lane)) return;
        if (FRAMES) {
            // 32-bit column 4c + t of the stage = word t of chunk c: the byte order of the
            // K-major shared-memory layout of the other operand
            uint32_t wr[32];
#pragma unroll
            for (int c = 0; c < 8; ++c) { wr[4 * c] = o[c].x; wr[4 * c + 1] = o[c].y; wr[4 * c + 2] = o[c].z; wr[4 * c + 3] = o[c].w; }
            tc_fence_after_sync();      // the MMAs that read these columns come first
            tmem_st32(tdst0 + s * A_COLS, wr);
            tmem_st_wait();
            tc_fence_before_sync();
        } else {
            const uint32_t dst = bdst0 + s * STAGE_BYTES;
#pragma unroll
            for (int c = 0; c < 8; ++c) sts128(dst + c * (PN / 2 * 16), o[c].x, o[c].y, o[c].z, o[c].w);
            fence_proxy_async_smem();
        }
        __syncwarp();
        if (a.lane == 0) {
            if (a.rank == 0) mbar_arrive(full0 + 8u * s);
            else mbar_arrive_cluster(full0 + 8u * s);
            // The staging slot is handed back only here, after the stores that consumed the loaded
            // words: a shared-memory load that has merely been issued does not hold back the TMA
            // write that refills the slot (that write belongs to the async proxy; only the data
            // dependency proves that the load has read its bytes).
            mbar_arrive(smem_u32(&ctl->group_empty[gslot]));
        }
        ks += TEAMS;
        if (ks >= 2 * a.rows.groups()) ks = team;
        if (++gslot == GROUPS) { gslot = 0; gph ^= 1u; }
        if ((s += TEAMS) >= STAGES) { s = team; ph ^= 1u; }
    }
}

template <int PN, bool STORE_C, bool SIGN_PACK>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Tile<PN>::THREADS, 1)
xnor_tc_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ CUtensorMap mapC, int tma_c,
                int M, int N, int K, int32_t* __restrict__ C, int ldc,
                const int32_t* __restrict__ thr, const uint32_t* __restrict__ flip,
                uint32_t* __restrict__ out_bits, int ldob, int zo, TcStatus status) {
    using Tl = Tile<PN>;
    constexpr int BN = Tl::BN, B_WARPS = Tl::B_WARPS, TMA_WARP = Tl::TMA_WARP, STAGE_BYTES = Tl::STAGE_BYTES, PART_BYTES = Tl::PART_BYTES;
    constexpr int GB_BYTES = Tl::GB_BYTES, GROUP_BYTES = Tl::GROUP_BYTES;
    constexpr uint32_t TMEM_A_COL = Tl::TMEM_A_COL, TMEM_SF_COL = Tl::TMEM_SF_COL;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t cstage = smem_u32(smem) + STAGES * STAGE_BYTES + GROUPS * GROUP_BYTES;
    Control* ctl = reinterpret_cast<Control*>(smem + STAGES * STAGE_BYTES + GROUPS * GROUP_BYTES + Cfg<STORE_C>::CSTAGE_BYTES);
    volatile int* abort_flag = &ctl->wait.abort;

    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const both::Rows rows(K);
    const int nks = rows.nks;
    const int n_tiles = ceil_div(N, BN), tiles = ceil_div(M, 2 * BM) * n_tiles;
    const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;      // tiles pair, pair + pairs, ..; unit tiles vary fastest

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full[s]), 2 * (A_WARPS + B_WARPS));     // rank 0: the widening warps of both CTAs
            mbar_init(smem_u32(&ctl->empty[s]), PARTS);                      // a commit of each issuing warp
        }
        for (int b = 0; b < PARTS; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), 2 * EPI_WARPS);          // rank 0: the epilogue warps of both CTAs
        }
        for (int b = 0; b < GROUPS; ++b) {
            mbar_init(smem_u32(&ctl->group_full[b]), 1);            // the issuing thread (+ bytes)
            mbar_init(smem_u32(&ctl->group_empty[b]), TEAMS * (A_WARPS + B_WARPS));  // every warp that reads it
        }
        wait_state_init(&ctl->wait, status);
        mbar_init_fence();
    }
    __syncwarp();
    if (warp == MMA_WARP) tmem_alloc_pair(smem_u32(&ctl->tmem_base), TMEM_COLS);
    tc_fence_before_sync();
    cluster_sync();           // barriers of both CTAs initialised, tensor memory of both allocated
    tc_fence_after_sync();
    const uint32_t tmem = ctl->tmem_base;
    pdl_trigger();
    // The set-up above overlaps the end of the kernel before this one (products of one size in a row, us: 4096 x 2048 x 4096
    // 26.5 -> 23.7, 700 x 1024 x 1024 9.7 -> 7.2).
    pdl_wait();
    if (warp < 4) {
        // Block scales of both operands: every byte 127, the ue8m0 code of 2^0.  The whole
        // region is filled, so the values do not depend on how the scales are laid out in it.
        uint32_t ones[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) ones[j] = 0x7F7F7F7Fu;
        tmem_st32(tmem + ((uint32_t)(warp * 32) << 16) + TMEM_SF_COL, ones);
        tmem_st_wait();
    }
    tc_fence_before_sync();
    cluster_sync();
    tc_fence_after_sync();

    if (warp >= PROD_WARP0) {
        const int my_tiles = pair < tiles ? (tiles - 1 - pair) / pairs + 1 : 0;
        const ProducerArgs pa{smem_u32(smem), tmem, ctl, abort_flag, my_tiles * 2 * rows.groups(), rows, rank, lane};
        if (warp == TMA_WARP) {
            // ---------------- one thread feeds the staging ring, a group of two stages at a time
            if (lane == 0) {
                const uint32_t stg = smem_u32(smem) + STAGES * STAGE_BYTES;
                const int ng = rows.groups();
                int slot = 0;
                uint32_t ph = 1;
                bool ok = true;
                for (int tile = pair; tile < tiles && ok; tile += pairs) {
                    const int n0 = (tile % n_tiles) * BN + rank * (PN / 2), m0 = (tile / n_tiles) * (2 * BM) + rank * BM;
                    for (int g = 0; g < ng; ++g) {
                        ok = mbar_wait_relaxed(smem_u32(&ctl->group_empty[slot]), ph, abort_flag);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&ctl->group_full[slot]), dst = stg + slot * GROUP_BYTES;
                        mbar_arrive_expect_tx(bar, GROUP_BYTES);
                        tma_load_2d(dst, &mapA, g * 16, m0, bar);
                        tma_load_2d(dst + GA_BYTES, &mapB, g * 16, n0, bar);
                        tma_load_2d(dst + GA_BYTES + GB_BYTES / 2, &mapB, g * 16, n0 + PN, bar);
                        if (++slot == GROUPS) { slot = 0; ph ^= 1u; }
                    }
                }
            }
            __syncwarp();
        } else if (warp < PROD_WARP0 + TEAMS * A_WARPS) {
            const int row = (warp & 3) * 32 + lane, team = (warp - PROD_WARP0) / A_WARPS;
            if (zo) produce<PN, true, true, false>(pa, row, team);
            else produce<PN, true, false, false>(pa, row, team);
        } else {
            const int pw = warp - PROD_WARP0 - TEAMS * A_WARPS, team = pw / B_WARPS, row = (pw - team * B_WARPS) * 32 + lane;
            rows.ragged() ? produce<PN, false, false, true>(pa, row, team) : produce<PN, false, false, false>(pa, row, team);
        }
    } else if (warp >= EPI_WARPS) {
        // ---------------- MMA issue: two converged warps of rank 0, each with its part of every tile.  What an issuing warp does
        // besides its MMAs (waits, commits) is time the tensor pipe idles unless the other warp fills it.
        const int part = warp - MMA_WARP;
        constexpr uint32_t idesc = instr_desc_mxf4(2 * BM, PN);
        const uint32_t sfa = tmem + TMEM_SF_COL, sfb = tmem + TMEM_SF_COL + SF_COLS / 2;
        const uint64_t desc = smem_desc_kmajor(smem_u32(smem) + part * PART_BYTES, PN / 2 * 16, 128);
        const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
        constexpr uint32_t kStepJ = (2 * (PN / 2) * 16) >> 4, kStepS = STAGE_BYTES >> 4;
        const uint32_t d = tmem + (uint32_t)(part * PN);
        int s = 0;
        uint32_t ph = 0, pacc = 1;
        bool ok = rank == 0;
        for (int tile = pair; tile < tiles && ok; tile += pairs) {
            ok = warp_wait(smem_u32(&ctl->acc_empty[part]), pacc, abort_flag, lane);
            if (!ok) break;
            pacc ^= 1u;
            tc_fence_after_sync();
            const bool beyond = (tile % n_tiles) * BN + part * PN >= N;      // no such units: nothing to multiply
            for (int ks = 0; ks < 2 * rows.groups(); ++ks) {
                ok = warp_wait(smem_u32(&ctl->full[s]), ph, abort_flag, lane);
                if (!ok) break;
                tc_fence_after_sync();
                // the address field (16-byte units) is advanced by plain additions: the ring lies below 2^14 * 16
                // bytes.  An MMA takes 64 positions of K = 32 bytes: 8 columns of A, two 16-byte chunks of B
                const uint32_t db = desc_lo + (uint32_t)s * kStepS;
                const uint32_t ta = tmem + TMEM_A_COL + s * A_COLS;
                if (elect_one()) {
                    if (ks < nks && !beyond) {        // (not the empty partner of an odd last stage)
                        mma_mxf4_ts_pair(d, ta, db, desc_hi, idesc, sfa, sfb, ks != 0);
                        mma_mxf4_ts_pair(d, ta + 8, db + kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                        mma_mxf4_ts_pair(d, ta + 16, db + 2 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                        mma_mxf4_ts_pair(d, ta + 24, db + 3 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                    }
                    mma_commit_pair(smem_u32(&ctl->empty[s]));
                }
                if (++s == STAGES) { s = 0; ph ^= 1u; }
            }
            if (ok && elect_one()) mma_commit_pair(smem_u32(&ctl->acc_full[part]));
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: thread = one frame (TMEM lane); of a part's units warps 0-3 take the first half, warps 4-7 the second
        const int half = warp >> 2, quarter = warp & 3;
        const float magic = __int_as_float(kMagicBits);
        uint32_t par = 0;
        bool ok = true;
        for (int tile = pair; tile < tiles && ok; tile += pairs, par ^= 1u) {
            const int m0 = (tile / n_tiles) * (2 * BM) + rank * BM + quarter * 32, m = m0 + lane;
            for (int part = 0; part < PARTS; ++part) {
                const int n0 = (tile % n_tiles) * BN + part * PN + half * (PN / 2);       // the first of this warp's PN / 2 units
                if (SIGN_PACK) {
#pragma unroll
                    for (int h = 0; h < PN / 64; ++h) ctl->T[warp][h * 32 + lane] = kMagicBits + (n0 + h * 32 + lane < N ? thr[n0 + h * 32 + lane] : 0);
                    __syncwarp();
                }
                ok = warp_wait_relaxed(smem_u32(&ctl->acc_full[part]), par, abort_flag, lane);
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(part * PN + half * (PN / 2));
                uint32_t words[PN / 64];
#pragma unroll
                for (int g = 0; g < PN / 64; ++g) {
                    uint32_t acc[32];
                    tmem_ld32(taddr + g * 32, acc);
                    tmem_ld_wait();
                    if (g + 1 == PN / 64) {
                        // the accumulator is read: the part's next tile may start on it
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive_cluster(peer_addr(smem_u32(&ctl->acc_empty[part]), 0));
                    }
                    const int nb = n0 + g * 32;
                    // The accumulator holds the integer dot product as a float; adding 1.5 * 2^23
                    // leaves that integer, offset by kMagicBits, in the bit pattern of the sum.
                    int q[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) q[j] = __float_as_int(__uint_as_float(acc[j]) + magic);
                    if (STORE_C)
                        both::store_block(cstage + (uint32_t)(warp * 8192), PN == 64 ? part : g & 1, g == 0, g + 1 == PN / 64, q, &mapC, tma_c, C, ldc, M, N,
                                          m0, nb, lane);
                    if (SIGN_PACK) {
                        const int valid = N - nb;  // columns of this word that exist
                        words[g] = valid > 0 ? (both::sign_word(q, ctl->T[warp] + g * 32) ^ __ldg(flip + (nb >> 5))) & (valid < 32 ? (1u << valid) - 1u : 0xFFFFFFFFu) : 0u;
                    }
                }
                if (SIGN_PACK) {
                    if (m < M) {
                        const int nw = words_for(N), w0 = n0 >> 5;
                        uint32_t* dst = out_bits + (size_t)m * ldob + w0;
                        if (PN == 128 && w0 + 2 <= nw) {   // rows are 16-byte aligned, n0/32 is even
                            *reinterpret_cast<uint2*>(dst) = make_uint2(words[0], words[PN / 64 - 1]);
                        } else if (w0 < nw) {
                            dst[0] = words[0];
                        }
                    }
                    __syncwarp();           // T is read
                }
            }
        }
        if (STORE_C && lane == 0) bulk_wait<0>();
    }

    // ---------------- teardown: every thread arrives here, also after an aborted wait
    __syncwarp();
    tc_fence_before_sync();
    cluster_sync();           // nobody reads the partner's shared or tensor memory any more
    if (warp == MMA_WARP) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && ctl->wait.abort) atomicExch(status.word, 1);
}

template <int PN, bool STORE_C, bool SIGN_PACK>
int launch_variant(const uint32_t* Ap, int ldap, const uint32_t* Wp, int ldwp, int M, int N, int K,
                   int32_t* C, int ldc, const int32_t* thr, const uint32_t* flip,
                   uint32_t* out_bits, int ldob, int zo, cudaStream_t st) {
    auto kern = xnor_tc_kernel<PN, STORE_C, SIGN_PACK>;
    constexpr int SMEM = smem_bytes<STORE_C, PN>();
    const int sm_count = device_sm_count();
    if (sm_count < 2 || !ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM)) return BNN_ERR_CUDA;
    const long long tiles = (long long)ceil_div(M, 2 * BM) * ceil_div(N, Tile<PN>::BN);
    const int grid = 2 * (int)(tiles < sm_count / 2 ? tiles : sm_count / 2);
    const TcStatus status = tc_status();
    if (!status.word) return BNN_ERR_CUDA;
    // tensor maps of the two packed operands: [rows][ceil(K/32) words] with the caller's pitch;
    // boxes of 16 words x (128 | PN / 2) rows; whatever lies outside the tensor reads as zero
    CUtensorMap mapA, mapB;
    if (!encode_packed_map(&mapA, Ap, ldap, M, K, BM) || !encode_packed_map(&mapB, Wp, ldwp, N, K, PN / 2))
        return BNN_ERR_CUDA;
    const int tma_c = C && ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
    CUtensorMap mapC{};
    if (tma_c && !encode_int32_map(&mapC, C, ldc, M, N)) return BNN_ERR_CUDA;
    const cudaError_t e = launch_pdl(kern, dim3(grid), dim3(Tile<PN>::THREADS), SMEM, st, mapA, mapB, mapC, tma_c, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, status);
    return e == cudaSuccess ? launch_status() : BNN_ERR_CUDA;
}

}  // namespace

// The variant with the least estimated time: CTA pairs with parts of 128 or 64 units, or single CTAs.  A launch takes ceil(tiles / CTAs or pairs) turns of nks
// stages and an epilogue, which depends on the results: Sign bits, int32 rows that tile stores take, other int32 rows.  Clocks fitted to 336 sizes on B200
// (64 .. 40000 frames, 100 .. 8192 units, 256 .. 8192 inputs); the choice takes 0.1 % more than the best on the mean, 11 % at most (6996 x 566 x 6524, bound by its stores).
// Measured, us, parts of 128 / of 64 / single: int32 4096 x 2048 x 4096 22.0 / 24.6 / 23.5, 300 x 8000 x 1501 24.4 / 18.5 / 24.5, 6270 x 8192 x 520
// 25.9 / 23.7 / 18.8; Sign bits 4096 x 2048 x 4096 20.3 / 23.9 / 21.8, 11302 x 5912 x 1039 43.6 / 52.3 / 46.1, 6270 x 2048 x 576 10.9 / 9.8 / 7.8.
int launch_xnor_tc(const uint32_t* Ap, int ldap, const uint32_t* Wp, int ldwp, int M, int N,
                   int K, int32_t* C, int ldc, const int32_t* thr, const uint32_t* flip,
                   uint32_t* out_bits, int ldob, int zo, cudaStream_t st) {
    constexpr struct { int frames, units, per_launch, stage, epilogue[3], fixed; } variants[] = {{256, 256, 2, 660, {2300, 4250, 9300}, 1250}, {256, 128, 2, 575, {1050, 1950, 5000}, 0}, {128, 192, 1, 670, {2750, 3200, 10200}, 550}};
    const int results = !C ? 0 : N % 4 == 0 && ldc % 4 == 0 && aligned16(C) ? 1 : 2, sms = device_sm_count();
    int best = 0;
    long long least = -1;
    for (int v = 0; v < 3; ++v) {
        const auto& x = variants[v];
        const long long at_once = sms / x.per_launch, tiles = (long long)ceil_div(M, x.frames) * ceil_div(N, x.units);
        if (at_once < 1) continue;
        const long long clocks = (tiles + at_once - 1) / at_once * ((long long)ceil_div(K, BK) * x.stage + x.epilogue[results]) + x.fixed;
        if (least < 0 || clocks < least) { least = clocks; best = v; }
    }
    if (best == 2) return launch_xnor_cta(Ap, ldap, Wp, ldwp, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, st);
    const bool sp = out_bits != nullptr;
    auto go = [&](auto wide, auto narrow) { return (best == 1 ? narrow : wide)(Ap, ldap, Wp, ldwp, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, st); };
    if (C && sp) return go(launch_variant<128, true, true>, launch_variant<64, true, true>);
    if (C) return go(launch_variant<128, true, false>, launch_variant<64, true, false>);
    return go(launch_variant<128, false, true>, launch_variant<64, false, true>);
}

}  // namespace bnn
