// The XNOR GEMM of xnor_gemm_tc.cu on single CTAs, each with tiles of 128 frames x 192 units.  CTA pairs widen each row for more results, and are faster
// where their tiles of 256 frames fill the chip; a launch that needs one turn of these tiles may need two of those (launch_xnor_tc).
//
// Roles in a CTA of 27 warps (persistent, one CTA per SM):
//   warp 26      one thread issues 2-D TMA tile loads of the packed rows (64 bytes per row =
//                two stages) into a staging ring (64-byte swizzle, no multicast)
//   warps 6-13   two teams widen the frame rows, thread = one row, 32 bytes -> 128 bytes per stage,
//                written to tensor memory (the MMA reads its A operand from there); they take alternate stages
//   warps 14-25  two teams widen the unit rows the same way into shared memory, two stages per iteration
//   warps 4, 5   issue the MMAs (4 per stage, K = 64 each) and the commits; the two warps take the stages in turn
//   warps 0-3    epilogue: accumulator -> Sign/threshold -> repacked bits (or int32 output);
//                two accumulators in tensor memory, so it overlaps the next tile's MMAs
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles fall
// through to the common teardown and the device status word is set.
//
// What bounds it, measured on B200: the widening (two teams per operand; a stage takes about 700 clocks against 384
// of MMA).  6270 x 8192 x 520, one turn of 147 tiles where the pairs take two, us, int32 / Sign bits: 18.8 / 17.3 (pairs 23.7 / 23.1).
#include "bnn_common.cuh"
#include "tcgen05.cuh"
#include "xnor_both.cuh"

namespace bnn {

namespace {

using namespace tc;

constexpr int BM = 128, BN = 192;
constexpr int BK = 256;                                   // bits of K per stage = nibbles per widened row
constexpr int ROW_BYTES = BK / 2;                         // widened bytes per row and stage (128)
constexpr int B_BYTES = BN * ROW_BYTES, STAGE_BYTES = B_BYTES;   // only the unit operand lives in shared memory
constexpr int A_STAGES = 3, B_STAGES = 4;               // rings of the frame operand (tensor memory) and the unit operand
// A stage `it` of the CTA's sequence has barrier it % A_BARS, an even number, so that a barrier always belongs to the same
// team and issuing warp (a wait on a parity holds only for one who has seen every phase before it).
constexpr int A_BARS = 2 * A_STAGES;
static_assert(B_STAGES % 2 == 0, "a stage of units always belongs to the same issuing warp");
constexpr int EPI_WARPS = 4, MMA_WARP = 4, MMA_WARP2 = 5, PROD_WARP0 = 6, TEAMS = 2, A_WARPS = BM / 32, B_WARPS = BN / 32;
constexpr int PROD_WARPS = TEAMS * (A_WARPS + B_WARPS);
constexpr int TMA_WARP = PROD_WARP0 + PROD_WARPS;
constexpr int THREADS = (TMA_WARP + 1) * 32;              // 864
constexpr int GROUPS = 4;                                 // staging ring: groups of two stages (an odd last stage has an empty partner)
constexpr int GA_BYTES = BM * 64, GB_BYTES = BN * 64, GROUP_BYTES = GA_BYTES + GB_BYTES;
constexpr uint32_t TMEM_A_COL = 2 * BN;                   // A stages start after the two accumulators
constexpr uint32_t A_COLS = ROW_BYTES / 4;                // 32-bit columns per A stage
constexpr uint32_t TMEM_SF_COL = TMEM_A_COL + A_STAGES * A_COLS, SF_COLS = 32;   // block scales: 16 columns per operand
constexpr uint32_t TMEM_COLS = 512;

// With int32 output each epilogue warp needs two staging blocks of 32 rows x 128 bytes (1024-byte aligned).
template <bool STORE_C> struct Cfg {
    static constexpr int CSTAGE_BYTES = STORE_C ? EPI_WARPS * 2 * 32 * 128 : 0;
};

struct Control {
    int T[BN];               // per unit: threshold + kMagicBits (Sign epilogue only)
    uint64_t full_a[A_BARS], empty_a[A_BARS], full_b[B_STAGES], empty_b[B_STAGES], acc_full[2], acc_empty[2], started[2];
    uint64_t group_full[GROUPS], group_empty[GROUPS];
    uint32_t tmem_base;
    WaitState wait;
};
template <bool STORE_C> constexpr int smem_bytes() {
    return B_STAGES * STAGE_BYTES + GROUPS * GROUP_BYTES + (int)sizeof(Control) + Cfg<STORE_C>::CSTAGE_BYTES + 1024;
}
static_assert(smem_bytes<false>() <= 232448 && smem_bytes<true>() <= 232448, "shared memory of one CTA");
static_assert(TMEM_SF_COL + SF_COLS <= TMEM_COLS, "tensor memory columns");

struct ProducerArgs {
    uint32_t smem;        // shared-space address of stage 0
    uint32_t tmem;        // base of the tensor-memory allocation
    Control* ctl;
    volatile int* abort_flag;
    int tiles;
    both::Rows rows;
    int lane;
};

// Producer of the frame operand: thread = row `r` of every tile of this CTA; team `team` takes one of the two stages of every
// group, widened rows written to tensor memory.
// Template arguments say what the loops of the producers have to deal with: code that is there for another case costs this
// one, though it is not executed.
template <bool ZO>
__device__ __forceinline__ void produce_a(const ProducerArgs& a, int r, int team) {
    Control* ctl = a.ctl;
    const int my_tiles = (a.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
    const int ng = a.rows.groups(), total = 2 * my_tiles * ng;
    // TMEM lane of this thread's frame row: a warp may only touch lanes 32*(warp%4)..+31
    const uint32_t tdst0 = a.tmem + ((uint32_t)(r & ~31) << 16) + TMEM_A_COL;
    // this row inside a staging group: 64 bytes per row, 16-byte chunk c stored at c ^ ((r/2)%4)
    const uint32_t sw = (uint32_t)(r >> 1) & 3u;
    const uint32_t stg0 = a.smem + B_STAGES * STAGE_BYTES + r * 64 + (((2u * team) ^ (sw & 2u)) << 4);
    const uint32_t lo = (sw & 1u) << 4;
    int ks = team;
    for (int it = team; it < total; it += TEAMS) {
        const int g = it >> 1, gslot = g % GROUPS;
        if (!warp_wait(smem_u32(&ctl->group_full[gslot]), (uint32_t)((g / GROUPS) & 1), a.abort_flag, a.lane)) break;
        const uint32_t src = stg0 + gslot * GROUP_BYTES;
        const uint4 v0 = lds128u(src + lo), v1 = lds128u(src + (lo ^ 16u));
        const int s = it % A_STAGES;
        const int e = it + A_BARS - A_STAGES;          // the stage that had this slot; a fresh barrier passes parity 1
        if (!warp_wait(smem_u32(&ctl->empty_a[e % A_BARS]), (uint32_t)(((e / A_BARS) & 1) ^ 1), a.abort_flag, a.lane)) break;
        uint4 o[8];
        both::widen_stage<ZO, false>(a.rows, ks, v0, v1, o);
        // 32-bit column 4c + t of the stage = word t of chunk c: the byte order of the
        // K-major shared-memory layout of the other operand
        uint32_t wr[32];
#pragma unroll
        for (int c = 0; c < 8; ++c) { wr[4 * c] = o[c].x; wr[4 * c + 1] = o[c].y; wr[4 * c + 2] = o[c].z; wr[4 * c + 3] = o[c].w; }
        tc_fence_after_sync();          // the MMAs that read these columns come first
        tmem_st32(tdst0 + s * A_COLS, wr);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (a.lane == 0) {
            mbar_arrive(smem_u32(&ctl->full_a[it % A_BARS]));
            // The staging slot is handed back only here, after the stores that consumed the loaded
            // words: a shared-memory load that has merely been issued does not hold back the TMA
            // write that refills the slot (that write belongs to the async proxy; only the data
            // dependency proves that the load has read its bytes).
            mbar_arrive(smem_u32(&ctl->group_empty[gslot]));
        }
        ks += TEAMS;
        if (ks >= 2 * ng) ks = team;
    }
}

// Producer of the unit operand: thread = row `r`; the teams take the staging groups in turn, two stages per
// iteration, so the fixed costs of an iteration (group wait, proxy fence, warp barrier, release) are paid once per
// two stages; widened rows go to shared memory, each team to its half of the ring.
template <bool RAGGED>
__device__ __forceinline__ void produce_b(const ProducerArgs& a, int r, int team) {
    Control* ctl = a.ctl;
    const int my_tiles = (a.tiles - 1 - (int)blockIdx.x) / (int)gridDim.x + 1;
    const int ng = a.rows.groups(), total = my_tiles * ng;
    const int s = 2 * team;
    const uint32_t dst0 = a.smem + s * STAGE_BYTES + r * 16;
    const uint32_t stg0 = a.smem + B_STAGES * STAGE_BYTES + GA_BYTES + r * 64;
    const uint32_t sw = (uint32_t)(r >> 1) & 3u;
    uint32_t ph = 1;
    int kg = team;
    for (int g = team; g < total; g += TEAMS) {
        while (kg >= ng) kg -= ng;
        const int gslot = g % GROUPS;
        if (!warp_wait(smem_u32(&ctl->group_full[gslot]), (uint32_t)((g / GROUPS) & 1), a.abort_flag, a.lane)) break;
        const uint32_t src = stg0 + gslot * GROUP_BYTES;
        const uint4 v0 = lds128u(src + ((0u ^ sw) << 4)), v1 = lds128u(src + ((1u ^ sw) << 4));
        const uint4 v2 = lds128u(src + ((2u ^ sw) << 4)), v3 = lds128u(src + ((3u ^ sw) << 4));
        if (!warp_wait(smem_u32(&ctl->empty_b[s]), ph, a.abort_flag, a.lane)) break;
        uint4 o[8];
        both::widen_stage<false, RAGGED>(a.rows, 2 * kg, v0, v1, o);
#pragma unroll
        for (int c = 0; c < 8; ++c) sts128(dst0 + c * (BN * 16), o[c].x, o[c].y, o[c].z, o[c].w);
        if (!warp_wait(smem_u32(&ctl->empty_b[s + 1]), ph, a.abort_flag, a.lane)) break;
        both::widen_stage<false, RAGGED>(a.rows, 2 * kg + 1, v2, v3, o);
#pragma unroll
        for (int c = 0; c < 8; ++c) sts128(dst0 + STAGE_BYTES + c * (BN * 16), o[c].x, o[c].y, o[c].z, o[c].w);
        fence_proxy_async_smem();
        __syncwarp();
        if (a.lane == 0) {
            mbar_arrive(smem_u32(&ctl->full_b[s]));
            mbar_arrive(smem_u32(&ctl->full_b[s + 1]));
            mbar_arrive(smem_u32(&ctl->group_empty[gslot]));   // after the stores that consumed the loaded words (see produce_a)
        }
        ph ^= 1u;
        kg += TEAMS;
    }
}

template <bool STORE_C, bool SIGN_PACK>
__global__ void __launch_bounds__(THREADS, 1)
xnor_cta_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapB,
                const __grid_constant__ CUtensorMap mapC, int tma_c,
                int M, int N, int K, int32_t* __restrict__ C, int ldc,
                const int32_t* __restrict__ thr, const uint32_t* __restrict__ flip,
                uint32_t* __restrict__ out_bits, int ldob, int zo, TcStatus status) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t cstage = smem_u32(smem) + B_STAGES * STAGE_BYTES + GROUPS * GROUP_BYTES;
    Control* ctl = reinterpret_cast<Control*>(smem + B_STAGES * STAGE_BYTES + GROUPS * GROUP_BYTES + Cfg<STORE_C>::CSTAGE_BYTES);
    volatile int* abort_flag = &ctl->wait.abort;

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const both::Rows rows(K);
    const int nks = rows.nks;
    const int m_tiles = ceil_div(M, BM), n_tiles = ceil_div(N, BN);
    const int tiles = m_tiles * n_tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < A_BARS; ++s) {
            mbar_init(smem_u32(&ctl->full_a[s]), A_WARPS);
            mbar_init(smem_u32(&ctl->empty_a[s]), 1);
        }
        for (int s = 0; s < B_STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full_b[s]), B_WARPS);
            mbar_init(smem_u32(&ctl->empty_b[s]), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 2);       // one commit of each issuing warp
            mbar_init(smem_u32(&ctl->started[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), EPI_WARPS);
        }
        for (int b = 0; b < GROUPS; ++b) {
            mbar_init(smem_u32(&ctl->group_full[b]), 1);            // the issuing thread (+ bytes)
            mbar_init(smem_u32(&ctl->group_empty[b]), TEAMS * A_WARPS + B_WARPS);  // every warp that reads it
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
    // The set-up above overlaps the end of the kernel before this one (products of one size in a row, us: 4096 x 2048 x 4096
    // 26.5 -> 23.7, 700 x 1024 x 1024 9.7 -> 7.2).
    pdl_wait();
    if (warp < EPI_WARPS) {
        // Block scales of both operands: every byte 127, the ue8m0 code of 2^0.  The whole
        // region is filled, so the values do not depend on how the scales are laid out in it.
        uint32_t ones[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) ones[j] = 0x7F7F7F7Fu;
        tmem_st32(tmem + ((uint32_t)(warp * 32) << 16) + TMEM_SF_COL, ones);
        tmem_st_wait();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();

    if (warp >= PROD_WARP0) {
        const ProducerArgs pa{smem_u32(smem), tmem, ctl, abort_flag, tiles, rows, lane};
        if (warp == TMA_WARP) {
            // ---------------- one thread feeds the staging ring, a group of two stages at a time
            if (lane == 0) {
                const uint32_t stg = smem_u32(smem) + B_STAGES * STAGE_BYTES;
                const int ng = rows.groups();
                int gc = 0;
                bool ok = true;
                for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
                    const int n0 = (tile % n_tiles) * BN, m0 = (tile / n_tiles) * BM;   // unit tiles vary fastest
                    for (int g = 0; g < ng; ++g, ++gc) {
                        const int slot = gc % GROUPS;
                        if (gc >= GROUPS) {
                            ok = mbar_wait_relaxed(smem_u32(&ctl->group_empty[slot]), (uint32_t)(((gc / GROUPS) - 1) & 1), abort_flag);
                            if (!ok) break;
                        }
                        const uint32_t bar = smem_u32(&ctl->group_full[slot]);
                        mbar_arrive_expect_tx(bar, GROUP_BYTES);
                        tma_load_2d(stg + slot * GROUP_BYTES, &mapA, g * 16, m0, bar);
                        tma_load_2d(stg + slot * GROUP_BYTES + GA_BYTES, &mapB, g * 16, n0, bar);
                    }
                }
            }
            __syncwarp();
        } else if (warp < PROD_WARP0 + TEAMS * A_WARPS) {
            const int row = (warp & 3) * 32 + lane, team = (warp - PROD_WARP0) / A_WARPS;
            zo ? produce_a<true>(pa, row, team) : produce_a<false>(pa, row, team);
        } else {
            const int pw = warp - PROD_WARP0 - TEAMS * A_WARPS, team = pw / B_WARPS, row = (pw - team * B_WARPS) * 32 + lane;
            rows.ragged() ? produce_b<true>(pa, row, team) : produce_b<false>(pa, row, team);
        }
    } else if (warp == MMA_WARP || warp == MMA_WARP2) {
        // ---------------- MMA issue: two converged warps, which take the CTA's stages in turn and accumulate into the
        // same accumulator (the sums are exact integers, so their order does not matter; only the stage that
        // overwrites the accumulator has to come first, see `started`).  What an issuing warp does besides its
        // MMAs (waits, commits) is time the tensor pipe idles unless the other warp fills it.
        const int w = warp - MMA_WARP;
        constexpr uint32_t idesc = instr_desc_mxf4(BM, BN);
        const uint32_t sfa = tmem + TMEM_SF_COL, sfb = tmem + TMEM_SF_COL + SF_COLS / 2;
        const uint64_t desc = smem_desc_kmajor(smem_u32(smem), BN * 16, 128);
        const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
        constexpr uint32_t kStepJ = (2 * BN * 16) >> 4, kStepS = STAGE_BYTES >> 4;
        int sa = w, ba = w, sb = w;     // this warp's next stage: slot of the A ring, its barrier, slot of the B ring
        uint32_t pa = 0, pb = 0;        // ... and the parities the `full` barriers show next
        int tl = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++tl) {
            const int b = tl & 1;
            ok = warp_wait(smem_u32(&ctl->acc_empty[b]), (uint32_t)(((tl >> 1) & 1) ^ 1), abort_flag, lane);
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t d = tmem + (uint32_t)(b * BN);
            for (int ks = w; ks < 2 * rows.groups(); ks += 2) {
                ok = warp_wait(smem_u32(&ctl->full_b[sb]), pb, abort_flag, lane) && warp_wait(smem_u32(&ctl->full_a[ba]), pa, abort_flag, lane) &&
                     (ks != 1 || warp_wait(smem_u32(&ctl->started[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane));
                if (!ok) break;
                tc_fence_after_sync();
                // the address field (16-byte units) is advanced by plain additions: the ring lies below 2^14 * 16
                // bytes.  An MMA takes 64 positions of K = 32 bytes: 8 columns of A, two 16-byte chunks of B
                const uint32_t db = desc_lo + (uint32_t)sb * kStepS;
                const uint32_t ta = tmem + TMEM_A_COL + sa * A_COLS;
                if (ks == nks) {        // the empty partner of an odd last stage
                    if (elect_one()) {
                        mma_commit(smem_u32(&ctl->empty_a[ba]));
                        mma_commit(smem_u32(&ctl->empty_b[sb]));
                    }
                } else if (elect_one()) {
                    mma_mxf4_ts(d, ta, db, desc_hi, idesc, sfa, sfb, ks != 0);
                    if (ks == 0) mma_commit(smem_u32(&ctl->started[b]));
                    mma_mxf4_ts(d, ta + 8, db + kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                    mma_mxf4_ts(d, ta + 16, db + 2 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                    mma_mxf4_ts(d, ta + 24, db + 3 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                    mma_commit(smem_u32(&ctl->empty_a[ba]));
                    mma_commit(smem_u32(&ctl->empty_b[sb]));
                }
                if ((sa += 2) >= A_STAGES) sa -= A_STAGES;
                if ((ba += 2) >= A_BARS) { ba -= A_BARS; pa ^= 1u; }
                if ((sb += 2) >= B_STAGES) { sb -= B_STAGES; pb ^= 1u; }
            }
            if (ok && elect_one()) mma_commit(smem_u32(&ctl->acc_full[b]));
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: 128 threads, thread = one frame (TMEM lane)
        const int row_in_tile = warp * 32 + lane;
        const float magic = __int_as_float(kMagicBits);
        int tl = 0;
        bool ok = true;
        for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x, ++tl) {
            const int n0 = (tile % n_tiles) * BN, m0 = (tile / n_tiles) * BM;   // unit tiles vary fastest
            const int m = m0 + row_in_tile;
            if (SIGN_PACK) {
                epi_bar_sync();  // previous tile's readers of T are done
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int nl = row_in_tile + h * 128, n = n0 + nl;
                    if (nl < BN) ctl->T[nl] = kMagicBits + (n < N ? thr[n] : 0);
                }
                epi_bar_sync();
            }
            const int b = tl & 1;
            // all four epilogue warps take the same decision, so none is left at a barrier
            ok = epi_all(warp_wait_relaxed(smem_u32(&ctl->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane));
            if (!ok) break;
            tc_fence_after_sync();
            const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(b * BN);
            uint32_t words[BN / 32];
#pragma unroll
            for (int g = 0; g < BN / 32; ++g) {
                uint32_t acc[32];
                tmem_ld32(taddr + g * 32, acc);
                tmem_ld_wait();
                if (g + 1 == BN / 32) {
                    // the accumulator is read: the MMA warps may start the tile after the next on it
                    tc_fence_before_sync();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                }
                const int nb = n0 + g * 32;
                // The accumulator holds the integer dot product as a float; adding 1.5 * 2^23
                // leaves that integer, offset by kMagicBits, in the bit pattern of the sum.
                int q[32];
#pragma unroll
                for (int j = 0; j < 32; ++j) q[j] = __float_as_int(__uint_as_float(acc[j]) + magic);
                if (STORE_C)
                    both::store_block(cstage + (uint32_t)(warp * 8192), g & 1, g == 0, g + 1 == BN / 32, q, &mapC, tma_c, C, ldc, M, N, m0 + warp * 32, nb, lane);
                if (SIGN_PACK) {
                    const int valid = N - nb;  // columns of this word that exist
                    words[g] = valid > 0 ? (both::sign_word(q, ctl->T + g * 32) ^ __ldg(flip + (nb >> 5))) & (valid < 32 ? (1u << valid) - 1u : 0xFFFFFFFFu) : 0u;
                }
            }
            if (SIGN_PACK && m < M) {
                const int nw = words_for(N), w0 = n0 >> 5;
                uint32_t* dst = out_bits + (size_t)m * ldob + w0;
                if (w0 + BN / 32 <= nw) {   // 6 words; rows are 16-byte aligned, n0/32 is a multiple of 6
#pragma unroll
                    for (int i = 0; i < BN / 64; ++i)
                        reinterpret_cast<uint2*>(dst)[i] = make_uint2(words[2 * i], words[2 * i + 1]);
                } else {
#pragma unroll
                    for (int g = 0; g < BN / 32; ++g)
                        if (w0 + g < nw) dst[g] = words[g];
                }
            }
        }
        if (STORE_C && lane == 0) bulk_wait<0>();
    }

    // ---------------- teardown: every thread arrives here, also after an aborted wait
    tc_fence_before_sync();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && ctl->wait.abort) atomicExch(status.word, 1);
}

template <bool STORE_C, bool SIGN_PACK>
int launch_variant(const uint32_t* Ap, int ldap, const uint32_t* Wp, int ldwp, int M, int N, int K,
                   int32_t* C, int ldc, const int32_t* thr, const uint32_t* flip,
                   uint32_t* out_bits, int ldob, int zo, cudaStream_t st) {
    auto kern = xnor_cta_kernel<STORE_C, SIGN_PACK>;
    constexpr int SMEM = smem_bytes<STORE_C>();
    const int sm_count = device_sm_count();
    if (sm_count <= 0 || !ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM)) return BNN_ERR_CUDA;
    const int tiles = ceil_div(M, BM) * ceil_div(N, BN);
    const int grid = tiles < sm_count ? tiles : sm_count;
    const TcStatus status = tc_status();
    if (!status.word) return BNN_ERR_CUDA;
    // tensor maps of the two packed operands: [rows][ceil(K/32) words] with the caller's pitch;
    // boxes of 16 words x (128 | 192) rows; whatever lies outside the tensor reads as zero
    CUtensorMap mapA, mapB;
    if (!encode_packed_map(&mapA, Ap, ldap, M, K, BM) || !encode_packed_map(&mapB, Wp, ldwp, N, K, BN))
        return BNN_ERR_CUDA;
    const int tma_c = C && ldc % 4 == 0 && (reinterpret_cast<uintptr_t>(C) & 15) == 0;
    CUtensorMap mapC{};
    if (tma_c && !encode_int32_map(&mapC, C, ldc, M, N)) return BNN_ERR_CUDA;
    const cudaError_t e = launch_pdl(kern, dim3(grid), dim3(THREADS), SMEM, st, mapA, mapB, mapC, tma_c, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, status);
    return e == cudaSuccess ? launch_status() : BNN_ERR_CUDA;
}

}  // namespace

int launch_xnor_cta(const uint32_t* Ap, int ldap, const uint32_t* Wp, int ldwp, int M, int N,
                    int K, int32_t* C, int ldc, const int32_t* thr, const uint32_t* flip,
                    uint32_t* out_bits, int ldob, int zo, cudaStream_t st) {
    const bool sp = out_bits != nullptr;
    if (C && sp) return launch_variant<true, true>(Ap, ldap, Wp, ldwp, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, st);
    if (C) return launch_variant<true, false>(Ap, ldap, Wp, ldwp, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, st);
    return launch_variant<false, true>(Ap, ldap, Wp, ldwp, M, N, K, C, ldc, thr, flip, out_bits, ldob, zo, st);
}

}  // namespace bnn
