// Binary hidden layers with fan-ins above 2048, in runs or by themselves, where that is estimated to be faster (xnor_pair_clocks): the layers of xnor_gemm_res.cu
// (weights resident in shared memory, one launch for a run, frame tiles handed from layer to layer through counters) on CTA pairs.
//
// There a CTA widens its frames for 192 units, or for 128 where the fan-in is above 2048, because the weights of more would not fit its shared
// memory; with 128 units a stage takes 430 clocks of widening for 256 of MMA.  Here a pair of CTAs (cluster of two, one per
// SM of a TPC) owns 256 units and each CTA holds half of their weights: 128 rows, 16 KB per stage of 256 positions, twelve stages.
// A tile is 256 frames x two parts of 128 units; each CTA widens its own 128 frames, and what is widened serves both parts, 512
// clocks of MMA per stage.
//
// Roles in a CTA of 20 warps:
//   warps 0-7    epilogue: accumulator -> threshold -> repacked bits, two warps per tensor-memory lane quarter, each with half of every part's units
//   warps 8, 9   rank 0: issue the MMAs (4 per stage and part, K = 64 each) and the commits, which arrive in both CTAs; a warp has a part with
//                its accumulator.  The epilogue reads one accumulator after the other, so one part runs ahead (by up to
//                the ring's six stages) and its epilogue is hidden behind the other's MMAs.
//   warp 10      one thread issues the TMA loads of the packed frame rows (64 bytes per row = two stages) into a staging ring
//   warp 11      one thread issues the TMA loads of the weight stages of all layers, round a ring of twelve
//   warps 12-19  two teams of four warps widen the frame rows into tensor memory; the teams take alternate stages
// What bounds it, measured on B200: 65536 frames x 3072, about 660 clocks per stage against 512 of MMA; a pass of the network of five
// such layers 3156 -> 2934 us.  (Its 640 threads have 96 registers each; the epilogue spills 72 bytes.)
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles of both CTAs fall
// through to the common teardown and the device status word is set.
#include "bnn_common.cuh"
#include "tcgen05.cuh"
#include "xnor_widen.cuh"

namespace bnn {

namespace {

using namespace tc;

constexpr int BM = 128;                                   // frames per CTA
constexpr int PARTS = 2, PN = 128, BN = PARTS * PN;       // units per part and tile
constexpr int BK = 256;                                   // positions of K per stage
constexpr int ROW_BYTES = BK / 2;                         // widened bytes per row and stage (128)
constexpr int PART_BYTES = PN / 2 * ROW_BYTES, B_BYTES = PARTS * PART_BYTES;      // one stage of weights in one CTA
constexpr int SLOTS = 12;                                 // weight stages
constexpr int A_STAGES = 6;                               // even: a slot always belongs to the same team
constexpr int EPI_WARPS = 8, MMA_WARP = 8, TMA_WARP = 10, WEIGHT_WARP = 11, PROD_WARP0 = 12, A_WARPS = BM / 32, TEAMS = 2;
constexpr int THREADS = (PROD_WARP0 + TEAMS * A_WARPS) * 32;              // 640
constexpr int GROUPS = 3;                                 // staging ring of the packed frame rows: groups of two stages (an odd last stage has an empty partner)
constexpr int GROUP_BYTES = BM * 64;
constexpr uint32_t A_COLS = ROW_BYTES / 4;                // 32-bit columns per A stage
constexpr uint32_t TMEM_A_COL = BN;                       // A stages start after the two accumulators
constexpr uint32_t TMEM_SF_COL = TMEM_A_COL + A_STAGES * A_COLS, SF_COLS = 32, TMEM_COLS = 512;
static_assert(TMEM_SF_COL + SF_COLS <= TMEM_COLS, "tensor memory columns");

struct Control {
    float T[EPI_WARPS][PARTS][PN / 2];       // per epilogue warp: threshold less 1/2 of its units
    uint64_t full_a[A_STAGES], empty_a[A_STAGES], full_b[SLOTS], b_free[SLOTS], acc_full[PARTS], acc_empty[PARTS];
    uint64_t group_full[GROUPS], group_empty[GROUPS];
    uint32_t tmem_base;
    WaitState wait;
};
constexpr int SMEM_BYTES = SLOTS * B_BYTES + GROUPS * GROUP_BYTES + (int)sizeof(Control) + 1024;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

struct Layer {
    const int32_t* thr;
    const uint32_t* flip;
    uint32_t* out_bits;
};
struct Args {
    Layer layer[kXnorStackMax];
    int n_layers;
    int M, N, K, ldob, zo;
    TcStatus status;
    int* progress;           // [n_layers - 1][frame tiles of 128] arrival counters, zero at launch
};
struct Maps {
    CUtensorMap in[kXnorStackMax], weights[kXnorStackMax];
};

// Frame tiles (of 256) of this pair, which works on unit tile `nt`: first, first + step, ...
struct Share {
    int nt, first, step, count;
    __device__ __forceinline__ Share(int m_tiles, int n_tiles) {
        const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
        nt = pair % n_tiles;
        first = pair / n_tiles;
        step = (pairs - 1 - nt) / n_tiles + 1;
        count = first < m_tiles ? (m_tiles - 1 - first) / step + 1 : 0;
    }
};

// Wait until `*p` has reached `target` (acquire at GPU scope); bounded like the mbarrier waits.
__device__ __forceinline__ bool wait_counter(const int* p, int target, volatile int* abort_flag) {
    const long long t0 = clock64(), limit = wait_limit_of(abort_flag);
#pragma unroll 1
    while (true) {
        int v;
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
        if (v >= target) return true;
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
            *abort_flag = 1;
            return false;
        }
        __nanosleep(64);
    }
}

// Producer of the frame operand: thread = row `r` of every tile of this CTA; team `team` takes one of the two stages of every staging
// group.  Positions >= K need no care: the weights' nibbles are +0 there.
template <bool ZO>
__device__ __forceinline__ void produce(uint32_t staging, uint32_t tmem, Control* ctl, volatile int* abort_flag, int total, int rank, int r, int team, int lane) {
    const uint32_t tdst0 = tmem + ((uint32_t)(r & ~31) << 16) + TMEM_A_COL;     // a warp may only touch lanes 32*(warp%4)..+31
    // this row inside a staging group: 64 bytes per row, 16-byte chunk c stored at c ^ ((r/2)%4)
    const uint32_t sw = (uint32_t)(r >> 1) & 3u;
    const uint32_t stg0 = staging + r * 64 + (((2u * team) ^ (sw & 2u)) << 4), lo = (sw & 1u) << 4;
    const uint32_t full0 = rank == 0 ? smem_u32(&ctl->full_a[0]) : peer_addr(smem_u32(&ctl->full_a[0]), 0);
    int gslot = 0, s = team;
    uint32_t gph = 0, ph = 1;                  // parities to wait for (a fresh barrier passes 1)
    for (int it = team; it < total; it += TEAMS) {
        if (!warp_wait(smem_u32(&ctl->group_full[gslot]), gph, abort_flag, lane)) return;
        const uint32_t src = stg0 + gslot * GROUP_BYTES;
        const uint4 v0 = lds128u(src + lo), v1 = lds128u(src + (lo ^ 16u));
        const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
        // 32-bit column 4c + t of the stage = word t of chunk c: the byte order of the
        // K-major shared-memory layout of the other operand
        uint32_t wr[32];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const uint4 o = ZO ? widen01(w[c]) : widen(w[c]);
            wr[4 * c] = o.x; wr[4 * c + 1] = o.y; wr[4 * c + 2] = o.z; wr[4 * c + 3] = o.w;
        }
        if (!warp_wait(smem_u32(&ctl->empty_a[s]), ph, abort_flag, lane)) return;
        tc_fence_after_sync();          // the MMAs that read these columns come first
        tmem_st32(tdst0 + s * A_COLS, wr);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {
            if (rank == 0) mbar_arrive(full0 + 8u * s);
            else mbar_arrive_cluster(full0 + 8u * s);
            // after the stores that consumed the loaded words: a load that has merely been issued does not hold back the
            // TMA write that refills the staging slot
            mbar_arrive(smem_u32(&ctl->group_empty[gslot]));
        }
        if (++gslot == GROUPS) { gslot = 0; gph ^= 1u; }
        if ((s += TEAMS) >= A_STAGES) { s = team; ph ^= 1u; }
    }
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(THREADS, 1)
xnor_pair_kernel(const __grid_constant__ Maps maps, const __grid_constant__ Args g) {
    const int M = g.M, N = g.N, L = g.n_layers;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Control* ctl = reinterpret_cast<Control*>(smem + SLOTS * B_BYTES + GROUPS * GROUP_BYTES);
    volatile int* abort_flag = &ctl->wait.abort;

    // The kernel that follows in the stream may be scheduled as soon as this one's CTAs leave their SMs.
    pdl_trigger();

    const int warp = warp_index(), lane = threadIdx.x & 31, rank = (int)cluster_rank();
    const int nks = ceil_div(g.K, BK), nkp = (nks + 1) & ~1;      // stages of a tile; with the empty partner of an odd last one
    const int m128 = ceil_div(M, BM), n_tiles = ceil_div(N, BN);
    const Share share(ceil_div(M, 2 * BM), n_tiles);
    const int n0 = share.nt * BN;

    if (threadIdx.x == 0) {
        for (int s = 0; s < A_STAGES; ++s) {
            mbar_init(smem_u32(&ctl->full_a[s]), 2 * A_WARPS);        // rank 0: the widening warps of both CTAs
            mbar_init(smem_u32(&ctl->empty_a[s]), PARTS);             // a commit of each issuing warp
        }
        for (int s = 0; s < SLOTS; ++s) {
            mbar_init(smem_u32(&ctl->full_b[s]), 1);                  // rank 0: its copying thread (+ bytes of both CTAs)
            mbar_init(smem_u32(&ctl->b_free[s]), PARTS);
        }
        for (int b = 0; b < PARTS; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), 2 * EPI_WARPS);   // rank 0: the epilogue warps of both CTAs
        }
        for (int b = 0; b < GROUPS; ++b) {
            mbar_init(smem_u32(&ctl->group_full[b]), 1);              // the issuing thread (+ bytes)
            mbar_init(smem_u32(&ctl->group_empty[b]), TEAMS * A_WARPS);
        }
        wait_state_init(&ctl->wait, g.status);
        mbar_init_fence();
    }
    __syncwarp();
    if (warp == MMA_WARP) tmem_alloc_pair(smem_u32(&ctl->tmem_base), TMEM_COLS);
    tc_fence_before_sync();
    cluster_sync();           // barriers of both CTAs initialised, tensor memory of both allocated
    tc_fence_after_sync();
    const uint32_t tmem = ctl->tmem_base;
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
        // ---------------- the layers follow one another in the producers' sequence of (tile, stage) pairs
        const uint32_t staging = smem_u32(smem) + SLOTS * B_BYTES;
        const int row = (warp & 3) * 32 + lane, team = (warp - PROD_WARP0) / A_WARPS, total = L * share.count * nkp;
        if (g.zo) produce<true>(staging, tmem, ctl, abort_flag, total, rank, row, team, lane);
        else produce<false>(staging, tmem, ctl, abort_flag, total, rank, row, team, lane);
    } else if (warp == WEIGHT_WARP) {
        // ---------------- one thread: the weight stages of all layers.  They do not depend on the kernel before this one nor on other
        // pairs; a slot is overwritten once the MMAs of this pair's last frame tile that read it have completed.
        if (lane == 0 && share.count > 0) {
            int slot = 0;
            uint32_t ph = 1;      // parity to wait for on `b_free`: a fresh barrier passes parity 1
            bool ok = true;
            for (int l = 0; l < L && ok; ++l)
                for (int ks = 0; ks < nks; ++ks) {
                    ok = mbar_wait(smem_u32(&ctl->b_free[slot]), ph, abort_flag);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&ctl->full_b[slot]), bar0 = peer_addr(bar, 0), dst = smem_u32(smem) + slot * B_BYTES;
                    if (rank == 0) mbar_arrive_expect_tx(bar, 2 * B_BYTES);
                    const int unit = n0 + rank * (PN / 2);
                    tma_load_2d_pair(dst, &maps.weights[l], unit * 2, ks * 8, bar0);
                    tma_load_2d_pair(dst + PART_BYTES, &maps.weights[l], (unit + PN) * 2, ks * 8, bar0);
                    if (++slot == SLOTS) { slot = 0; ph ^= 1u; }
                }
        }
        __syncwarp();
    } else if (warp == TMA_WARP) {
        // ---------------- one thread: the staging ring of frame rows
        if (lane == 0 && share.count > 0) {
            const uint32_t stg = smem_u32(smem) + SLOTS * B_BYTES;
            int slot = 0;
            uint32_t ph = 1;
            bool ok = true;
            for (int l = 0; l < L && ok; ++l)
                for (int t = 0; t < share.count && ok; ++t) {
                    const int mt = 2 * (share.first + t * share.step) + rank;          // in tiles of 128
                    if (l > 0 && mt < m128) {
                        // the frame tile's bits of the layer before: every unit tile's CTA has stored them
                        ok = wait_counter(g.progress + (size_t)(l - 1) * m128 + mt, n_tiles * EPI_WARPS, abort_flag);
                        if (!ok) break;
                        asm volatile("fence.proxy.async;" ::: "memory");   // generic-proxy writes of other CTAs -> this thread's TMA reads
                    }
                    for (int gi = 0; gi < nkp / 2; ++gi) {
                        ok = mbar_wait_relaxed(smem_u32(&ctl->group_empty[slot]), ph, abort_flag);
                        if (!ok) break;
                        const uint32_t bar = smem_u32(&ctl->group_full[slot]);
                        mbar_arrive_expect_tx(bar, GROUP_BYTES);
                        tma_load_2d(stg + slot * GROUP_BYTES, &maps.in[l], gi * 16, mt * BM, bar);
                        if (++slot == GROUPS) { slot = 0; ph ^= 1u; }
                    }
                }
        }
        __syncwarp();
    } else if (warp >= EPI_WARPS) {
        // ---------------- MMA issue: two converged warps of rank 0, each with its part of every tile
        const int part = warp - MMA_WARP;
        constexpr uint32_t idesc = instr_desc_mxf4(2 * BM, PN);
        const uint32_t sfa = tmem + TMEM_SF_COL, sfb = tmem + TMEM_SF_COL + SF_COLS / 2;
        const uint64_t desc = smem_desc_kmajor(smem_u32(smem) + part * PART_BYTES, PN / 2 * 16, 128);
        const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
        constexpr uint32_t kStepJ = (2 * (PN / 2) * 16) >> 4, kStepS = B_BYTES >> 4;
        const uint32_t d = tmem + (uint32_t)(part * PN);
        int s = 0;                        // slot of the A ring
        uint32_t pa = 0, pacc = 1;
        int slot0 = 0;                    // slot of the layer's first weight stage; its stages follow round the ring
        uint32_t pb0 = 0;                 // parity of `full` there
        bool ok = rank == 0;
        for (int l = 0; l < L && ok; ++l) {
            // A layer's weight stages arrive once and then stay; the last tile hands back a slot that is to be refilled.
            const int later = (L - 1 - l) * nks;
            for (int t = 0; t < share.count && ok; ++t) {
                const bool first = t == 0, last = t == share.count - 1;
                ok = warp_wait(smem_u32(&ctl->acc_empty[part]), pacc, abort_flag, lane);
                if (!ok) break;
                pacc ^= 1u;
                tc_fence_after_sync();
                for (int ks = 0; ks < nkp; ++ks) {
                    int slot = slot0 + ks;
                    const uint32_t wrapped = slot >= SLOTS ? 1u : 0u;
                    if (wrapped) slot -= SLOTS;
                    ok = (!first || ks >= nks || warp_wait(smem_u32(&ctl->full_b[slot]), pb0 ^ wrapped, abort_flag, lane)) &&
                         warp_wait(smem_u32(&ctl->full_a[s]), pa, abort_flag, lane);
                    if (!ok) break;
                    tc_fence_after_sync();
                    // the address field (16-byte units) is advanced by plain additions: the ring lies below 2^14 * 16 bytes.  An
                    // MMA takes 64 positions of K = 32 bytes: 8 columns of A, two 16-byte chunks of B
                    const uint32_t db = desc_lo + (uint32_t)slot * kStepS;
                    const uint32_t ta = tmem + TMEM_A_COL + s * A_COLS;
                    if (elect_one()) {
                        if (ks < nks) {           // (not the empty partner of an odd last stage)
                            mma_mxf4_ts_pair(d, ta, db, desc_hi, idesc, sfa, sfb, ks != 0);
                            mma_mxf4_ts_pair(d, ta + 8, db + kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                            mma_mxf4_ts_pair(d, ta + 16, db + 2 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                            mma_mxf4_ts_pair(d, ta + 24, db + 3 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                        }
                        mma_commit_pair(smem_u32(&ctl->empty_a[s]));
                        if (last && ks < nks && later + nks - ks > SLOTS) mma_commit_pair(smem_u32(&ctl->b_free[slot]));
                    }
                    if (++s == A_STAGES) { s = 0; pa ^= 1u; }
                }
                if (ok && elect_one()) mma_commit_pair(smem_u32(&ctl->acc_full[part]));
            }
            slot0 += nks;
            if (slot0 >= SLOTS) { slot0 -= SLOTS; pb0 ^= 1u; }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: thread = one frame (TMEM lane)
        const int half = warp >> 2, quarter = warp & 3, nw = words_for(N);
        uint32_t par = 0;
        bool ok = true;
        for (int l = 0; l < L && ok; ++l) {
            const int32_t* __restrict__ thr = g.layer[l].thr;
            const uint32_t* __restrict__ flip = g.layer[l].flip;
            uint32_t* __restrict__ out_bits = g.layer[l].out_bits;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < PARTS * PN / 64; ++i) {
                const int n = n0 + (i >> 1) * PN + half * (PN / 2) + (i & 1) * 32 + lane;
                // half-way between two sums: exact for every threshold a sum can meet, and no difference is a zero
                // (whose sign would depend on that of a sum of zeros)
                ctl->T[warp][i >> 1][(i & 1) * 32 + lane] = n < N ? (float)thr[n] - 0.5f : 0.0f;
            }
            __syncwarp();
            for (int t = 0; t < share.count && ok; ++t, par ^= 1u) {
                const int mt = 2 * (share.first + t * share.step) + rank, m = mt * BM + quarter * 32 + lane;
#pragma unroll 1
                for (int part = 0; part < PARTS; ++part) {
                    ok = warp_wait_relaxed(smem_u32(&ctl->acc_full[part]), par, abort_flag, lane);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t taddr = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(part * PN + half * (PN / 2));
                    const float* T = ctl->T[warp][part];
                    const int w0 = (n0 + part * PN + half * (PN / 2)) >> 5;
                    uint32_t acc[16], words[2] = {0u, 0u};
                    tmem_ld16(taddr, acc);
#pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        tmem_ld_wait();
                        // The accumulator holds the integer dot product as a float: the
                        // sign of its difference from T is the decision.  The sign bits are shifted in from the top, the last
                        // element first, so element j ends up in bit j, inverted; two chains of eight, joined at the end
                        uint32_t chain[2] = {0u, 0u};
#pragma unroll
                        for (int j = 7; j >= 0; --j)
#pragma unroll
                            for (int c = 0; c < 2; ++c)
                                chain[c] = __funnelshift_l(__float_as_uint(__uint_as_float(acc[8 * c + j]) - T[h * 16 + 8 * c + j]), chain[c], 1);
                        if (h < 3) {
                            tmem_ld16(taddr + 16 * (h + 1), acc);
                        } else {
                            // the accumulator is read: the part's next tile may start on it
                            tc_fence_before_sync();
                            __syncwarp();
                            if (lane == 0) mbar_arrive_cluster(peer_addr(smem_u32(&ctl->acc_empty[part]), 0));
                        }
                        words[h >> 1] |= (chain[0] | (chain[1] << 8)) << (16 * (h & 1));
                    }
#pragma unroll
                    for (int gq = 0; gq < 2; ++gq) {
                        const int wi = w0 + gq, valid = N - wi * 32;          // columns of this word that exist
                        words[gq] = wi < nw ? (~words[gq] ^ __ldg(flip + wi)) & (valid < 32 ? (1u << valid) - 1u : 0xFFFFFFFFu) : 0u;
                    }
                    if (m < M) {
                        uint32_t* dst = out_bits + (size_t)m * g.ldob + w0;
                        if (w0 + 1 < nw) *reinterpret_cast<uint2*>(dst) = make_uint2(words[0], words[1]);     // rows are 16-byte aligned, w0 is even
                        else if (w0 < nw) dst[0] = words[0];
                    }
                }
                if (ok && l + 1 < L && mt < m128) {
                    // this warp's share of the frame tile is stored: tell the CTAs that read it in the next layer (the fence covers what the
                    // lanes stored before the warp barrier)
                    __syncwarp();
                    if (lane == 0) {
                        __threadfence();
                        asm volatile("fence.proxy.async;" ::: "memory");
                        asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(g.progress + (size_t)l * m128 + mt) : "memory");
                    }
                    __syncwarp();
                }
            }
        }
    }

    // ---------------- teardown: every thread of both CTAs arrives here, also after an aborted wait
    __syncwarp();
    tc_fence_before_sync();
    cluster_sync();           // nobody reads the partner's shared or tensor memory any more
    if (warp == MMA_WARP) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && ctl->wait.abort) atomicExch(g.status.word, 1);
}

}  // namespace

long long xnor_pair_clocks(int M, int N, int K, int sm_count) {
    const int nks = ceil_div(K, BK), n_tiles = ceil_div(N, BN), pairs = sm_count / 2;
    if (nks > SLOTS || n_tiles > pairs) return 0;
    // what of the next layer's weights does not fit beside this one's arrives behind the last tile's MMAs
    const int reload = 2 * nks > SLOTS ? (2 * nks - SLOTS) * 540 : 0;
    return (long long)ceil_div(ceil_div(M, 2 * BM), pairs / n_tiles) * nks * 660 + reload;      // clocks of a stage as measured
}

int launch_xnor_pair(const uint32_t* Ap, int ldap, const XnorStackLayer* layers, int n_layers, int M, int N, int K, int ldob,
                     int zo, int* progress, cudaStream_t st) {
    const int sms = device_sm_count();
    if (sms < 2 || !ensure_dynamic_smem(reinterpret_cast<const void*>(xnor_pair_kernel), SMEM_BYTES)) return BNN_ERR_CUDA;
    const long long tiles = (long long)ceil_div(M, 2 * BM) * ceil_div(N, BN);
    const int grid = 2 * (int)(tiles < sms / 2 ? tiles : sms / 2);
    Args a{};
    Maps maps{};
    a.n_layers = n_layers; a.M = M; a.N = N; a.K = K; a.ldob = ldob; a.zo = zo;
    a.status = tc_status();
    a.progress = progress;
    if (!a.status.word) return BNN_ERR_CUDA;
    for (int l = 0; l < n_layers; ++l) {
        a.layer[l] = Layer{layers[l].thr, layers[l].flip, layers[l].out_bits};
        // a layer reads what the layer before it wrote
        const uint32_t* in = l == 0 ? Ap : layers[l - 1].out_bits;
        if (!encode_packed_map(&maps.in[l], in, l == 0 ? ldap : ldob, M, K, BM)) return BNN_ERR_CUDA;
        if (!encode_digit_map(&maps.weights[l], layers[l].image, xnor_image_npad(N), 8 * ceil_div(K, BK), PN / 2, 8)) return BNN_ERR_CUDA;
    }
    // The CTAs of a run wait for one another: see launch_bn in xnor_gemm_res.cu.
    if (n_layers > 1) {
        if (launch_cooperative(xnor_pair_kernel, dim3(grid), dim3(THREADS), SMEM_BYTES, st, maps, a) != cudaSuccess) return BNN_ERR_CUDA;
    } else {
        xnor_pair_kernel<<<grid, THREADS, SMEM_BYTES, st>>>(maps, a);
    }
    return launch_status();
}

}  // namespace bnn
