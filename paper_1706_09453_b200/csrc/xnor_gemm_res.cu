// Fused binary hidden layer on the tensor cores with the layer's weights RESIDENT in shared
// memory:  bits[m][n] = Sign(scale[n] * sum_k a[m][k] * w[n][k] + shift[n]),  a, w in {-1, +1}.
//
// Same contraction as xnor_gemm_tc.cu / xnor_gemm_img.cu (every +-1 widened to a 4-bit e2m1
// nibble, kind::mxf4, unit block scales, exact fp32 sums).  Measured on B200, streaming the
// widened weights from L2 for every tile of frames holds the tensor pipe at about a third of
// its rate (24 KB per 384 MMA clocks and SM is more than L2 delivers to 148 SMs at once).  So
// here a CTA owns ONE tile of units for the whole launch: it loads that tile's slice of the
// prepared weight image (all of K, up to 192 KB) into shared memory once and then walks over
// frame tiles, for which only the packed frame bits (4 KB per stage) cross L2.  CTA c works on
// unit tile c mod n_tiles and shares that tile's frame tiles with the other CTAs of the same
// residue.
//
// The image is the one xnor_gemm_img.cu describes: a tile of BN units is, per stage of 256
// positions of K, eight contiguous runs of BN x 16 bytes, copied to offsets c * BN * 16 of the
// stage's block (K-major core matrices).  BN is 192 while K <= 2048 and 128 while K <= 3072 for batches that fill the
// SMs, which keeps the slice within 192 KB; 96 or 32 for smaller ones, where more unit tiles occupy more SMs and the
// region holds the next layer's slice beside this one's (tile_units).  Other shapes are left to the streaming kernel.
//
// Roles in a CTA of 16 warps (one CTA per SM):
//   warp 15      one thread issues the bulk copies of the weight slices, layer after layer
//   warp 13      one thread issues the 2-D TMA tile loads of the packed frame rows (64 bytes per row = two stages)
//                into a staging ring (64-byte swizzle, no multicast)
//   warps 5-12   two teams of four warps widen the frame rows, thread = one row, 32 bytes ->
//                128 bytes per stage, into tensor memory (the MMA reads its A operand from
//                there); the teams take alternate stages
//   warps 4, 14  issue the MMAs (4 per stage, K = 64 each) and the commits; the two warps take a tile's stages in
//                turn and accumulate into the same accumulator
//   warps 0-3    epilogue: accumulator -> threshold -> repacked bits; two accumulators in
//                tensor memory, so it overlaps the next tile's MMAs
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles fall
// through to the common teardown and the device status word is set.
//
// A run of consecutive hidden layers of the same shape (the forward loop of Algorithm 2 over
// l = 2 .. L-1) is ONE launch: the roles above loop over the layers.  Between layers nothing is
// torn down; a CTA keeps its unit tile index and its frame tiles.  What a layer needs from the
// one before it is tracked per frame tile: a counter in global memory that every epilogue warp increments
// (after a fence) once its bits of that frame tile and layer are stored, and the thread that loads a frame
// tile waits (acquire, bounded) until the warps of all unit tiles have arrived.  The weight stages of the layers
// follow one another round a ring of as many as fit, each slot refilled as soon as the last frame tile's MMAs that read it
// have completed.  (Measured on B200: five launches of one layer each spent 6 us per layer between the end of one
// kernel and the first MMA of the next.)
//
// What bounds it, measured on B200: 65536 frames x 3072 the widening of the frame rows (2 teams, about 430 clocks per
// stage against 256 of MMA; five layers 1.18 ms: such runs go to pairs of CTAs, xnor_gemm_pair.cu); 8192 x 2048 MMA (384 clocks per stage of 192 units), epilogue and the fill of a layer's pipeline in like parts
// (five layers 76 us, 91 before); a layer of one frame tile per CTA the chain store - count - load - widen -
// MMA - decide, about 7 us (731 frames 36 us, 50 before, when all tiles were 192 wide).
#include <type_traits>

#include "bnn_common.cuh"
#include "tcgen05.cuh"
#include "xnor_widen.cuh"

namespace bnn {

namespace {

using namespace tc;

constexpr int BM = 128;
constexpr int BK = 256;                                   // positions of K per stage
constexpr int ROW_BYTES = BK / 2;                         // widened bytes per row and stage (128)
constexpr int B_REGION = 192 * 1024;                      // shared memory that holds the weight slice
constexpr int EPI_WARPS = 4, MMA_WARP = 4, PROD_WARP0 = 5, A_WARPS = BM / 32, TEAMS = 2;
constexpr int TMA_WARP = PROD_WARP0 + TEAMS * A_WARPS;
constexpr int MMA_WARP2 = TMA_WARP + 1;                   // the second issuing warp
constexpr int WEIGHT_WARP = MMA_WARP2 + 1;                // loads the weight stages
constexpr int THREADS = (WEIGHT_WARP + 1) * 32;           // 512
constexpr int GROUPS = 4;                                 // staging ring of the packed frame rows: groups of two stages
constexpr int GROUP_BYTES = BM * 64;
constexpr uint32_t A_COLS = ROW_BYTES / 4;                // 32-bit columns per A stage
constexpr uint32_t SF_COLS = 32, TMEM_COLS = 512;
constexpr int MAX_SLOTS = 48, MAX_A_BARS = 6;

template <int BN> struct Cfg {
    static constexpr int B_BYTES = BN * ROW_BYTES;                 // one stage of the unit operand
    static constexpr int SLOTS = B_REGION / B_BYTES;               // weight stages that fit: 8 (BN 192), 12 (128), 16 (96), 48 (32)
    static constexpr int A_STAGES = (int)((TMEM_COLS - SF_COLS - 2 * BN) / A_COLS) > 6 ? 6 : (int)((TMEM_COLS - SF_COLS - 2 * BN) / A_COLS);
    // A stage `it` of the CTA's sequence has barrier it % A_BARS, an even number, so that a barrier always belongs to the
    // same team and issuing warp.  (A wait on a parity holds only for one who has seen every phase before it: with
    // three barriers the warps would take turns on each, and the one ahead could take the phase before for its own.)
    static constexpr int A_BARS = A_STAGES % 2 ? 2 * A_STAGES : A_STAGES;
    static constexpr uint32_t TMEM_A_COL = 2 * BN;                 // A stages start after the two accumulators
    static constexpr uint32_t TMEM_SF_COL = TMEM_A_COL + A_STAGES * A_COLS;
    static_assert(SLOTS <= MAX_SLOTS && A_STAGES >= 3 && A_BARS <= MAX_A_BARS && TMEM_SF_COL + SF_COLS <= TMEM_COLS, "tile configuration");
};

constexpr int MAX_STACK = kXnorStackMax;

struct Control {
    float T[192];            // per unit: threshold less 1/2
    uint32_t flipw[8];
    uint64_t full_a[MAX_A_BARS], empty_a[MAX_A_BARS], full_b[MAX_SLOTS], b_free[MAX_SLOTS], acc_full[2], acc_empty[2];
    uint64_t group_full[GROUPS], group_empty[GROUPS];
    uint64_t started[2];
    uint32_t tmem_base;
    WaitState wait;
};
constexpr int SMEM_BYTES = B_REGION + GROUPS * GROUP_BYTES + (int)sizeof(Control) + 1024;
static_assert(SMEM_BYTES <= 232448, "shared memory of one CTA");

// 1-D bulk asynchronous copy global -> shared; completion is counted in bytes on `bar`.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Frame tiles of this CTA: mt = first, first + step, ... < m_tiles.
struct Share {
    int first, step, count;
};
__device__ __forceinline__ Share my_share(int m_tiles, int n_tiles) {
    const int nt = (int)blockIdx.x % n_tiles, r = (int)blockIdx.x / n_tiles;
    const int peers = ((int)gridDim.x - 1 - nt) / n_tiles + 1;    // CTAs that work on unit tile nt
    Share s;
    s.first = r; s.step = peers;
    s.count = r < m_tiles ? (m_tiles - 1 - r) / peers + 1 : 0;
    return s;
}

struct ProducerArgs {
    uint32_t smem_stage;  // shared-space address of the staging ring
    uint32_t tmem_a;      // tensor-memory address of A stage 0 (lane 0)
    Control* ctl;
    volatile int* abort_flag;
    int my_tiles, nks, kw;
    uint32_t tmask;
    int lane;
};

// Producer of the frame operand: thread = row `r` of every tile of this CTA; team `team`
// takes the stages it = team, team + TEAMS, ... of the CTA's sequence of (tile, stage) pairs.
// Template arguments say what the loop has to deal with: code that is there for another case costs this one, though it is
// not executed, where this role is the bottleneck (five 3072-wide layers of 65536 frames 1.50 ms with the case of an
// odd number of stages behind a branch, 1.24 ms without it).
// ODD: a row has an odd number of stages; ZO: bits stand for (0,1); RAGGED: the last stage has positions >= K.
template <int A_STAGES, int A_BARS, bool ODD, bool ZO, bool RAGGED>
__device__ __forceinline__ void produce_a(const ProducerArgs& a, int r, int team) {
    Control* ctl = a.ctl;
    const int total = a.my_tiles * a.nks;
    const int ng = ceil_div(a.nks, 2);
    // TMEM lane of this thread's frame row: a warp may only touch lanes 32*(warp%4)..+31
    const uint32_t tdst0 = a.tmem_a + ((uint32_t)(r & ~31) << 16);
    // this row inside a staging group: 64 bytes per row, 16-byte chunk c stored at c ^ ((r/2)%4)
    const uint32_t stg0 = a.smem_stage + r * 64;
    const uint32_t sw = (uint32_t)(r >> 1) & 3u;
    // A group that holds a single stage, of the other team: every team sees every phase of a group's barriers.
    auto visit = [&](int gidx) {
        const int gslot = gidx % GROUPS;
        if (!warp_wait(smem_u32(&ctl->group_full[gslot]), (uint32_t)((gidx / GROUPS) & 1), a.abort_flag, a.lane)) return false;
        if (a.lane == 0) mbar_arrive(smem_u32(&ctl->group_empty[gslot]));
        return true;
    };
    if (ODD && a.nks == 1 && team == 1 && total > 0 && !visit(0)) return;
    int ks = team, tl = 0;
    while (ks >= a.nks) { ks -= a.nks; ++tl; }
    for (int it = team; it < total; it += TEAMS) {
        const int gidx = tl * ng + (ks >> 1);          // staging group that holds this stage
        const int gslot = gidx % GROUPS;
        const uint32_t gi = (uint32_t)ks & 1u;         // stage inside its group of two
        if (!warp_wait(smem_u32(&ctl->group_full[gslot]), (uint32_t)((gidx / GROUPS) & 1), a.abort_flag, a.lane)) break;
        const uint32_t src = stg0 + gslot * GROUP_BYTES;
        const uint4 v0 = lds128u(src + (((2u * gi) ^ sw) << 4));
        const uint4 v1 = lds128u(src + (((2u * gi + 1u) ^ sw) << 4));
        const int s = it % A_STAGES;
        const int e = it + A_BARS - A_STAGES;          // the stage that had this slot; a fresh barrier passes parity 1
        if (!warp_wait(smem_u32(&ctl->empty_a[e % A_BARS]), (uint32_t)(((e / A_BARS) & 1) ^ 1), a.abort_flag, a.lane)) break;
        const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
        // 32-bit column 4c + t of the stage = word t of chunk c: the byte order of the
        // K-major shared-memory layout of the other operand
        uint32_t wr[32];
        if (ZO) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int g = 8 * ks + c;   // index of the word in the row
                const uint32_t valid = (!RAGGED || g < a.kw - 1) ? 0xFFFFFFFFu : (g == a.kw - 1 ? a.tmask : 0u);
                const uint4 o = widen01_masked(w[c], valid);
                wr[4 * c] = o.x; wr[4 * c + 1] = o.y; wr[4 * c + 2] = o.z; wr[4 * c + 3] = o.w;
            }
        } else if (RAGGED && ks == a.nks - 1) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int g = 8 * ks + c;   // index of the word in the row
                const uint32_t valid = g < a.kw - 1 ? 0xFFFFFFFFu : (g == a.kw - 1 ? a.tmask : 0u);
                const uint4 o = widen_masked(w[c], valid);
                wr[4 * c] = o.x; wr[4 * c + 1] = o.y; wr[4 * c + 2] = o.z; wr[4 * c + 3] = o.w;
            }
        } else {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 o = widen(w[c]);
                wr[4 * c] = o.x; wr[4 * c + 1] = o.y; wr[4 * c + 2] = o.z; wr[4 * c + 3] = o.w;
            }
        }
        tc_fence_after_sync();          // the MMAs that read these columns come first
        tmem_st32(tdst0 + s * A_COLS, wr);
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (a.lane == 0) {
            mbar_arrive(smem_u32(&ctl->full_a[it % A_BARS]));
            // The staging slot is handed back only after the stores that consumed the loaded
            // words: a shared-memory load that has merely been issued does not hold back the
            // TMA write that refills the slot.  A group counts one arrival per warp of both teams.
            mbar_arrive(smem_u32(&ctl->group_empty[gslot]));
        }
        if (ODD && it + 1 < total && (a.nks == 1 || ks + 2 == a.nks)) {
            if (!visit(gidx + 1)) break;
        }
        ks += TEAMS;
        while (ks >= a.nks) { ks -= a.nks; ++tl; }
    }
}

// One layer of the run: its prepared weight image, folded thresholds and output.
struct StackLayer {
    const uint8_t* img;
    const int32_t* thr;
    const uint32_t* flip;
    uint32_t* out_bits;
};
struct StackArgs {
    StackLayer layer[MAX_STACK];
    int n_layers;
    int M, N, K, ldob, zo;
    TcStatus status;
    int* progress;           // [n_layers - 1][frame tiles] arrival counters, zero at launch (unused for one layer)
};
struct StackMaps {
    CUtensorMap m[MAX_STACK];   // packed input of each layer
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

template <int BN>
__global__ void __launch_bounds__(THREADS, 1)
xnor_res_kernel(const __grid_constant__ StackMaps maps, const __grid_constant__ StackArgs g) {
    using C = Cfg<BN>;
    const int M = g.M, N = g.N, K = g.K, ldob = g.ldob, zo = g.zo, L = g.n_layers;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    Control* ctl = reinterpret_cast<Control*>(smem + B_REGION + GROUPS * GROUP_BYTES);
    volatile int* abort_flag = &ctl->wait.abort;

    // The kernel that follows in the stream may be scheduled as soon as this one's CTAs leave their SMs.
    pdl_trigger();

    const int warp = warp_index(), lane = threadIdx.x & 31;
    const int kw = words_for(K);
    const int nks = ceil_div(K, BK);
    const int m_tiles = ceil_div(M, BM), n_tiles = ceil_div(N, BN);
    const Share share = my_share(m_tiles, n_tiles);
    const int nt = (int)blockIdx.x % n_tiles, n0 = nt * BN;

    if (threadIdx.x == 0) {
        for (int s = 0; s < C::A_BARS; ++s) {
            mbar_init(smem_u32(&ctl->full_a[s]), A_WARPS);
            mbar_init(smem_u32(&ctl->empty_a[s]), 1);
        }
        for (int s = 0; s < C::SLOTS; ++s) {
            mbar_init(smem_u32(&ctl->full_b[s]), 1);   // the copying thread (+ bytes)
            mbar_init(smem_u32(&ctl->b_free[s]), 2);   // one commit of each issuing warp
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(smem_u32(&ctl->acc_full[b]), 2);       // one commit of each issuing warp
            mbar_init(smem_u32(&ctl->started[b]), 1);
            mbar_init(smem_u32(&ctl->acc_empty[b]), EPI_WARPS);
        }
        for (int b = 0; b < GROUPS; ++b) {
            mbar_init(smem_u32(&ctl->group_full[b]), 1);              // the issuing thread (+ bytes)
            mbar_init(smem_u32(&ctl->group_empty[b]), 2 * A_WARPS);   // every warp of both teams
        }
        wait_state_init(&ctl->wait, g.status);
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
    if (warp < EPI_WARPS) {
        // Block scales of both operands: every byte 127, the ue8m0 code of 2^0.  The whole
        // region is filled, so the values do not depend on how the scales are laid out in it.
        uint32_t ones[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) ones[j] = 0x7F7F7F7Fu;
        tmem_st32(tmem + ((uint32_t)(warp * 32) << 16) + C::TMEM_SF_COL, ones);
        tmem_st_wait();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();

    if (warp == WEIGHT_WARP) {
        // ---------------- one thread: the weight stages of all layers, in a ring of as many stages as fit.  The weights
        // do not depend on the kernel before this one in the stream nor on other CTAs, so with narrow tiles the next
        // layer's arrive while this one runs; a slot is overwritten once the MMAs of this CTA's last frame
        // tile that read it have completed.
        if (lane == 0 && share.count > 0) {
            const size_t run = (size_t)xnor_image_npad(N) * 16;   // bytes between chunks of the image
            int slot = 0;
            uint32_t ph = 1;      // parity to wait for on `b_free`: a fresh barrier passes parity 1
            bool ok = true;
            for (int l = 0; l < L && ok; ++l) {
                const uint8_t* src = g.layer[l].img + (size_t)n0 * 16;
                for (int ks = 0; ks < nks; ++ks) {
                    ok = mbar_wait(smem_u32(&ctl->b_free[slot]), ph, abort_flag);
                    if (!ok) break;
                    const uint32_t bar = smem_u32(&ctl->full_b[slot]);
                    mbar_arrive_expect_tx(bar, C::B_BYTES);
#pragma unroll
                    for (int c = 0; c < 8; ++c)
                        bulk_g2s(smem_u32(smem + slot * C::B_BYTES + c * (BN * 16)), src + (size_t)(ks * 8 + c) * run, BN * 16, bar);
                    if (++slot == C::SLOTS) { slot = 0; ph ^= 1u; }
                }
            }
        }
        __syncwarp();
    } else if (warp == TMA_WARP) {
        // ---------------- one thread: the staging ring of frame rows
        if (lane == 0 && share.count > 0) {
            const uint32_t stg = smem_u32(smem) + B_REGION;
            const int ng = ceil_div(nks, 2);
            int gc = 0;   // groups issued so far, over all layers: slot gc % GROUPS, < GROUPS ahead of its consumers
            bool ok = true;
            for (int l = 0; l < L && ok; ++l)
                for (int t = 0; t < share.count && ok; ++t) {
                    const int mt = share.first + t * share.step;
                    if (l > 0) {
                        // the frame tile's bits of the layer before: every unit tile's CTA has stored them
                        ok = wait_counter(g.progress + (size_t)(l - 1) * m_tiles + mt, n_tiles * EPI_WARPS, abort_flag);
                        if (!ok) break;
                        asm volatile("fence.proxy.async;" ::: "memory");   // generic-proxy writes of other CTAs -> this thread's TMA reads
                    }
                    for (int gi = 0; gi < ng; ++gi, ++gc) {
                        const int slot = gc % GROUPS;
                        if (gc >= GROUPS) {
                            ok = mbar_wait_relaxed(smem_u32(&ctl->group_empty[slot]), (uint32_t)(((gc / GROUPS) - 1) & 1), abort_flag);
                            if (!ok) break;
                        }
                        const uint32_t bar = smem_u32(&ctl->group_full[slot]);
                        mbar_arrive_expect_tx(bar, GROUP_BYTES);
                        tma_load_2d(stg + slot * GROUP_BYTES, &maps.m[l], gi * 16, mt * BM, bar);
                    }
                }
        }
        __syncwarp();
    } else if (warp >= PROD_WARP0 && warp < TMA_WARP) {
        // the layers follow one another in the producers' sequence of (tile, stage) pairs
        ProducerArgs pa{smem_u32(smem) + B_REGION, tmem + C::TMEM_A_COL, ctl, abort_flag, L * share.count, nks, kw, tail_mask(K), lane};
        const int row = (warp & 3) * 32 + lane, team = (warp - PROD_WARP0) / A_WARPS;
        const bool ragged = (kw % 8 != 0) || pa.tmask != 0xFFFFFFFFu;   // last stage has positions >= K
        auto go = [&](auto odd, auto zero_one) {
            constexpr bool ODD = decltype(odd)::value, ZO = decltype(zero_one)::value;
            if (ragged) produce_a<C::A_STAGES, C::A_BARS, ODD, ZO, true>(pa, row, team);
            else produce_a<C::A_STAGES, C::A_BARS, ODD, ZO, false>(pa, row, team);
        };
        using T = std::true_type;
        using F = std::false_type;
        if (nks & 1) zo ? go(T{}, T{}) : go(T{}, F{});
        else zo ? go(F{}, T{}) : go(F{}, F{});
    } else if (warp == MMA_WARP || warp == MMA_WARP2) {
        // ---------------- MMA issue: two converged warps.  A tile's stages go to the two warps in turn, and both
        // accumulate into the tile's accumulator: the sums are exact integers (|sum| <= K < 2^24), so the
        // order of the accumulations does not matter.  Only the stage that overwrites the accumulator has
        // to come first: the warp that takes it commits it to `started`, and the other one waits for that
        // before its first MMA of the tile (the same one for every tile of an accumulator, whether nks is even or odd).  (Measured on B200: what an issuing warp does between MMAs
        // -- polls, commits, bookkeeping -- is time the tensor pipe idles unless the other warp fills it.  The four MMAs of
        // a stage go out together from one elected lane, see elect_one: five 3072-wide layers of 65536 frames 1.53 ->
        // 1.35 ms against MMAs predicated on lane 0.)
        {
            const int w = warp == MMA_WARP ? 0 : 1;
            constexpr uint32_t idesc = instr_desc_mxf4(BM, BN);
            const uint32_t sfa = tmem + C::TMEM_SF_COL, sfb = tmem + C::TMEM_SF_COL + SF_COLS / 2;
            const uint64_t desc = smem_desc_kmajor(smem_u32(smem), BN * 16, 128);
            const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
            constexpr uint32_t kStepJ = (2 * BN * 16) >> 4, kStepS = C::B_BYTES >> 4;
            const uint32_t tmem_a = tmem + C::TMEM_A_COL;
            bool ok = true;
            int tl = 0;          // tiles so far, over all layers
            int sa = w, ba = w;  // slot of the A ring and barrier of this warp's next stage, and that barrier's parity
            uint32_t pa = 0;
            int slot0 = 0;       // slot of the layer's first weight stage; its stages follow round the ring
            uint32_t pb0 = 0;    // parity of `full` there
            int turn = w;        // this warp's first stage of the tile: stages go to the two warps in turn, across tiles
            for (int l = 0; l < L && ok; ++l) {
                // A layer's weight stages arrive once and then stay; the last tile hands back a slot that is to be
                // refilled.  Both warps see every phase of these barriers, whoever takes the stage.
                const int later = (L - 1 - l) * nks;
                for (int t = 0; t < share.count && ok; ++t, ++tl) {
                    const bool first = t == 0, last = t == share.count - 1;
                    const int b = tl & 1;
                    ok = warp_wait(smem_u32(&ctl->acc_empty[b]), (uint32_t)(((tl >> 1) & 1) ^ 1), abort_flag, lane);
                    if (!ok) break;
                    tc_fence_after_sync();
                    const uint32_t d = tmem + (uint32_t)(b * BN);
                    for (int ks = first || last ? 0 : turn; ks < nks; ++ks) {
                        int slot = slot0 + ks;
                        const uint32_t wrapped = slot >= C::SLOTS ? 1u : 0u;
                        if (wrapped) slot -= C::SLOTS;
                        const bool hand_over = last && later + nks - ks > C::SLOTS;
                        if (first) {
                            ok = warp_wait(smem_u32(&ctl->full_b[slot]), pb0 ^ wrapped, abort_flag, lane);
                            if (!ok) break;
                        }
                        if ((ks & 1) != turn) {
                            if (hand_over && elect_one()) mma_commit(smem_u32(&ctl->b_free[slot]));
                            continue;
                        }
                        ok = warp_wait(smem_u32(&ctl->full_a[ba]), pa, abort_flag, lane) &&
                             (ks != 1 || warp_wait(smem_u32(&ctl->started[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane));
                        if (!ok) break;
                        tc_fence_after_sync();
                        // the address field (16-byte units) is advanced by plain additions: the whole region lies
                        // below 2^14 * 16 bytes.  An MMA takes 64 positions of K = 32 bytes: 8 columns of A, two
                        // 16-byte chunks of B
                        const uint32_t db = desc_lo + (uint32_t)slot * kStepS;
                        const uint32_t ta = tmem_a + sa * A_COLS;
                        if (elect_one()) {
                            mma_mxf4_ts(d, ta, db, desc_hi, idesc, sfa, sfb, ks != 0);
                            if (ks == 0) mma_commit(smem_u32(&ctl->started[b]));
                            mma_mxf4_ts(d, ta + 8, db + kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                            mma_mxf4_ts(d, ta + 16, db + 2 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                            mma_mxf4_ts(d, ta + 24, db + 3 * kStepJ, desc_hi, idesc, sfa, sfb, 1u);
                            mma_commit(smem_u32(&ctl->empty_a[ba]));
                            if (hand_over) mma_commit(smem_u32(&ctl->b_free[slot]));
                        }
                        if ((sa += 2) >= C::A_STAGES) sa -= C::A_STAGES;
                        if ((ba += 2) >= C::A_BARS) { ba -= C::A_BARS; pa ^= 1u; }
                        if (!(first || last)) ++ks;      // the next one is the other warp's
                    }
                    if (ok && elect_one()) mma_commit(smem_u32(&ctl->acc_full[b]));
                    turn ^= nks & 1;
                }
                slot0 += nks;
                if (slot0 >= C::SLOTS) { slot0 -= C::SLOTS; pb0 ^= 1u; }
            }
        }
        __syncwarp();
    } else {
        // ---------------- epilogue: 128 threads, thread = one frame (TMEM lane)
        const int row_in_tile = warp * 32 + lane;
        bool ok = true;
        int tl = 0;              // tiles so far, over all layers
        for (int l = 0; l < L && ok; ++l) {
            // thresholds of this CTA's units for this layer (the unit tile never changes); the
            // barriers keep them apart from the previous layer's last readers
            const int32_t* __restrict__ thr = g.layer[l].thr;
            const uint32_t* __restrict__ flip = g.layer[l].flip;
            uint32_t* __restrict__ out_bits = g.layer[l].out_bits;
            if (l > 0) epi_bar_sync();
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int nl = row_in_tile + h * 128, n = n0 + nl;
                // half-way between two sums: exact for every threshold a sum can meet, and no difference is a zero
                // (whose sign would depend on that of a sum of zeros)
                if (nl < BN) ctl->T[nl] = n < N ? (float)thr[n] - 0.5f : 0.0f;
            }
            if (row_in_tile < BN / 32) {
                const int wi = (n0 >> 5) + row_in_tile;
                ctl->flipw[row_in_tile] = wi < words_for(N) ? flip[wi] : 0u;
            }
            epi_bar_sync();
            for (int t = 0; t < share.count && ok; ++t, ++tl) {
                const int mt = share.first + t * share.step;
                const int m = mt * BM + row_in_tile;
                const int b = tl & 1;
                // all four epilogue warps take the same decision, so none is left at a barrier
                ok = epi_all(warp_wait_relaxed(smem_u32(&ctl->acc_full[b]), (uint32_t)((tl >> 1) & 1), abort_flag, lane));
                if (!ok) break;
                tc_fence_after_sync();
                const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(b * BN);
                const int nw = words_for(N), w0 = n0 >> 5;
                uint32_t* dst = out_bits + (size_t)(m < M ? m : 0) * ldob + w0;
                uint32_t acc[32], held = 0u;
                tmem_ld32(taddr, acc);
#pragma unroll
                for (int gq = 0; gq < BN / 32; ++gq) {
                    tmem_ld_wait();
                    // The accumulator holds the integer dot product as a float, T the threshold less 1/2: the
                    // sign of their difference is the decision.  The sign bits are shifted in from the top, the last
                    // element first, so element j ends up in bit j, inverted; four chains of eight, joined at the end
                    uint32_t part[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                    for (int j = 7; j >= 0; --j)
#pragma unroll
                        for (int c = 0; c < 4; ++c)
                            part[c] = __funnelshift_l(__float_as_uint(__uint_as_float(acc[8 * c + j]) - ctl->T[gq * 32 + 8 * c + j]), part[c], 1);
                    if (gq + 1 < BN / 32) {
                        tmem_ld32(taddr + (gq + 1) * 32, acc);
                    } else {
                        // the accumulator is read: the MMA warps may start the tile after the next on it
                        tc_fence_before_sync();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(smem_u32(&ctl->acc_empty[b]));
                    }
                    uint32_t wd = __byte_perm(__byte_perm(part[0], part[1], 0x0040), __byte_perm(part[2], part[3], 0x0040), 0x5410);
                    wd = ~wd ^ ctl->flipw[gq];
                    const int valid = N - (n0 + gq * 32);  // columns of this word that exist
                    if (valid < 32) wd = valid > 0 ? (wd & ((1u << valid) - 1u)) : 0u;
                    if (BN % 64 == 0) {      // rows are 16-byte aligned and BN / 32 is even: 8-byte stores
                        if (gq & 1) {
                            if (m < M) {
                                if (w0 + gq < nw) *reinterpret_cast<uint2*>(dst + gq - 1) = make_uint2(held, wd);
                                else if (w0 + gq - 1 < nw) dst[gq - 1] = held;
                            }
                        } else {
                            held = wd;
                        }
                    } else if (m < M && w0 + gq < nw) {
                        dst[gq] = wd;
                    }
                }
                if (l + 1 < L) {
                    // this warp's share of frame tile mt is stored: tell the CTAs that read it in the next layer.  The
                    // fence (about 1200 clocks) covers what the lanes stored before the warp barrier; no barrier
                    // over the four warps, and the count itself needs no second fence.
                    __syncwarp();
                    if (lane == 0) {
                        __threadfence();
                        asm volatile("fence.proxy.async;" ::: "memory");
                        asm volatile("red.relaxed.gpu.global.add.s32 [%0], 1;" ::"l"(g.progress + (size_t)l * m_tiles + mt) : "memory");
                    }
                    __syncwarp();
                }
            }
        }
    }

    // ---------------- teardown: every thread arrives here, also after an aborted wait
    tc_fence_before_sync();
    __syncthreads();
    if (warp == MMA_WARP) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && ctl->wait.abort) atomicExch(g.status.word, 1);
}

template <int BN>
int launch_bn(const uint32_t* Ap, int ldap, const XnorStackLayer* layers, int n_layers, int M, int N, int K, int ldob,
              int zo, int* progress, int sm_count, cudaStream_t st) {
    auto kern = xnor_res_kernel<BN>;
    if (!ensure_dynamic_smem(reinterpret_cast<const void*>(kern), SMEM_BYTES)) return BNN_ERR_CUDA;
    const long long tiles = (long long)ceil_div(M, BM) * ceil_div(N, BN);
    const int grid = tiles < sm_count ? (int)tiles : sm_count;
    StackArgs a{};
    StackMaps maps{};
    a.n_layers = n_layers; a.M = M; a.N = N; a.K = K; a.ldob = ldob; a.zo = zo;
    a.status = tc_status();
    a.progress = progress;
    if (!a.status.word) return BNN_ERR_CUDA;
    for (int l = 0; l < n_layers; ++l) {
        a.layer[l] = StackLayer{static_cast<const uint8_t*>(layers[l].image), layers[l].thr, layers[l].flip, layers[l].out_bits};
        // a layer reads what the layer before it wrote
        const uint32_t* in = l == 0 ? Ap : layers[l - 1].out_bits;
        if (!encode_packed_map(&maps.m[l], in, l == 0 ? ldap : ldob, M, K, BM)) return BNN_ERR_CUDA;
    }
    // The CTAs of a run wait for one another.  (Launched so, it starts when the kernel before it has ended; as a programmatic
    // dependent launch it would save 2 us, and two runs on two streams could each be placed in part and wait until they give up.)
    if (n_layers > 1) {
        if (launch_cooperative(kern, dim3(grid), dim3(THREADS), SMEM_BYTES, st, maps, a) != cudaSuccess) return BNN_ERR_CUDA;
    } else {
        kern<<<grid, THREADS, SMEM_BYTES, st>>>(maps, a);
    }
    return launch_status();
}

}  // namespace

// Units per tile for a layer of this shape, or 0 when the kernel does not apply: the stages of a layer must fit the
// shared-memory region, and every unit tile needs a CTA of its own.  Of the tiles that fit the one with the least estimated
// time per layer: the stages of the busiest CTA's frame tiles (clocks as measured), and where the region does not hold the
// next layer's weights beside this one's what their reload adds.  Wide tiles win for large batches (fewer, fuller MMAs),
// narrow ones where there are too few frame tiles for all SMs.  Measured on B200, four 2048-wide layers, microseconds with
// 192 / 128 / 96 / 32 units: 100 frames 29.5 / 27.3 / 27.0 / 25.5, 731 frames 30.4 / 28.5 / 28.8 / 33.5, 2000 frames
// 35.4 / 33.8 / 37.3 / 71, 4000 frames 43 / 47 / 62 / 128.
static int tile_units(int M, int N, int K, int sm_count, long long& best_cost) {
    const int nks = ceil_div(K, BK), m_tiles = ceil_div(M, BM);
    if (nks > Cfg<128>::SLOTS) return 0;
    struct Candidate { int bn, slots, stage; };
    const Candidate all[] = {{192, Cfg<192>::SLOTS, 480}, {128, Cfg<128>::SLOTS, 460}, {96, Cfg<96>::SLOTS, 450}, {32, Cfg<32>::SLOTS, 400}};
    int best = 0;
    best_cost = 0;
    for (const Candidate& c : all) {
        const int n_tiles = ceil_div(N, c.bn);
        if (nks > c.slots || n_tiles > sm_count) continue;
        const int peers = sm_count / n_tiles;
        const long long cost = (long long)ceil_div(m_tiles, peers) * nks * c.stage + (2 * nks <= c.slots ? 0 : c.bn * nks * 2 / 3);
        if (best == 0 || cost < best_cost) { best = c.bn; best_cost = cost; }
    }
    return best;
}

static int sm_count_of_device() { return device_sm_count(); }

bool xnor_res_applicable(int N, int K) {
    const int sms = sm_count_of_device();
    long long cost;
    return sms > 0 && tile_units(BM, N, K, sms, cost) != 0;
}

size_t xnor_stack_sync_bytes(int M, int n_layers) {
    return n_layers > 1 ? (size_t)(n_layers - 1) * ceil_div(M, BM) * sizeof(int) : 0;
}

int launch_xnor_stack(const uint32_t* Ap, int ldap, const XnorStackLayer* layers, int n_layers, int M, int N, int K,
                      int ldob, int zo, int* progress, cudaStream_t st) {
    const int sms = sm_count_of_device();
    if (sms <= 0) return BNN_ERR_CUDA;
    if (n_layers < 1 || n_layers > kXnorStackMax || (n_layers > 1 && (N != K || !progress))) return BNN_ERR_UNSUPPORTED;
    long long cost;
    const int bn = tile_units(M, N, K, sms, cost);
    // Pairs of CTAs for fan-ins above 2048, whose weights leave a CTA 128 units, where they are estimated to be faster (passes of six layers, us: 65536 frames of
    // 3072 units 3156 -> 2934, 16384 448 -> 384, 8192 239 -> 214, 2500 112 -> 98; 9000 of 2900 258 -> 216; 5000 of 2560 138 -> 120).  Elsewhere tiles of 256 frames x 256 units leave
    // more of the last turn empty than they save (8192 x 2048: a pass 237 -> 240 us; 731 frames 84 -> 91).
    const long long pair_cost = xnor_pair_clocks(M, N, K, sms);
    if (bn != 0 && K > 2048 && pair_cost > 0 && pair_cost < cost)
        return launch_xnor_pair(Ap, ldap, layers, n_layers, M, N, K, ldob, zo, progress, st);
    if (bn == 192) return launch_bn<192>(Ap, ldap, layers, n_layers, M, N, K, ldob, zo, progress, sms, st);
    if (bn == 128) return launch_bn<128>(Ap, ldap, layers, n_layers, M, N, K, ldob, zo, progress, sms, st);
    if (bn == 96) return launch_bn<96>(Ap, ldap, layers, n_layers, M, N, K, ldob, zo, progress, sms, st);
    if (bn == 32) return launch_bn<32>(Ap, ldap, layers, n_layers, M, N, K, ldob, zo, progress, sms, st);
    return BNN_ERR_UNSUPPORTED;
}

int launch_xnor_res(const uint32_t* Ap, int ldap, const void* image, int M, int N, int K,
                    const int32_t* thr, const uint32_t* flip, uint32_t* out_bits, int ldob, int zo, cudaStream_t st) {
    const XnorStackLayer one{image, thr, flip, out_bits};
    return launch_xnor_stack(Ap, ldap, &one, 1, M, N, K, ldob, zo, nullptr, st);
}

}  // namespace bnn
