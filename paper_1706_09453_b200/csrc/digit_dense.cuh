// The layers with binary weights on real-valued input (signw_digit_tc.cu), and top layers whose weights lose as pairs (out_digit_tc.cu): every number by itself in
// byte digits (digit_gemm.cuh has the products of sums and differences of pairs), exact integer products with packed sign bits on the tensor cores (tcgen05 kind::i8), on CTA pairs.
//
//   S[a][b] = sum_k sigma[a][k] * v[b][k],    sigma in {-1, +1} (or {0, 1}),  v = round(real[b][k] * 2^e_b)
//
// Every row of the real operand is scaled by a power of two (out_digit_tc.cu: by any number) of its own to a fixed-point number of about 23 bits (or, with four digits, 31) and
// written in base 256 with balanced digits, v = d0 + 256 d1 + 65536 d2 (-128 <= d <= 127), i.e. three bytes per
// element; the 32-bit sums are exact (K <= kMaxKDigit), so the only rounding is that of v, at most
// 1.01 * 2^-23 of the row's largest magnitude per element (1 / 0x7F7F7F, see scale_exponent), and those of the result.
// A sum of a pair needs a bit more than its two numbers.  These are not known before the call, and may all be of about the row's largest
// magnitude: as pairs such rows were up to 1.4 times as far off (rms; uniform in +-0.99: 1.3), and a pass gained 1-2 % at most
// (8192 frames, six layers 2048 wide 728 -> 720 us, 517 frames 101 -> 99; 14000 x 1035 -> 314 units by itself 52 -> 60).
//
// Layout: the bits are the M operand, the digits the N operand.  A pair of CTAs (cluster of two, one per SM of
// a TPC) works on a tile of 256 bit rows x N digit rows; each CTA widens its own 128 bit rows into its
// tensor memory (the MMA reads its A operand from there, so the widened bits cost the shared memory nothing) and
// loads half of the digit rows into its shared memory.  Granules of digit rows as in digit_gemm.cuh; the image is [K / 16][rows][16 bytes]; inside a group of
// 32 positions of K byte 4 t + j belongs to k = t + 8 j, which makes widening a shift and one logic operation per four positions.
// N is a launch argument, 192 or 96 (64 or 32 b): the narrow tile fills more SMs when the batch is small (tile_rows).
//
// Roles in a CTA of 20 warps:
//   warps 0-7    epilogue (the kernel's own), two warps per tensor-memory lane quarter; two accumulators, so the
//                epilogue of a tile overlaps the MMAs of the next
//   warps 8, 9   rank 0: issue the MMAs of the pair and the commits, which arrive in both CTAs.  The two warps
//                take blocks of 256 positions in turn; the sums are exact, so their order does not matter
//   warp 10      one thread issues the TMA loads of the digit image
//   warps 12-19  two teams of four warps widen the bit rows, thread = one row; each team one half of every stage
// A stage is complete when rank 0's barriers have the arrivals (or bytes) of BOTH CTAs; the partner arrives there directly.
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles of both CTAs fall through
// to the common teardown (the partner's waits run out too) and the device status word is set.
#pragma once

#include "digit_gemm.cuh"

namespace bnn {
namespace digit {
namespace dense {

constexpr uint32_t A_COLS = KB / 4;           // 32-bit tensor-memory columns per stage of bits
constexpr int B_STAGE = MAX_N / 2 * KB;       // 24 KB: shared memory of a stage of digits (half of it used when N = 96)
constexpr int B_STAGES = 7, MAX_B_STAGES = 14, MAX_A_STAGES = 4;
constexpr int RING_BYTES = B_STAGES * B_STAGE;

struct Bars {
    uint64_t full_a[2 * MAX_A_STAGES], empty_a[2 * MAX_A_STAGES];      // per half of a stage (one team's share)
    uint64_t full_b[MAX_B_STAGES], empty_b[MAX_B_STAGES];
    uint64_t acc_full[2], acc_empty[2], started[2];
    uint32_t tmem_base;
    WaitState wait;
};

// The tiles of a launch: 256 bit rows x `n` digit rows.
struct Work {
    int a_rows, b_rows;        // rows of the two operands
    int n, nd;                 // digit rows per tile, digits per element
    int steps;                 // groups of 32 positions of K
    int b_fast;
    __device__ __forceinline__ int grans() const { return n / (GRAN * nd); }                // granules per tile
    __device__ __forceinline__ int nb() const { return grans() * GRAN; }                    // b per tile
    __device__ __forceinline__ int a_tiles() const { return (a_rows + 2 * ROWS - 1) / (2 * ROWS); }
    __device__ __forceinline__ int b_tiles() const { return (b_rows + nb() - 1) / nb(); }
    __device__ __forceinline__ int a_stages() const { return n == MAX_N ? 2 : MAX_A_STAGES; }
    __device__ __forceinline__ int b_stages() const { return n == MAX_N ? B_STAGES : MAX_B_STAGES; }
    __device__ __forceinline__ uint32_t b_stage_bytes() const { return (uint32_t)(n / 2 * KB); }
    __device__ __forceinline__ uint32_t a_col() const { return 2u * (uint32_t)n; }          // bits start after the two accumulators
};

// By one thread, or every `step`th barrier of a kind by each of `step` threads (one thread takes half a microsecond).
__device__ __forceinline__ void init_bars(Bars* bars, int first = 0, int step = 1) {
    for (int s = first; s < 2 * MAX_A_STAGES; s += step) {
        mbar_init(smem_u32(&bars->full_a[s]), 2 * TEAM_WARPS);     // rank 0: the widening warps of both CTAs
        mbar_init(smem_u32(&bars->empty_a[s]), 1);
    }
    for (int s = first; s < MAX_B_STAGES; s += step) {
        mbar_init(smem_u32(&bars->full_b[s]), 1);                  // rank 0: its copying thread (+ bytes of both CTAs)
        mbar_init(smem_u32(&bars->empty_b[s]), 1);
    }
    for (int b = first; b < 2; b += step) {
        mbar_init(smem_u32(&bars->acc_full[b]), 2);                // one commit of each issuing warp
        mbar_init(smem_u32(&bars->acc_empty[b]), 2 * EPI_WARPS);   // rank 0: the epilogue warps of both CTAs
        mbar_init(smem_u32(&bars->started[b]), 1);
    }
}
// Common set-up; returns the tensor-memory base.  Called by all threads of both CTAs.
__device__ __forceinline__ uint32_t set_up(Bars* bars, const TcStatus& status, int warp) {
    if (threadIdx.x == 0) init_bars(bars);
    return finish_set_up(bars, status, warp);
}

// Warp COPY_WARP, one thread.  `map`: the image as rows (16 positions of K) of 8-byte elements, boxes of N / 2
// digit rows x 16.  What lies beyond the image reads as zeros.
__device__ __forceinline__ void copy_digits(const Work& w, const CUtensorMap* map, uint32_t ring, Bars* bars, int rank) {
    volatile int* abort_flag = &bars->wait.abort;
    const int stages = w.b_stages();
    const uint32_t bytes = w.b_stage_bytes();
    int s = 0;
    uint32_t ph = 1;          // parity to wait for on `empty`: a fresh barrier passes parity 1
    for (Tiles t(w); t.left > 0; t.next()) {
        const int row0 = t.b * w.nb() * w.nd + rank * (w.n / 2);
        for (int k = 0; k < w.steps; k += KB / 32) {
            if (!mbar_wait(smem_u32(&bars->empty_b[s]), ph, abort_flag)) return;
            const uint32_t bar = smem_u32(&bars->full_b[s]);
            if (rank == 0) mbar_arrive_expect_tx(bar, 2 * bytes);
            tma_load_2d_pair(ring + s * bytes, map, row0 * 2, k * 2, peer_addr(bar, 0));
            if (++s == stages) { s = 0; ph ^= 1u; }
        }
    }
}

// Eight words of four bytes: word t holds bits t, t + 8, t + 16, t + 24 as +64 / -64 (or, ZO, 64 / 0): 64 and -64
// differ in the top bit of the byte alone, so that a word is a shift and one three-input logic operation (+1 / -1 would
// take a third).  The sums come out 64 times as large.
template <bool ZO>
__device__ __forceinline__ void widen_bytes(uint32_t word, uint32_t* o) {
#pragma unroll
    for (int t = 0; t < 8; ++t) {
        if (ZO) o[t] = (t < 7 ? word << (6 - (t < 7 ? t : 6)) : word >> 1) & 0x40404040u;
        else o[t] = (~(word << (7 - t)) & 0x80808080u) ^ 0x40404040u;
    }
}

// Warps PROD_WARP0 ..: thread = one bit row of this CTA; each team takes 128 positions of every stage.  The packed row is
// read 16 bytes (the team's share of a stage) at a time, two stages ahead of use.  Bits at positions >= K may
// hold anything: the digits are zero there.
template <bool ZO>
__device__ __forceinline__ void widen_bits(const Work& w, const uint32_t* __restrict__ P, int ldp, Bars* bars, uint32_t tmem,
                                           int rank, int warp, int lane) {
    volatile int* abort_flag = &bars->wait.abort;
    Tiles t(w);
    const int total_tiles = t.left;
    const int team = (warp - PROD_WARP0) / TEAM_WARPS;
    const int r = (warp & 3) * 32 + lane;                   // a warp may only touch the lanes of its quarter
    const uint32_t tdst = tmem + ((uint32_t)((warp & 3) * 32) << 16) + w.a_col() + (uint32_t)team * (A_COLS / 2);
    const int groups = (w.steps + 3) >> 2, blocks = (w.steps + 7) >> 3;     // 128-position groups and stages per tile
    const int a_stages = w.a_stages();
    int pf_g = team;                                        // the next group to fetch, of the tile `t` is at
    auto row_of = [&]() {
        const int row = t.a * (2 * ROWS) + rank * ROWS + r;
        return t.left > 0 && row < w.a_rows ? reinterpret_cast<const uint4*>(P + (size_t)row * ldp) : nullptr;
    };
    const uint4* pf_row = row_of();
    auto fetch = [&]() {
        uint4 o = make_uint4(0u, 0u, 0u, 0u);
        if (pf_row && pf_g < groups) o = ldg_nc_u4(pf_row + pf_g);
        pf_g += TEAMS;
        if (pf_g >= 2 * blocks) { pf_g = team; t.next(); pf_row = row_of(); }
        return o;
    };
    int s = 0;
    uint32_t ph = 1;
    const int total = total_tiles * blocks;
    uint4 cur = fetch(), nxt = fetch();
    uint32_t o[32];
    auto widen = [&](const uint4& v) {
        widen_bytes<ZO>(v.x, o); widen_bytes<ZO>(v.y, o + 8); widen_bytes<ZO>(v.z, o + 16); widen_bytes<ZO>(v.w, o + 24);
    };
    widen(cur);
    for (int it = 0; it < total; ++it) {
        // what lies between a free slot and a full one is kept short: the row was widened before the wait
        if (!warp_wait(smem_u32(&bars->empty_a[2 * s + team]), ph, abort_flag, lane)) return;
        tc_fence_after_sync();
        tmem_st32(tdst + s * A_COLS, o);
        cur = nxt;
        nxt = fetch();
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {
            const uint32_t bar = smem_u32(&bars->full_a[2 * s + team]);
            if (rank == 0) mbar_arrive(bar);
            else mbar_arrive_cluster(peer_addr(bar, 0));
        }
        if (++s == a_stages) { s = 0; ph ^= 1u; }
        widen(cur);
    }
}

// Both barriers of a stage: polled together first, so that a stage that is ready costs one round trip.
__device__ __forceinline__ bool warp_wait_both(uint32_t bar0, uint32_t par0, uint32_t bar1, uint32_t par1, volatile int* abort_flag) {
    const bool r0 = mbar_try_wait(bar0, par0), r1 = mbar_try_wait(bar1, par1);
    if (__all_sync(0xFFFFFFFFu, r0 && r1)) return true;
    return warp_wait(bar0, par0, abort_flag, 0) && warp_wait(bar1, par1, abort_flag, 0);
}

// Warps MMA_WARP and MMA_WARP2 of rank 0, converged; they take the stages of a tile in turn.  What an issuing
// warp does besides its MMAs (waits about 100 clocks each even when they succeed, commits) is time that only the
// other warp's MMAs can fill.  The bits of a stage come and go in two halves: tensor memory holds only two stages
// beside the accumulators, and a half that is handed back after its four MMAs has the time of twelve to be refilled.
__device__ __forceinline__ void issue(const Work& w, uint32_t ring, Bars* bars, uint32_t tmem, int which) {
    volatile int* abort_flag = &bars->wait.abort;
    const int tiles = Tiles(w).left;
    const uint32_t idesc = instr_desc(kAccS32, kFmtS8, kFmtS8, 2 * ROWS, w.n);
    const int a_stages = w.a_stages(), b_stages = w.b_stages();
    const uint32_t chunk16 = (uint32_t)(w.n / 2);            // 16-byte units between chunks of 16 positions
    const uint32_t stage16 = w.b_stage_bytes() >> 4;
    const uint64_t desc = smem_desc_kmajor(ring, chunk16 * 16u, 128);
    const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32), step16 = 2 * chunk16;   // an MMA takes two chunks
    const uint32_t ta0 = tmem + w.a_col();
    const int blocks = (w.steps + 7) >> 3;
    int sa = 0, sb = 0;
    uint32_t pa = 0, pb = 0;
    for (int tl = 0; tl < tiles; ++tl) {
        const int b = tl & 1;
        if (!warp_wait(smem_u32(&bars->acc_empty[b]), (uint32_t)(((tl >> 1) & 1) ^ 1), abort_flag, 0)) return;
        tc_fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(b * w.n);
        for (int kb = 0; kb < blocks; ++kb) {
            if ((kb & 1) == which) {
                // The MMA that overwrites the accumulator has to come first.  This wait also stands before those for the
                // stage, because a wait on a parity holds only for one who knows that the phase before it is over.  With
                // an odd number of stages per tile the other warp takes two in a row, the last of a tile and the first
                // of the next; when there are two slots the former had this stage's.  `started` says that the other
                // warp has issued the latter, so it has found the former full.
                if (kb == 1 && !warp_wait(smem_u32(&bars->started[b]), (uint32_t)((tl >> 1) & 1), abort_flag, 0)) return;
                if (!warp_wait_both(smem_u32(&bars->full_b[sb]), pb, smem_u32(&bars->full_a[2 * sa]), pa, abort_flag)) return;
                tc_fence_after_sync();
                // the address field (16-byte units) is advanced by plain additions: the ring lies below 2^14 * 16 bytes
                const uint32_t db = desc_lo + (uint32_t)sb * stage16;
                const uint32_t ta = ta0 + (uint32_t)sa * A_COLS;
                const int n_mma = w.steps - 8 * kb;           // 8 but for the last stage
                if (elect_one()) {
                    mma_i8_ts_pair(d, ta, db, desc_hi, idesc, kb != 0);
                    if (kb == 0) mma_commit_pair(smem_u32(&bars->started[b]));
                    if (n_mma >= 4) {
                        mma_i8_ts_pair(d, ta + 8, db + step16, desc_hi, idesc, 1u);
                        mma_i8_ts_pair(d, ta + 16, db + 2 * step16, desc_hi, idesc, 1u);
                        mma_i8_ts_pair(d, ta + 24, db + 3 * step16, desc_hi, idesc, 1u);
                    } else {
                        for (int j = 1; j < n_mma; ++j) mma_i8_ts_pair(d, ta + 8 * j, db + j * step16, desc_hi, idesc, 1u);
                    }
                    mma_commit_pair(smem_u32(&bars->empty_a[2 * sa]));
                }
                if (!warp_wait(smem_u32(&bars->full_a[2 * sa + 1]), pa, abort_flag, 0)) return;
                tc_fence_after_sync();
                if (elect_one()) {
                    if (n_mma >= 8) {
                        mma_i8_ts_pair(d, ta + 32, db + 4 * step16, desc_hi, idesc, 1u);
                        mma_i8_ts_pair(d, ta + 40, db + 5 * step16, desc_hi, idesc, 1u);
                        mma_i8_ts_pair(d, ta + 48, db + 6 * step16, desc_hi, idesc, 1u);
                        mma_i8_ts_pair(d, ta + 56, db + 7 * step16, desc_hi, idesc, 1u);
                    } else {
                        for (int j = 4; j < n_mma; ++j) mma_i8_ts_pair(d, ta + 8 * j, db + j * step16, desc_hi, idesc, 1u);
                    }
                    mma_commit_pair(smem_u32(&bars->empty_a[2 * sa + 1]));
                    mma_commit_pair(smem_u32(&bars->empty_b[sb]));
                }
            }
            if (++sa == a_stages) { sa = 0; pa ^= 1u; }
            if (++sb == b_stages) { sb = 0; pb ^= 1u; }
        }
        if (elect_one()) mma_commit_pair(smem_u32(&bars->acc_full[b]));
    }
}

// ---- scales: powers of two, so that a number is rounded once and a scale costs no rounding -------------------
// 2^h for -126 <= h <= 127.
__device__ __forceinline__ float power_of_two(int h) { return __int_as_float((127 + h) << 23); }
// What a unit of a row whose scale_exponent is e stands for: 2^-e.
__device__ __forceinline__ float inverse_scale(int e) {
    const int h = e >> 1;
    return power_of_two(-h) * power_of_two(h - e);
}
// x * 2^e rounded to an integer; 2^e comes as two powers of two (e may be beyond the exponent range of one).
struct Scale {
    float a, b;
    __device__ __forceinline__ explicit Scale(int e) : a(power_of_two(e >> 1)), b(power_of_two(e - (e >> 1))) {}
    __device__ __forceinline__ int fixed_point(float x) const { return __float2int_rn(x * a * b); }
};

// Digit rows per tile (192 or 96) for `a_rows` x `b_rows` outputs on `pairs` CTA pairs: the one with the least
// estimated time.  An MMA of 32 positions takes N / 2 clocks in the tensor pipe but not less than about 70, the
// rate at which it can be issued; a launch takes ceil(tiles / pairs) turns.
inline long long tile_count(int a_rows, int b_rows, int n) { return (long long)ceil_div(a_rows, 2 * ROWS) * ceil_div(b_rows, n / 3); }
inline int tile_rows(int a_rows, int b_rows, int steps, int pairs) {
    auto cost = [&](int n, int clocks) { return (tile_count(a_rows, b_rows, n) + pairs - 1) / pairs * ((long long)steps * clocks + 800); };
    return cost(96, 70) < cost(192, 100) ? 96 : 192;
}

}  // namespace dense
}  // namespace digit
}  // namespace bnn
