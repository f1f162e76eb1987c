// Products of a real-valued operand with packed sign bits as exact integer products on the tensor cores
// (tcgen05 kind::i8, 2:4 sparse), on CTA pairs: the engine of the top layer on packed activations (out_digit_tc.cu), and what it
// shares with that of the layers with binary weights on real-valued input (digit_dense.cuh).
//
// Two signs times two numbers are one sign times one number: s1 v1 + s2 v2 = s1 (v1 + v2) where s1 = s2 and s1 (v1 - v2)
// elsewhere.  With the digits operand holding the sum and the difference of every pair (k, k + 16) in place of the two values,
// a row of signs has exactly one +-1 and one 0 for each pair: the 2:4 sparsity of the tensor core, which takes 64
// positions in the time of 32 (measured on B200, 256 x 192 outputs per CTA pair: 96 clocks either way).
//
//   S[a][b] = sum over pairs of sigma[a][k] * v[b][pair, choice],    v = round((real[b][k] +- real[b][k + 16]) / r_b)
//
// Every row of the real operand has a scale r_b of its own, such that its largest pair comes close to 0x7F7F7F, and is written in
// base 256 with balanced digits, v = d0 + 256 d1 + 65536 d2 (-128 <= d <= 127), i.e. three bytes per
// element.  The tensor core multiplies bytes at twice the rate of half-precision numbers, and
// its 32-bit sums are exact (K <= kMaxKDigit), so S is exact: the only roundings are that of v, at most
// r_b / 2 <= 1.01 * 2^-23 of the row's largest magnitude per pair (v is formed in double precision), and those of the result to fp32.  A pair's sum
// has a bit more than its two values.  Half as many roundings and scales that use
// the whole range make up for it unless a row fills its range evenly just below a power of two: rms error of a sum, over that of rounding every value
// to a power of two, 440 / 2048 values: N(0, 1) 0.74 - 0.80, uniform in +-0.7 0.88, in +-0.033 0.72, but in +-0.99 1.21 - 1.23, of 0.9 .. 1 1.15.  Such matrices go
// to digit_dense.cuh (out_digit_tc.cu).
//
// Layout: the bits are the M operand, the digits the N operand.  A pair of CTAs (cluster of two, one per SM of
// a TPC) works on a tile of 256 bit rows x two parts of N digit rows; each CTA widens its own 128 bit rows into its
// tensor memory (the MMA reads its A operand and its metadata from there, so the widened bits cost the shared memory nothing) and
// loads half of the digit rows into its shared memory.  The digits of 8 consecutive b are one granule of 8 ND
// digit rows, row = (b / 8) 8 ND + q 8 + b % 8, so a thread of the epilogue finds the ND sums of an output in its own
// tensor-memory lane.  The image is [K / 16][rows][16 bytes]; which byte of a group of 64 positions belongs to which
// pair is chosen so that widening is cheap (widen_pairs, image_byte).
// N is a launch argument, 192, 96 or 48 (64, 32 or 16 b with three digits): narrow tiles fill more SMs when the batch is small
// (tile_rows).  Both parts meet the same widened bits: what widening costs (some 60 instructions per thread and 128
// positions, and shifts and logic operations share a pipe of half the rate) is spread over 384 digit rows.  The other
// way to share, two blocks of 256 bit rows on one part of digits, halves the bytes from L2 instead, but widens twice as much:
// 8192 x 3400 x 2048, 84 us.
//
// Roles in a CTA of 20 warps:
//   warps 0-7    epilogue (the kernel's own), two warps per tensor-memory lane quarter
//   warps 8, 9   rank 0: issue the MMAs of the pair and the commits, which arrive in both CTAs.  Each warp has a part with its
//                accumulator; since the epilogue reads one accumulator after the other, one part runs ahead and its
//                epilogue is hidden behind the other's MMAs.
//   warp 10      one thread issues the TMA loads of the digit image
//   warps 12-19  widen the bit rows, thread = one row; two teams of four warps, each one half of every stage
// A stage, 256 positions of K, is one barrier: it is complete when rank 0's has the arrivals and bytes of BOTH CTAs; the partner arrives there
// directly.  (Measured on B200: a thread of rank 1 that waits for its own CTA's stage and passes it on with a
// cluster-scope release costs 1200 clocks per stage, whatever its size.  A wait costs an issuing warp some 180 clocks even when it
// succeeds at once, beside 16 warps that compute: one wait for the bits and one for the digits, of 128 positions each, left
// the tensor pipe idle half of the time.)
// Every wait is bounded; a wait that runs out sets the CTA's abort flag, all roles of both CTAs fall through
// to the common teardown (the partner's waits run out too) and the device status word is set.
#pragma once

#include "bnn_common.cuh"
#include "tcgen05.cuh"

namespace bnn {
namespace digit {

using namespace tc;

constexpr int ROWS = 128;                     // bit rows per CTA
constexpr int GRAN = 8;                       // b per granule
constexpr int KB = 256;                       // positions of K per stage
constexpr int GROUP = 64;                     // positions per MMA
constexpr uint32_t TEAM_COLS = KB / GROUP / 2 * 10, STAGE_COLS = 2 * TEAM_COLS;    // 32-bit tensor-memory columns: 8 of signs and 2 of metadata per group
constexpr int PARTS = 2;                      // of a tile: accumulators, issuing warps
constexpr int MAX_N = 192;
constexpr int MAX_STAGES = 8;
constexpr int RING_BYTES = 7 * 96 * KB;       // 168 KB of digits: 3 stages of N = 192, 7 of 96, 8 of 48
constexpr int EPI_WARPS = 8, MMA_WARP = 8, MMA_WARP2 = 9, COPY_WARP = 10, PROD_WARP0 = 12, TEAM_WARPS = 4, TEAMS = 2;
constexpr int THREADS = (PROD_WARP0 + TEAMS * TEAM_WARPS) * 32;
// What the kernels declare as their largest block: caps them at 80 registers a thread, which leaves room on the SM for
// the block of the log-softmax that follows the top layer (four warps of 96).
constexpr int REG_THREADS = 768;
constexpr uint32_t TMEM_COLS = 512;

struct Bars {
    uint64_t full[MAX_STAGES], empty[MAX_STAGES];
    uint64_t acc_full[PARTS], acc_empty[PARTS];
    uint32_t tmem_base;
    WaitState wait;
};

// The tiles of a launch: 256 bit rows x 2 parts of `n` digit rows; consecutive tiles share the bit rows (b_fast) or the digits.
struct Work {
    int a_rows, b_rows;        // rows of the two operands
    int n, nd;                 // digit rows per part, digits per element
    int steps, half_tail;      // groups of 64 positions of K; whether the last one has 32 at most
    int b_fast;
    __device__ __forceinline__ int grans() const { return n / (GRAN * nd); }                // granules per part (the rows left over are not used)
    __device__ __forceinline__ int part_b() const { return grans() * GRAN; }
    __device__ __forceinline__ int a_tiles() const { return (a_rows + 2 * ROWS - 1) / (2 * ROWS); }
    __device__ __forceinline__ int b_tiles() const { return (b_rows + PARTS * part_b() - 1) / (PARTS * part_b()); }
    __device__ __forceinline__ int ring() const { return n == MAX_N ? 3 : n == MAX_N / 2 ? 7 : MAX_STAGES; }
    __device__ __forceinline__ uint32_t stage_bytes() const { return (uint32_t)(n * KB); }  // digits of both parts in one CTA
    __device__ __forceinline__ int stages() const { return (steps + KB / GROUP - 1) / (KB / GROUP); }          // of a tile
    __device__ __forceinline__ uint32_t a_col() const { return (uint32_t)(PARTS * n); }     // bits start after the accumulators
    // Epilogue warps 0-3 and 4-7 halve every part (of 192 digit rows), or have a part each: 32 b per warp with three digits, so
    // that a row of its stores is 128 bytes (64 take twice as many sectors at odd offsets: 731 frames x 3307 classes, 89 us
    // a pass against 85).
    __device__ __forceinline__ bool halved() const { return n == MAX_N; }
    // Whether a part of a tile lies beyond the digits; such a part is left out.
    __device__ __forceinline__ bool beyond(int tile_b, int part) const { return (tile_b * PARTS + part) * part_b() >= b_rows; }
};
// The tiles of this CTA pair in order.  Integer divisions only here, once per role: one per tile, let alone per stage,
// costs the producers more than the widening itself.
struct Tiles {
    int a, b;                  // coordinates of the current tile
    int left;                  // tiles from the current one on
    template <typename W>
    __device__ __forceinline__ explicit Tiles(const W& w) {
        const int pairs = (int)gridDim.x >> 1, first = (int)blockIdx.x >> 1;
        const int na = w.a_tiles(), nb = w.b_tiles(), count = na * nb;
        left = first < count ? (count - 1 - first) / pairs + 1 : 0;
        b_fast_ = w.b_fast;
        fast_n_ = b_fast_ ? nb : na;
        step_slow_ = pairs / fast_n_;
        step_fast_ = pairs - step_slow_ * fast_n_;
        const int slow = first / fast_n_;
        set(first - slow * fast_n_, slow);
    }
    __device__ __forceinline__ void next() {
        --left;
        int fast = (b_fast_ ? b : a) + step_fast_, slow = (b_fast_ ? a : b) + step_slow_;
        if (fast >= fast_n_) { fast -= fast_n_; ++slow; }
        set(fast, slow);
    }

private:
    int b_fast_, fast_n_, step_fast_, step_slow_;
    __device__ __forceinline__ void set(int fast, int slow) { a = b_fast_ ? slow : fast; b = b_fast_ ? fast : slow; }
};

// The end of the set-up: thread 0 has initialised the barriers of `bars`.  Returns the tensor-memory base.
template <typename B>
__device__ __forceinline__ uint32_t finish_set_up(B* bars, const TcStatus& status, int warp) {
    if (threadIdx.x == 0) {
        wait_state_init(&bars->wait, status);
        mbar_init_fence();
    }
    __syncwarp();
    if (warp == MMA_WARP) tmem_alloc_pair(smem_u32(&bars->tmem_base), TMEM_COLS);
    tc_fence_before_sync();
    cluster_sync();           // barriers of both CTAs initialised, tensor memory of both allocated
    tc_fence_after_sync();
    return bars->tmem_base;
}
// Common set-up; returns the tensor-memory base.  Called by all threads of both CTAs.
__device__ __forceinline__ uint32_t set_up(Bars* bars, const TcStatus& status, int warp, bool halved) {
    if (threadIdx.x == 0) {
        for (int s = 0; s < MAX_STAGES; ++s) {
            mbar_init(smem_u32(&bars->full[s]), 2 * TEAMS * TEAM_WARPS + 1);  // rank 0: the widening warps of both CTAs, its copying thread (+ bytes of both CTAs)
            mbar_init(smem_u32(&bars->empty[s]), PARTS);               // a commit of each issuing warp
        }
        for (int b = 0; b < PARTS; ++b) {
            mbar_init(smem_u32(&bars->acc_full[b]), 1);
            mbar_init(smem_u32(&bars->acc_empty[b]), halved ? 2 * EPI_WARPS : EPI_WARPS);   // rank 0: the epilogue warps of both CTAs that read it
        }
    }
    return finish_set_up(bars, status, warp);
}

// Common teardown; every thread of both CTAs arrives here, also after an aborted wait.
template <typename B>
__device__ __forceinline__ void tear_down(B* bars, const TcStatus& status, int warp, uint32_t tmem) {
    __syncwarp();
    tc_fence_before_sync();
    cluster_sync();           // nobody reads the partner's shared or tensor memory any more
    if (warp == MMA_WARP) {
        tc_fence_after_sync();
        tmem_dealloc_pair(tmem, TMEM_COLS);
    }
    if (threadIdx.x == 0 && bars->wait.abort) atomicExch(status.word, 1);
}

// Warp COPY_WARP, one thread.  `map`: the image as rows (16 positions of K) of 8-byte elements, boxes of N / 2
// digit rows x 16.  What lies beyond the image reads as zeros.
__device__ __forceinline__ void copy_digits(const Work& w, const CUtensorMap* map, uint32_t ring, Bars* bars, int rank) {
    volatile int* abort_flag = &bars->wait.abort;
    const int ring_stages = w.ring(), stages = w.stages(), part_rows = w.part_b() * w.nd;
    const uint32_t bytes = w.stage_bytes();
    int s = 0;
    uint32_t ph = 1;          // parity to wait for on `empty`: a fresh barrier passes parity 1
    for (Tiles t(w); t.left > 0; t.next()) {
        const int row0 = t.b * PARTS * part_rows + rank * (w.n / 2);
        for (int kb = 0; kb < stages; ++kb) {
            if (!mbar_wait(smem_u32(&bars->empty[s]), ph, abort_flag)) return;
            const uint32_t bar = smem_u32(&bars->full[s]), bar0 = peer_addr(bar, 0), dst = ring + s * bytes;
            if (rank == 0) mbar_arrive_expect_tx(bar, 2 * bytes);
            tma_load_2d_pair(dst, map, row0 * 2, kb * (KB / 16), bar0);
            tma_load_2d_pair(dst + (bytes >> 1), map, (row0 + part_rows) * 2, kb * (KB / 16), bar0);
            if (++s == ring_stages) { s = 0; ph ^= 1u; }
        }
    }
}

// A group of 64 positions, two packed words.  Its 32 pairs are bit i of `sign` (position i of w0's lower half, or of w1's) and bit i
// of `other` (16 positions on); the pair takes the difference where the two differ.  Compressed byte 4 j + q is pair
// t(j) + 8 q, t(j) = 4 (j / 2 % 2) + 2 (j % 2) + j / 4, so that
//   - a word of signs, o[j], is a shift and one three-input logic operation: 64 and -64 differ in the top bit of the byte alone (+1 / -1
//     would take a third; the sums come out 64 times as large);
//   - the metadata, o[8] and o[9], are the choices with two pairs of bits of the bit index exchanged (16 with 4, 8 with 2).  The
//     indices of compressed bytes 2 c and 2 c + 1, positions 0 or 1 and 2 or 3 of group c of four, are 0 + choice and 2 + choice.
__device__ __forceinline__ void widen_pairs(uint32_t w0, uint32_t w1, uint32_t* signs, uint32_t* meta) {
    const uint32_t sign = __byte_perm(w0, w1, 0x5410), other = __byte_perm(w0, w1, 0x7632);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        const int t = 4 * ((j >> 1) & 1) + 2 * (j & 1) + (j >> 2);
        signs[j] = (~(sign << (7 - t)) & 0x80808080u) ^ 0x40404040u;
    }
    uint32_t x = sign ^ other, y = ((x >> 12) ^ x) & 0x0000F0F0u;
    x ^= y ^ (y << 12);
    y = ((x >> 6) ^ x) & 0x00CC00CCu;
    x ^= y ^ (y << 6);
    meta[0] = (x & 0x55555555u) | 0x88888888u;
    meta[1] = ((x >> 1) & 0x55555555u) | 0x88888888u;
}
// The other side of it: where in the 64 bytes of a group the digits of pair (k, k + 16) lie, k = 32 w + t + 8 q (w, q = 0, 1; t < 8):
// the sum at image_byte, the difference behind it.  A last group that is one word (`half`) has its 16 pairs in its first two
// chunks of 16 bytes, and the image ends there; w = 0.
__host__ __device__ __forceinline__ constexpr int image_byte(bool half, int w, int t, int q) {
    return half ? 8 * (t & 3) + 4 * (t >> 2) + 2 * q : 32 * (t & 1) + 16 * (t >> 2) + 8 * ((t >> 1) & 1) + 4 * w + 2 * q;
}
// The bits of such a word, spread over the two words of a whole group: bit t + 8 q of either half goes to bit 16 (t / 4) + 8 q + 2 (t % 4)
// of `sign` or `other`.
__device__ __forceinline__ uint32_t spread_pairs(uint32_t x) {
    x = (x & 0x0F0Fu) | ((x & 0xF0F0u) << 12);
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}
__device__ __forceinline__ void spread_half_group(uint32_t& w0, uint32_t& w1) {
    const uint32_t sign = spread_pairs(w0 & 0xFFFFu), other = spread_pairs(w0 >> 16);
    w0 = __byte_perm(sign, other, 0x5410);
    w1 = __byte_perm(sign, other, 0x7632);
}

// Warps PROD_WARP0 ..: thread = one bit row of this CTA; each team takes 128 positions of every stage.  The packed row is
// read 16 bytes (the team's share of a stage) at a time, two stages ahead of use.
// Bits at positions >= K may hold anything: a pair's sum and difference are the same number where its second position is
// beyond K, and zero where both are.
__device__ __forceinline__ void widen_bits(const Work& w, const uint32_t* __restrict__ P, int ldp, Bars* bars, uint32_t tmem,
                                           int rank, int warp, int lane) {
    volatile int* abort_flag = &bars->wait.abort;
    Tiles t(w);
    const int team = (warp - PROD_WARP0) / TEAM_WARPS;
    const int r = rank * ROWS + (warp & 3) * 32 + lane;         // (a warp may only touch the lanes of its quarter)
    const uint32_t tdst = tmem + ((uint32_t)((warp & 3) * 32) << 16) + w.a_col() + (uint32_t)team * TEAM_COLS;
    const int words4 = (w.steps + 1) >> 1;                      // 16-byte pieces of a row
    const int stages = w.stages();
    const int missing = (stages - 1) * TEAMS + team >= words4 ? 1 : 0;           // of this team's pieces, in the last stage
    // of the stages of a tile, counted down: the one whose last group is half a group
    const int tail = w.half_tail && ((words4 - 1) & 1) == team ? 1 + missing : -1;
    const bool tail_high = !(w.steps & 1);
    const uint4* next_piece = nullptr;
    int pieces = 0;                                             // left of the tile that is being fetched
    int left = t.left * stages;                                 // stages still to be filled
    auto next_tile = [&]() {
        const int row = t.left > 0 ? t.a * (2 * ROWS) + r : 0;
        next_piece = reinterpret_cast<const uint4*>(P + (size_t)(row < w.a_rows ? row : 0) * ldp) + team;    // (rows beyond go nowhere)
        pieces = stages;
        t.next();
    };
    next_tile();
    auto fetch = [&]() {
        uint4 o = make_uint4(0u, 0u, 0u, 0u);
        if (pieces > missing) o = ldg_nc_u4(next_piece);
        next_piece += TEAMS;
        if (--pieces == 0) next_tile();
        return o;
    };
    const uint32_t end = tdst + (uint32_t)w.ring() * STAGE_COLS;
    uint32_t dst = tdst, empty = smem_u32(&bars->empty[0]), full = smem_u32(&bars->full[0]);
    if (rank != 0) full = peer_addr(full, 0);
    uint32_t ph = 1;
    uint4 cur = fetch(), nxt = fetch();
    uint32_t o[20];
    int at = stages;                                            // stages left of the tile that is being widened
    auto widen = [&](uint4 v) {
        if (at == tail) {
            if (tail_high) spread_half_group(v.z, v.w);
            else spread_half_group(v.x, v.y);
        }
        if (--at == 0) at = stages;
        widen_pairs(v.x, v.y, o, o + 16);
        widen_pairs(v.z, v.w, o + 8, o + 18);
    };
    widen(cur);
    for (; left > 0; --left) {
        // what lies between a free stage and a full one is kept short: the row was widened before the wait
        if (!warp_wait(empty, ph, abort_flag, lane)) return;
        tc_fence_after_sync();          // the MMAs that read these columns come first
        tmem_st16(dst, o);
        tmem_st4(dst + 16, o + 16);
        cur = nxt;
        nxt = fetch();
        tmem_st_wait();
        tc_fence_before_sync();
        __syncwarp();
        if (lane == 0) {
            if (rank == 0) mbar_arrive(full);
            else mbar_arrive_cluster(full);
        }
        dst += STAGE_COLS; empty += 8; full += 8;
        if (dst == end) {
            dst = tdst; empty -= 8 * (uint32_t)w.ring(); full -= 8 * (uint32_t)w.ring();
            ph ^= 1u;
        }
        widen(cur);
    }
}

// Warps MMA_WARP and MMA_WARP2 of rank 0, converged, each with its part of every tile.  What an issuing warp does besides its MMAs is
// time that only the other warp's MMAs can fill.
__device__ __forceinline__ void issue(const Work& w, uint32_t ring, Bars* bars, uint32_t tmem, int part) {
    volatile int* abort_flag = &bars->wait.abort;
    const uint32_t idesc = instr_desc(kAccS32, kFmtS8, kFmtS8, 2 * ROWS, w.n) | kSparse;
    const int ring_stages = w.ring(), stages = w.stages();
    const uint32_t chunk16 = (uint32_t)(w.n / 2);            // 16-byte units between chunks of 16 positions
    const uint32_t stage16 = w.stage_bytes() >> 4;
    const uint64_t desc = smem_desc_kmajor(ring + (uint32_t)part * (w.stage_bytes() >> 1), chunk16 * 16u, 128);
    const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32), step16 = 4 * chunk16;   // an MMA takes four chunks
    const uint32_t d = tmem + (uint32_t)(part * w.n), ta0 = tmem + w.a_col();
    int s = 0;
    uint32_t ph = 0, pacc = 1;
    for (Tiles t(w); t.left > 0; t.next()) {
        const bool beyond = w.beyond(t.b, part);
        if (!beyond) {
            if (!warp_wait(smem_u32(&bars->acc_empty[part]), pacc, abort_flag, 0)) return;
            tc_fence_after_sync();
            pacc ^= 1u;
        }
        for (int kb = 0; kb < stages; ++kb) {
            if (!warp_wait(smem_u32(&bars->full[s]), ph, abort_flag, 0)) return;
            tc_fence_after_sync();
            // the address field (16-byte units) is advanced by plain additions: the ring lies below 2^14 * 16 bytes
            const uint32_t db = desc_lo + (uint32_t)s * stage16, ta = ta0 + (uint32_t)s * STAGE_COLS;
            const int left = beyond ? 0 : w.steps - 4 * kb;   // groups: 4 but for the last stage
            if (elect_one()) {
                if (left > 0) mma_i8_sp_ts_pair(d, ta, ta + 16, db, desc_hi, idesc, kb != 0);
                if (left > 1) mma_i8_sp_ts_pair(d, ta + 8, ta + 18, db + step16, desc_hi, idesc, 1u);
                if (left > 2) mma_i8_sp_ts_pair(d, ta + TEAM_COLS, ta + TEAM_COLS + 16, db + 2 * step16, desc_hi, idesc, 1u);
                if (left > 3) mma_i8_sp_ts_pair(d, ta + TEAM_COLS + 8, ta + TEAM_COLS + 18, db + 3 * step16, desc_hi, idesc, 1u);
                mma_commit_pair(smem_u32(&bars->empty[s]));
                if (kb + 1 == stages && !beyond) mma_commit_pair(smem_u32(&bars->acc_full[part]));
            }
            if (++s == ring_stages) { s = 0; ph ^= 1u; }
        }
    }
}

// Epilogue warps: this warp has read its share of the tile's accumulator.
template <typename B>
__device__ __forceinline__ void release_acc(B* bars, int b, int lane) {
    tc_fence_before_sync();
    __syncwarp();
    if (lane == 0) mbar_arrive_cluster(peer_addr(smem_u32(&bars->acc_empty[b]), 0));
}

// The sums S of one granule (8 outputs of this thread's bit row) in fp32: with three digits the two low sums are
// joined exactly as an integer (below 2^24, i.e. an exact float, unless a row's middle digits add up almost
// without cancelling; then the rounding is still below the row's quantisation steps); with four, digit sums are carried
// into one another first.
__device__ __forceinline__ void load_granule(uint32_t taddr, int nd, uint32_t (&d)[4][8]) {
    tmem_ld8(taddr, d[0]);
    tmem_ld8(taddr + 8, d[1]);
    tmem_ld8(taddr + 16, d[2]);
    if (nd == 4) tmem_ld8(taddr + 24, d[3]);
}
// (2^24 high + more is added)
__device__ __forceinline__ float join4(int s0, int s1, int s2, int s3, int high = 0, int more = 0) {
    const int d0 = s0 >> 6;
    const int d1 = (s1 >> 6) + (d0 >> 8);
    const int d2 = (s2 >> 6) + (d1 >> 8);
    const int low = ((d2 & 255) << 16) | ((d1 & 255) << 8) | (d0 & 255);
    return fmaf((float)((s3 >> 6) + (d2 >> 8) + high), 16777216.0f, (float)(low + more));
}
// low + 65536 high, the two parts of a sum of three digits.
__device__ __forceinline__ float low_part(int s0, int s1) { return (float)(s1 * 4 + (s0 >> 6)); }
// The high sum is below 2^22: adding 1.5 * 2^23 as an integer to its bits makes it a float without the
// conversion unit, which the other conversion of every output already keeps busy.
__device__ __forceinline__ float high_part(int s2, int more = 0) { return __int_as_float((s2 >> 6) + more + 0x4B400000) - 12582912.0f; }
// Largest e (up to 140) such that mx * 2^e is a balanced number of three digits: at most 127 * (65536 + 256 + 1) = 0x7F7F7F.
// mx >= 0; its exponent and fraction fields are compared with those of the limit.
__device__ __forceinline__ int scale_exponent(float mx) {
    const int bits = __float_as_int(mx);
    if (bits == 0) return 0;
    const int e = 22 + 127 - (bits >> 23) - ((bits & 0x7FFFFF) > 0x7EFEFE ? 1 : 0);     // 0x7F7F7F / 2^22
    return e > 140 ? 140 : e;
}
// Half of |x1| + |x2|.
__device__ __forceinline__ float half_sum(float x1, float x2) { return fmaf(0.5f, x1, 0.5f * x2); }
// The balanced base-256 digits of v in the bytes of a word: the sum of 128 at every place turns them into ordinary
// bytes (no borrows), and the exclusive or takes 128 off each byte again.
__device__ __forceinline__ uint32_t digits3(int v) { return ((uint32_t)v + 0x00808080u) ^ 0x00808080u; }
__device__ __forceinline__ uint32_t digits4(int v) { return ((uint32_t)v + 0x80808080u) ^ 0x80808080u; }
// Bytes q of four words, in their order.
template <int Q>
__device__ __forceinline__ uint32_t gather_bytes(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    constexpr uint32_t lo = (uint32_t)Q | ((uint32_t)(4 + Q) << 4);
    return __byte_perm(__byte_perm(a, b, lo), __byte_perm(c, d, lo), 0x5410);
}

// Digit rows per part of a tile (192, 96 or 48).
inline long long tile_count(int a_rows, int b_rows, int n) { return (long long)ceil_div(a_rows, 2 * ROWS) * ceil_div(b_rows, PARTS * n / 3); }
// For `a_rows` x `b_rows` outputs of `steps` groups of 64 positions on `pairs` CTA pairs: the width with the least
// estimated time.  A launch takes ceil(tiles / pairs) turns of so many clocks per group and for an epilogue, by rows or (not of 48) by blocks; fitted to
// 74 launches of each width on B200 (16 .. 16384 rows x 500 .. 6000, 5 .. 56 groups), of which the choice takes 0.2 % more than the best width on the mean, 3 % at most.
// us, 192 / 96 / 48: 1461 x 1823, 7 groups 12.4 / 10.3 / 12.0; 4844 x 678, 8 groups 12.5 / 11.1 / 14.3; 8192 x 3400, 32 groups 74 / 88 / 158.
inline int tile_rows(int a_rows, int b_rows, int steps, int pairs, bool blocks) {
    constexpr struct { int n, clocks, by_rows, by_blocks; } widths[] = {{192, 215, 6300, 3300}, {96, 155, 3150, 1650}, {48, 142, 1900, 1900}};
    int best = 0;
    long long least = -1;
    for (const auto& s : widths) {
        const long long cost = (tile_count(a_rows, b_rows, s.n) + pairs - 1) / pairs * ((long long)steps * s.clocks + (blocks ? s.by_blocks : s.by_rows));
        if (least < 0 || cost < least) { least = cost; best = s.n; }
    }
    return best;
}

}  // namespace digit

}  // namespace bnn
