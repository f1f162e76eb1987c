// What the kernels that widen both operands as they go have in common (xnor_gemm_tc.cu on CTA pairs, xnor_gemm_cta.cu on single CTAs):
// a stage of a row, and a block of 32 x 32 results of an epilogue warp.
#pragma once

#include "bnn_common.cuh"
#include "tcgen05.cuh"
#include "xnor_widen.cuh"

namespace bnn {
namespace both {

using namespace tc;

// The rows of either operand: stages of 256 positions, words, valid bits of the last word.
struct Rows {
    int nks, kw;
    uint32_t tmask;
    __device__ __forceinline__ explicit Rows(int K) : nks(ceil_div(K, 256)), kw(words_for(K)), tmask(tail_mask(K)) {}
    __device__ __forceinline__ bool ragged() const { return kw % 8 != 0 || tmask != 0xFFFFFFFFu; }     // the last stage has positions >= K
    __device__ __forceinline__ int groups() const { return ceil_div(nks, 2); }                         // of two stages (an odd last stage has an empty partner)
};

// The eight 16-byte chunks of one widened row and stage; `ks` is the stage's index in the row.
// ZO: the row's bits stand for (0,1) instead of (-1,+1); RAGGED: the last stage has positions >= K, whose nibbles are set to +0 (in the
// unit rows; what the frame rows hold there then does not matter).
template <bool ZO, bool RAGGED>
__device__ __forceinline__ void widen_stage(const Rows& rows, int ks, const uint4& v0, const uint4& v1, uint4 (&o)[8]) {
    const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
    if (RAGGED && ks >= rows.nks - 1) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const int g = 8 * ks + c;   // index of the word in the row
            const uint32_t valid = g < rows.kw - 1 ? 0xFFFFFFFFu : (g == rows.kw - 1 ? rows.tmask : 0u);
            o[c] = widen_masked(w[c], valid);
        }
    } else {
#pragma unroll
        for (int c = 0; c < 8; ++c) o[c] = ZO ? widen01(w[c]) : widen(w[c]);
    }
}

// An epilogue warp's 32 frames x 32 units of integers, offset by kMagicBits, to C, from row m0 and column nb on.  `staging`: two blocks of 32 rows x 128 bytes (1024-byte
// aligned) of this warp's own, taken in turn.  first, last: of the blocks of a run of columns that this warp stores one after the other.
//
// Each thread parks its 32 integers (128 bytes of one output row) in shared memory, 16-byte
// chunk i at i ^ (row % 8).  One thread then has the 32 x 128-byte block stored, which goes on while
// the warp turns to the next 32 columns.  (Measured on B200: written by the warp with 16-byte stores,
// 8 lanes to a row, the epilogue took as long as 16 stages of MMAs.)
// A tile store clips a row to 16 bytes, not to elements, and wants an aligned pitch (tma_c).  Elsewhere the
// warp writes the block a row at a time, and each row from the 32-byte sector its first
// column lies in (from the block before) to the one of its last column, which is left to the next
// block: every store but those at the run's edges then covers whole sectors.  (4096 x 2048 x
// 4095, microseconds: a thread a row 102, rows of 32 columns 68, whole sectors 57; 4096 columns 29.)
__device__ __forceinline__ void store_block(uint32_t staging, int which, bool first, bool last, const int (&q)[32], const CUtensorMap* mapC, int tma_c,
                                            int32_t* C, int ldc, int M, int N, int m0, int nb, int lane) {
    const bool whole = tma_c && (nb + 31 < N || N % 4 == 0);
    const uint32_t blk = staging + (uint32_t)(which * 4096);
    if (lane == 0) bulk_wait_read<1>();      // the block's store of two rounds ago has read it
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 8; ++i)
        sts128(blk + lane * 128 + ((i ^ (lane & 7)) << 4), (uint32_t)(q[4 * i] - kMagicBits), (uint32_t)(q[4 * i + 1] - kMagicBits),
               (uint32_t)(q[4 * i + 2] - kMagicBits), (uint32_t)(q[4 * i + 3] - kMagicBits));
    if (whole) fence_proxy_async_smem();
    __syncwarp();
    if (whole) {
        if (lane == 0 && nb < N && m0 < M) tma_store_2d(mapC, nb, m0, blk);
    } else if (nb < N) {
        const int rows = M - m0 < 32 ? M - m0 : 32;
        const bool tail = last || nb + 32 >= N;             // the last block of this warp's row
        int32_t* dst = C + (size_t)m0 * ldc + nb;
        uint32_t at = (uint32_t)(reinterpret_cast<uintptr_t>(dst) >> 2);   // in words; its low bits count
#pragma unroll 4
        for (int r = 0; r < rows; ++r, dst += ldc, at += (uint32_t)ldc) {
            const int back = first ? 0 : (int)(at & 7u);        // columns of the block before that this store takes along
            const int lead = (int)(at & 7u) - back;             // the run's first block starts inside a sector
            const int col = lane - back - lead;                 // from -7 to 31
            const uint32_t buf = staging + (uint32_t)((which ^ (col < 0)) * 4096) + r * 128;
            const uint32_t v = lds32u(buf + ((((uint32_t)col >> 2) & 7u) ^ ((uint32_t)r & 7u)) * 16 + (col & 3) * 4);
            if (col >= -back && nb + col < N) dst[col] = (int32_t)v;
            if (tail) {
                const int rest = col + 32;                      // the columns that stay over
                const uint32_t t = lds32u(blk + r * 128 + ((((uint32_t)rest >> 2) & 7u) ^ ((uint32_t)r & 7u)) * 16 + (rest & 3) * 4);
                if (rest < 32 && nb + rest < N) dst[rest] = (int32_t)t;
            }
        }
    }
    if (lane == 0) bulk_commit();            // (an empty group keeps the count)
}

// The Sign bits of 32 such integers, given their thresholds + kMagicBits: bit j = (q[j] >= T[j]).  The sign bits of the differences are shifted in from the top, element 31
// first, so element j ends up in bit j, inverted.
__device__ __forceinline__ uint32_t sign_word(const int (&q)[32], const int* T) {
    uint32_t wd = 0u;
#pragma unroll
    for (int j = 31; j >= 0; --j) wd = __funnelshift_l((uint32_t)(q[j] - T[j]), wd, 1);
    return ~wd;
}

}  // namespace both
}  // namespace bnn
