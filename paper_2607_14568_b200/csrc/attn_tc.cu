// Causal softmax attention with grouped queries on the 5th-generation tensor core (sm_100a).
//
// Sections "The layout trick" and "Prefill attention: finding and removing the O(N^2) wall" of the
// paper turn the prefill attention of the softmax layers into matrix products: scores for a whole block of queries at once, a softmax that normalises
// the causally valid prefix and leaves exact zeros beyond it, a second product with V, and
// grouped queries by pointing several query heads at one key/value block.  The paper materialises
// the score matrix in a buffer it already owned; here a tile of scores lives only in tensor
// memory: a CTA takes 128 or 256 queries of one head and walks the key/value tiles up to its diagonal,
//
//   S  = Q K^T                      tcgen05.mma, both operands from shared memory (TMA, 128-B swizzle)
//   P  = 2^(S c - m), l += sum P    one thread per query row, straight out of tensor memory
//   O += P V                        tcgen05.mma, P read back from tensor memory as the A operand
//
// with the running maximum m only raised when it grew by more than 8 (so O in tensor memory is
// rescaled rarely; the final division by l uses the same m, so the result is exact).  Score tiles
// are double buffered in tensor memory, so the next Q K^T runs under the current softmax.
//
// Every wait is bounded (about a second): a waiter that gives up raises the CTA's abort flag and
// GDN_ERR_TIMEOUT in the status word; all roles then fall through their loops and the kernel ends.

#include <cuda.h>

#include "gdn_internal.h"
#include "sm100_ptx.cuh"

namespace gdn {

__device__ int g_attn_status = 0;

namespace {

using namespace ptx;

constexpr int BM = 128;                 // queries per tile (two tiles per work item, or one)
constexpr int BN = 128;                 // keys per tile
constexpr int HD = 128;                 // head dimension
constexpr int ATTN_THREADS = 320;       // warps 0-3 / 4-7: softmax of query tile A / B (thread = query), 8 MMA issue, 9 TMA
constexpr unsigned long long ATTN_TIMEOUT_NS = 1000000000ull;
constexpr float RESCALE_THRESHOLD = 8.f;   // in log2 units: P stays below 2^8

// tensor memory columns (512): scores of tile A and B (their bf16 probabilities overwrite the first
// 64 columns of the scores they came from), output accumulators of A and B
constexpr uint32_t TM_S = 0, TM_O = 256;
constexpr uint32_t AT_COLS = 512;

// shared memory: a tile is [2 halves of the head dimension][128 rows][64 values], 128-byte rows
constexpr uint32_t TILE_BYTES = 32768;
constexpr uint32_t AS_Q = 0, AS_K = 2 * TILE_BYTES, AS_V = 4 * TILE_BYTES;      // Q: A, B; K, V: two stages each
constexpr uint32_t AS_BARS = 6 * TILE_BYTES;
constexpr uint32_t AS_MISC = AS_BARS + 24 * 8;
constexpr uint32_t AS_TAKEN = AS_MISC + 48;
constexpr uint32_t AS_TOTAL = AS_MISC + 64;
constexpr uint32_t ATTN_SMEM = AS_TOTAL + 1024;

enum ABar : uint32_t { AB_Q = 0, AB_KFULL0 = 1, AB_KFREE0 = 3, AB_VFULL0 = 5, AB_VFREE0 = 7, AB_SFULL0 = 9 /* A, B */,
                       AB_PFULL0 = 11 /* A, B: first 64 keys */, AB_PVDONE0 = 13 /* A, B */, AB_PFULL1 = 15 /* A, B: other 64 */,
                       AB_QFREE = 17 /* Q tiles and item slot read */, AB_TAKEN = 18, AB_DRAIN = 19 };

struct AWaiter {
    uint32_t bars;
    volatile int* abort_flag;
    __device__ __forceinline__ uint32_t bar(uint32_t i) const { return bars + i * 8; }
    __device__ __forceinline__ void wait(uint32_t idx, uint32_t parity) const {
        const uint32_t b = bar(idx);
#pragma unroll 1
        for (int i = 0; i < 2048; ++i)
            if (mbar_try_wait(b, parity)) return;
        const unsigned long long t0 = globaltimer_ns();
        while (true) {
            if (mbar_try_wait_suspend(b, parity, 100000u)) return;
            if (*abort_flag) return;
            if (globaltimer_ns() - t0 > ATTN_TIMEOUT_NS) {
                *abort_flag = 1;
                atomicCAS(&g_attn_status, 0, (int)GDN_ERR_TIMEOUT);
                return;
            }
        }
    }
};

struct AttnParams {
    __nv_bfloat16* out;      // [B, T, Hq, 128], or packed [T, Hq, 128]
    const int32_t* cu;       // packed input: B + 1 sequence boundaries (device), else nullptr
    int B, T, Hq, Hkv;
    int per;                 // query tiles per work item: 2 (neighbours) or 1
    float scale_log2e;       // scale * log2(e)
};

constexpr uint32_t ID_QK = make_idesc(128, 128, kFmtBF16, kFmtBF16, kMajorK, kMajorK);
constexpr uint32_t ID_PV = make_idesc(128, 128, kFmtBF16, kFmtBF16, kMajorK, kMajorMN);

// A work item is two neighbouring query tiles A = 2t, B = 2t + 1 of one head.  Both read the same key
// and value tiles, and their softmax warpgroups alternate: while one turns its scores into
// probabilities, the tensor core runs P V and the next Q K^T of the other.  (Items of a single tile when
// there are few: the rule is at the launch.)
//
// The grid has one CTA per item, the longest items first.  A CTA that has issued its item's last copies takes the item of a
// CTA that has not started (which then never does), so every SM goes on to the longest item that is left, and the copies,
// first Q K^T and softmax of the next item run under the last softmax and the output of the current one; started as a
// CTA, each item left 5 us open.  16 heads: 6000 tokens 136 -> 124 us, 10240 tokens 400 -> 383 us at the power limit,
// packed 1711 + 402 + 2048 + 65 + 977 tokens 54 -> 43 us, eight packed prompts of 33 to 3000 tokens 84 -> 66 us (short runs; in a long
// alternation of builds the first packed case takes 50 us, 10240 tokens 390).  (One CTA per SM and the items dealt out back and forth in
// advance: 126, 383, 47, 75 us.)
// The copy warp looks the items up and publishes them in shared memory (item k in slot k & 1, barrier AB_Q; t < 0 is the
// end); a slot and the Q tiles are free again when the softmax warps have read the one and the tensor core the others
// (AB_QFREE).
__global__ void __launch_bounds__(ATTN_THREADS, 1)
attn_causal_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                   const __grid_constant__ CUtensorMap map_v, AttnParams p) {
    extern __shared__ uint8_t smem_raw[];
    const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* sm = smem_raw + (base - smem_u32(smem_raw));
    volatile uint32_t* sMisc = reinterpret_cast<volatile uint32_t*>(sm + AS_MISC);
    AWaiter w{base + AS_BARS, reinterpret_cast<volatile int*>(sm + AS_MISC + 4)};

    const int tid = threadIdx.x, warp = (int)warp_uniform(tid >> 5), lane = tid & 31;
    pdl_trigger();                      // a following kernel of this library may set itself up as SMs come free
    struct Item {
        int tok0, len, t, h, nA, nB, ntiles;
        bool hasB;
    };
    auto shape = [&](Item& it) {                           // what follows from the sequence and the index
        const int nqt = (it.len + BM - 1) / BM;
        it.hasB = p.per == 2 && 2 * it.t + 1 < nqt;
        it.nA = p.per * it.t + 1;                          // key tiles of A: 0 .. (the last is its diagonal)
        it.nB = it.hasB ? it.nA + 1 : 0;
        it.ntiles = it.hasB ? it.nB : it.nA;
    };
    auto fetch = [&](int k, Item& it) -> bool {            // item k as the copy warp published it; false at the end
        w.wait(AB_Q, k & 1);
        volatile uint32_t* m = sMisc + 4 + 4 * (k & 1);
        it.tok0 = (int)m[0]; it.len = (int)m[1]; it.t = (int)m[2]; it.h = (int)m[3];
        // (a whole warp leaves or none of its lanes: the flag may rise between two lanes' reads of it)
        if (__any_sync(0xffffffffu, it.t < 0 || *w.abort_flag)) return false;
        shape(it);
        return true;
    };

    // Items are numbered (y, x): x over heads (and sequences of one length), y from the last index of the longest sequence
    // down, over all sequences.  Packed: items with an index of at least i are sum max(0, count - i); the largest i with more
    // than y of them is the index of y, and its sequence follows from y's rank among the sequences that have it.  One warp does
    // this together (400 sequences of 64 tokens: 4.6 ms with a thread alone, 0.21 ms).
    const int span = p.per * BM;
    int first = 0;                                         // items of sequence `lane`: the first 32 are read once
    int most = 0, ny = (p.T + span - 1) / span;            // items of the longest sequence, items of one head
    auto count_of = [&](int n) { return n < 32 ? first : (p.cu[n + 1] - p.cu[n] + span - 1) / span; };
    auto at_least = [&](int i) {
        int sum = max(0, first - i);
        for (int n = lane + 32; n < p.B; n += 32) sum += max(0, count_of(n) - i);
        return (int)__reduce_add_sync(0xffffffffu, sum);
    };
    auto find = [&](uint32_t i, Item& it) {                // item i, t < 0 if there are not that many
        const uint32_t X = p.cu ? p.Hq : p.Hq * p.B;
        const int y = (int)(i / X), x = (int)(i - y * X);
        it.t = -1;
        if (y >= ny) return;
        it.h = x % p.Hq;
        if (p.cu) {
            int lo = 0, hi = most;                         // at_least(lo) > y >= at_least(hi)
            while (hi - lo > 1) {
                const int mid = (lo + hi) >> 1;
                if (at_least(mid) > y) lo = mid; else hi = mid;
            }
            it.t = lo;
            int rank = y - at_least(lo + 1);
            for (int n0 = 0; n0 < p.B; n0 += 32) {
                const int n = n0 + lane;
                const bool has = n < p.B && count_of(n) > lo;
                const unsigned those = __ballot_sync(0xffffffffu, has);
                const unsigned me = __ballot_sync(0xffffffffu, has && __popc(those & ((1u << lane) - 1u)) == rank);
                if (me) {
                    const int c = n0 + __ffs(me) - 1;
                    it.tok0 = p.cu[c];
                    it.len = p.cu[c + 1] - it.tok0;
                    break;
                }
                rank -= __popc(those);
            }
        } else {
            it.tok0 = (x / p.Hq) * p.T;
            it.len = p.T;
            it.t = ny - 1 - y;
        }
        shape(it);
    };
    Item it{};
    if (warp == 9 && !p.cu) find(blockIdx.x, it);                   // the first one under the setup

    if (tid == 0) {
        mbar_init(w.bar(AB_Q), 1); mbar_init(w.bar(AB_TAKEN), 1); mbar_init(w.bar(AB_DRAIN), 1);
        mbar_init(w.bar(AB_QFREE), 9);                     // 8 softmax warps and the tensor core
        for (uint32_t s = 0; s < 2; ++s) {
            mbar_init(w.bar(AB_KFULL0 + s), 1); mbar_init(w.bar(AB_KFREE0 + s), 1);
            mbar_init(w.bar(AB_VFULL0 + s), 1); mbar_init(w.bar(AB_VFREE0 + s), 1);
            mbar_init(w.bar(AB_SFULL0 + s), 1); mbar_init(w.bar(AB_PFULL0 + s), 128); mbar_init(w.bar(AB_PFULL1 + s), 128);
            mbar_init(w.bar(AB_PVDONE0 + s), 1);
        }
        sMisc[1] = 0;
        fence_mbar_init();
    }
    if (warp == 0) {
        tmem_alloc(base + AS_MISC, AT_COLS);
        tmem_relinquish();
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = sMisc[0];
    pdl_wait();                         // the inputs, and the buffer of the outputs, belong to what ran before

    if (warp < 8) {
        // =========================== softmax: thread = query row ===========================
        const uint32_t X = warp >> 2;                      // 0 = tile A, 1 = tile B
        const int r = tid & 127;                           // row inside the tile = tensor-memory lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t ts = tmem + lane_base + TM_S + X * 128, to = tmem + lane_base + TM_O + X * 128;
        const float c = p.scale_log2e;
        uint32_t tiles = 0, outs = 0;                      // of this warpgroup, over all items (barrier phases)
        for (int k = 0; fetch(k, it); ++k) {
            __syncwarp();
            if (lane == 0) mbar_arrive(w.bar(AB_QFREE));   // the slot has been read
            const int nX = X ? it.nB : it.nA, qt = p.per * it.t + (int)X;
            if (nX == 0) continue;
            float m_ref = -INFINITY, l = 0.f;
            for (int j = 0; j < nX; ++j, ++tiles) {
                // S_X of tile j is complete; so is every earlier MMA of the issuing thread (P V of tile j - 1)
                w.wait(AB_SFULL0 + X, tiles & 1);
                tc_fence_after_sync();
                // row maximum of the raw scores (c >= 0, so max(c s) = c max(s)); the scores stay in registers
                float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
                uint32_t x[4][32];
                tmem_ld32(ts, x[0]);
                tmem_ld32(ts + 32, x[1]);
                tmem_wait_ld();
                tmem_ld32(ts + 64, x[2]);
                tmem_ld32(ts + 96, x[3]);
    #pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    if (q4 == 2) tmem_wait_ld();
                    if (j == qt) {                             // diagonal tile: keys after the query do not count
    #pragma unroll
                        for (int i = 0; i < 32; ++i)
                            if (32 * q4 + i > r) x[q4][i] = 0xff800000u;           // -inf
                    }
    #pragma unroll
                    for (int i = 0; i < 32; i += 2)
                        mx4[(i >> 1) & 3] = max3(mx4[(i >> 1) & 3], __uint_as_float(x[q4][i]), __uint_as_float(x[q4][i + 1]));
                }
                const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3])) * c;
                // raise the reference maximum only when it is first set or has grown by more than 2^8
                const bool grow = (mx > m_ref + RESCALE_THRESHOLD);
                const float m_new = grow ? mx : m_ref;
                const float alpha = grow ? ex2(m_ref - m_new) : 1.f;           // 0 on the first tile (m_ref = -inf)
                m_ref = m_new;
                if (j > 0 && __any_sync(0xffffffffu, grow)) {   // rescale the accumulator rows of this warp (P V of tile j - 1 is complete)
    #pragma unroll 1
                    for (int q4 = 0; q4 < 8; ++q4) {
                        uint32_t o[16];
                        tmem_ld16(to + 16 * q4, o);
                        tmem_wait_ld();
    #pragma unroll
                        for (int i = 0; i < 16; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
                        tmem_st16(to + 16 * q4, o);
                    }
                }
                // P = 2^(c s - m) as bf16 over the first 64 columns of the scores it came from.  The first 64 keys are handed
                // over while the others are worked on, so that half of P V runs under the second half of the softmax.
                // (masked scores are -inf: exact zeros after the query's own position)
                float sum[4] = {0.f, 0.f, 0.f, 0.f};
    #pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                    uint32_t pk[16];
    #pragma unroll
                    for (int i = 0; i < 16; ++i) {
                        const float p0 = ex2(fmaf(__uint_as_float(x[q4][2 * i]), c, -m_new));
                        const float p1 = ex2(fmaf(__uint_as_float(x[q4][2 * i + 1]), c, -m_new));
                        sum[i & 1] += p0;
                        sum[2 + (i & 1)] += p1;
                        pk[i] = pack_bf16(p0, p1);
                    }
                    tmem_st16(ts + 16 * q4, pk);
                    if (q4 & 1) {
                        tmem_wait_st();
                        tc_fence_before_sync();
                        mbar_arrive(w.bar((q4 == 1 ? AB_PFULL0 : AB_PFULL1) + X));
                    }
                }
                l = l * alpha + ((sum[0] + sum[1]) + (sum[2] + sum[3]));
            }
            // ---- epilogue: O / l -> bf16 -> global (one 256-byte row per thread) ----
            w.wait(AB_PVDONE0 + X, outs & 1);
            ++outs;
            tc_fence_after_sync();
            const float inv = 1.0f / l;
            const int row = qt * BM + r;
            __nv_bfloat16* dst = p.out + ((size_t)(it.tok0 + row) * p.Hq + it.h) * HD;
#pragma unroll
            for (int q4 = 0; q4 < 4; ++q4) {
                uint32_t o[32];
                tmem_ld32(to + 32 * q4, o);
                tmem_wait_ld();
                if (row < it.len) {
#pragma unroll
                    for (int cc = 0; cc < 4; ++cc) {
                        uint4 val;
                        val.x = pack_bf16(__uint_as_float(o[8 * cc + 0]) * inv, __uint_as_float(o[8 * cc + 1]) * inv);
                        val.y = pack_bf16(__uint_as_float(o[8 * cc + 2]) * inv, __uint_as_float(o[8 * cc + 3]) * inv);
                        val.z = pack_bf16(__uint_as_float(o[8 * cc + 4]) * inv, __uint_as_float(o[8 * cc + 5]) * inv);
                        val.w = pack_bf16(__uint_as_float(o[8 * cc + 6]) * inv, __uint_as_float(o[8 * cc + 7]) * inv);
                        *reinterpret_cast<uint4*>(dst + 32 * q4 + 8 * cc) = val;
                    }
                }
            }
        }
    } else if (warp == 8) {
        // =========================== MMA issue (one elected thread) ===========================
        {
            const uint32_t tmem = warp_uniform(sMisc[0]);
            const bool lead = elect_one();
            // operand descriptors are built once: issuing costs tens of nanoseconds per instruction and
            // sits on each tile's softmax -> P V -> Q K^T chain
            const uint64_t dq0 = make_smem_desc(base + AS_Q, 16, 1024), dk0 = make_smem_desc(base + AS_K, 16, 1024);
            const uint64_t dv0 = make_smem_desc(base + AS_V, 16384, 1024);
            // kt: key/value tile, counted over all items of the CTA (stage kt & 1); pt: tile of warpgroup X likewise
            auto issue_qk = [&](uint32_t X, uint32_t kt) {       // S_X = Q_X K^T
                const uint64_t dq = dq0 + ((uint64_t)(X * TILE_BYTES) >> 4), dk = dk0 + ((uint64_t)((kt & 1) * TILE_BYTES) >> 4);
#pragma unroll
                for (uint32_t ks = 0; ks < 8; ++ks) {
                    const uint64_t off = ((ks >> 2) * 16384 + (ks & 3) * 32) >> 4;   // the address field counts 16 bytes
                    if (lead) mma_ss(tmem + TM_S + X * 128, dq + off, dk + off, ID_QK, ks > 0);
                }
                if (lead) mma_commit(w.bar(AB_SFULL0 + X));
            };
            auto issue_pv = [&](uint32_t X, uint32_t kt, uint32_t pt, bool first) {   // O_X += P_X V, 16 keys per step, each half when its P is there
                const uint64_t dv = dv0 + ((uint64_t)((kt & 1) * TILE_BYTES) >> 4);
                w.wait(AB_PFULL0 + X, pt & 1);
                tc_fence_after_sync();
#pragma unroll
                for (uint32_t ks = 0; ks < 8; ++ks) {
                    if (ks == 4) {
                        w.wait(AB_PFULL1 + X, pt & 1);
                        tc_fence_after_sync();
                    }
                    if (lead) mma_ts(tmem + TM_O + X * 128, tmem + TM_S + X * 128 + ks * 8, dv + ((ks * 2048) >> 4), ID_PV,
                           (!first || ks > 0) ? 1u : 0u);
                }
            };
            uint32_t kt = 0, pa = 0, pb = 0;
            for (int k = 0; fetch(k, it); ++k) {
                __syncwarp();                              // every lane has read the slot before the lead can free it
                // the scores of the previous item have been read by its P V, issued before; its outputs are read before a warpgroup
                // hands over the first P of this one
                w.wait(AB_KFULL0 + (kt & 1), (kt >> 1) & 1);
                tc_fence_after_sync();
                issue_qk(0, kt);
                if (it.hasB) issue_qk(1, kt);
                if (lead) mma_commit(w.bar(AB_KFREE0 + (kt & 1)));
                if (it.ntiles == 1 && lead) mma_commit(w.bar(AB_QFREE));
                for (int j = 0; j < it.ntiles; ++j, ++kt) {
                    const uint32_t s = kt & 1, s1 = (kt + 1) & 1;
                    const bool more = (j + 1 < it.ntiles);
                    // the tiles are normally there long before the probabilities: these waits come first, so that
                    // nothing but the MMAs sits between "P ready" and "next scores ready"
                    w.wait(AB_VFULL0 + s, (kt >> 1) & 1);
                    if (more) {
                        w.wait(AB_KFULL0 + s1, ((kt + 1) >> 1) & 1);
                    } else if (it.ntiles * BN > it.len) {
                        // The last key tile is completed with the rows that follow the sequence in memory.  Their probabilities are
                        // zero, but zero times what is not finite is not zero: the value rows are cleared before P V of the tile
                        // (by this warp, which has the time of a softmax for it; in the softmax it cost 0.7 % on every call)
                        uint32_t row = (uint32_t)(it.len & (BN - 1)) + (lane >> 4);       // two rows of 256 bytes at a time
                        uint32_t dst = base + AS_V + s * TILE_BYTES + ((lane >> 3) & 1) * 16384 + row * 128 + (lane & 7) * 16;
#pragma unroll 4
                        for (; row < BN; row += 2, dst += 256)
                            asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0u) : "memory");
                        fence_proxy_async_smem();
                        __syncwarp();
                    }
                    if (j < it.nA) {
                        issue_pv(0, kt, pa++, j == 0);
                        if (j + 1 < it.nA) {
                            issue_qk(0, kt + 1);
                        } else {
                            if (lead) mma_commit(w.bar(AB_PVDONE0 + 0));
                        }
                    }
                    if (it.hasB) {
                        issue_pv(1, kt, pb++, j == 0);
                        if (more) {
                            issue_qk(1, kt + 1);
                        } else {
                            if (lead) mma_commit(w.bar(AB_PVDONE0 + 1));
                        }
                    }
                    if (lead) mma_commit(w.bar(AB_VFREE0 + s));
                    if (more && lead) mma_commit(w.bar(AB_KFREE0 + s1));
                    if (j + 2 == it.ntiles && lead) mma_commit(w.bar(AB_QFREE));      // the last Q K^T of the item is issued
                }
            }
            if (__any_sync(0xffffffffu, *w.abort_flag != 0)) {     // nobody may be waiting for the products in flight: they end first (bounded)
                if (lead) mma_commit(w.bar(AB_DRAIN));
#pragma unroll 1
                for (int i = 0; i < 1024 && !mbar_try_wait_suspend(w.bar(AB_DRAIN), 0, 1000000u); ++i) {}
            }
        }
    } else {
        // =========================== items (the warp) and TMA producer (its first lane) ===========================
        if (lane == 0) {
            prefetch_tensormap(&map_q);
            prefetch_tensormap(&map_k);
            prefetch_tensormap(&map_v);
        }
        auto load_tile = [&](uint32_t dst, const CUtensorMap* map, int head, int tok, uint32_t full) {
            tma_load_3d(dst, map, 0, head, tok, full);
            tma_load_3d(dst + 8192, map, 0, head, tok + 64, full);
            tma_load_3d(dst + 16384, map, 64, head, tok, full);
            tma_load_3d(dst + 24576, map, 64, head, tok + 64, full);
        };
        if (p.cu) {
            if (lane < p.B) first = (p.cu[lane + 1] - p.cu[lane] + span - 1) / span;
            most = first;
            for (int n = lane + 32; n < p.B; n += 32) most = max(most, count_of(n));
            most = (int)__reduce_max_sync(0xffffffffu, most);
            ny = at_least(0);
            find(blockIdx.x, it);
        }
        uint32_t kt = 0;
        int q_loads = 0, asked = 0;
        auto next = [&](Item& it) {
            do {
                uint32_t i = ~0u;
                if (lane == 0) {
                    fence_proxy_async_smem();              // (the previous answer has been read)
                    mbar_arrive_expect_tx(w.bar(AB_TAKEN), 16);
                    take_pending_cta(base + AS_TAKEN, w.bar(AB_TAKEN));
                    w.wait(AB_TAKEN, asked & 1);
                    if (*w.abort_flag == 0) i = taken_cta_x(base + AS_TAKEN);
                }
                ++asked;
                i = warp_uniform(i);
                it.t = -1;
                if (i == ~0u) return;
                find(i, it);
            } while (it.t < 0);
        };
        for (int k = 0;; ++k) {
            if (k > 0) next(it);                           // under the last two rounds of item k - 1
            if (lane == 0) {
                if (k > 0) w.wait(AB_QFREE, (k - 1) & 1);
                volatile uint32_t* m = sMisc + 4 + 4 * (k & 1);
                m[0] = (uint32_t)it.tok0; m[1] = (uint32_t)it.len; m[2] = (uint32_t)it.t; m[3] = (uint32_t)it.h;
                if (it.t < 0) {
                    mbar_arrive(w.bar(AB_Q));
                } else if (*w.abort_flag == 0) {
                    const int tok_q = it.tok0 + it.t * span, hk = it.h / (p.Hq / p.Hkv);   // the key/value head this query head reads
                    mbar_arrive_expect_tx(w.bar(AB_Q), it.hasB ? 2 * TILE_BYTES : TILE_BYTES);
                    load_tile(base + AS_Q, &map_q, it.h, tok_q, w.bar(AB_Q));
                    if (it.hasB) load_tile(base + AS_Q + TILE_BYTES, &map_q, it.h, tok_q + BM, w.bar(AB_Q));
                    for (int j = 0; j < it.ntiles; ++j, ++kt) {
                        const uint32_t s = kt & 1, free_parity = ((kt >> 1) - 1) & 1;
                        const int tok = it.tok0 + j * BN;
                        if (kt >= 2) w.wait(AB_KFREE0 + s, free_parity);
                        mbar_arrive_expect_tx(w.bar(AB_KFULL0 + s), TILE_BYTES);
                        load_tile(base + AS_K + s * TILE_BYTES, &map_k, hk, tok, w.bar(AB_KFULL0 + s));
                        if (kt >= 2) w.wait(AB_VFREE0 + s, free_parity);
                        mbar_arrive_expect_tx(w.bar(AB_VFULL0 + s), TILE_BYTES);
                        load_tile(base + AS_V + s * TILE_BYTES, &map_v, hk, tok, w.bar(AB_VFULL0 + s));
                    }
                    q_loads = k + 1;
                }
            }
            if (__any_sync(0xffffffffu, it.t < 0 || *w.abort_flag)) break;
        }
        if (lane == 0 && *w.abort_flag) {
            // let copies in flight land before shared memory is released (bounded)
            const unsigned long long t0 = globaltimer_ns();
            while (q_loads > 0 && !mbar_try_wait(w.bar(AB_Q), (q_loads - 1) & 1) && globaltimer_ns() - t0 < ATTN_TIMEOUT_NS) {}
            while (asked > 0 && !mbar_try_wait(w.bar(AB_TAKEN), (asked - 1) & 1) && globaltimer_ns() - t0 < ATTN_TIMEOUT_NS) {}
            for (uint32_t x = kt >= 2 ? kt - 2 : 0; x < kt; ++x)
                for (uint32_t which = 0; which < 2; ++which)
                    while (!mbar_try_wait(w.bar((which ? AB_VFULL0 : AB_KFULL0) + (x & 1)), (x >> 1) & 1) &&
                           globaltimer_ns() - t0 < ATTN_TIMEOUT_NS) {}
        }
    }
    tc_fence_before_sync();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after_sync();
        tmem_dealloc(tmem, AT_COLS);
    }
}

}  // namespace

bool attn_supported(int Hq, int Hkv, int d) { return d == HD && Hkv > 0 && Hq > 0 && Hq % Hkv == 0; }

int attn_status_async(int* host_dst, cudaStream_t stream) {
    return cudaMemcpyFromSymbolAsync(host_dst, g_attn_status, sizeof(int), 0, cudaMemcpyDeviceToHost, stream) == cudaSuccess
               ? GDN_OK : GDN_ERR_CUDA;
}

int attn_query_status() {
    int st = 0;
    if (cudaMemcpyFromSymbol(&st, g_attn_status, sizeof(int)) != cudaSuccess) return GDN_ERR_CUDA;
    return st;
}

int launch_attn(const void* q, const void* k, const void* v, void* out, const int32_t* cu_seqlens, int B, int T,
                int Hq, int Hkv, int d, float scale, cudaStream_t stream) {
    if (!attn_supported(Hq, Hkv, d)) return GDN_ERR_UNSUPPORTED;
    if (B > 65535 || T / (2 * BM) + B + 1 > 65535) return GDN_ERR_UNSUPPORTED;      // (the range accepted; the grid below would take more)
    if (B == 0 || T == 0) return GDN_OK;
    const uint64_t tokens = cu_seqlens ? (uint64_t)T : (uint64_t)B * T;
    if (tokens > 0x7fffffffull) return GDN_ERR_TOO_LARGE;
    CUtensorMap mq, mk, mv;
    if (!tc_make_map(&mq, q, tokens, Hq, d) || !tc_make_map(&mk, k, tokens, Hkv, d) ||
        !tc_make_map(&mv, v, tokens, Hkv, d))
        return GDN_ERR_CUDA;
    // masked scores are -inf, which a factor of zero would turn into NaN: the smallest normal number stands for zero (every
    // 2^(c s - m) is 1 with it)
    const float c = scale * 1.4426950408889634f;
    AttnParams p{static_cast<__nv_bfloat16*>(out), cu_seqlens, B, T, Hq, Hkv, 2, c > 1.17549435e-38f ? c : 1.17549435e-38f};
    const int sms = sm_count();
    if (sms <= 0) return GDN_ERR_CUDA;
    // Single tiles while they are fewer than two per SM: a round of one tile takes 1.5 us, of a pair 1.76 us, so halving the
    // longest item pays as long as no SM gets more than about its length (16 heads: 1024 tokens 19.2 -> 16.4 us, 2304 tokens 38.4 -> 34.4;
    // 3000 tokens, 384 single tiles: 48 -> 66 us with a CTA each).  Packed: sum over sequences of ceil(len / span) <= T / span + B.
    auto items_of = [&](int per) {
        const int span = per * BM;
        return cu_seqlens ? (long long)Hq * (T / span + B) : (long long)Hq * B * ((T + span - 1) / span);
    };
    p.per = items_of(1) < 2ll * sms ? 1 : 2;
    const long long items = items_of(p.per);
    if (items > 0x7fffffffll) return GDN_ERR_TOO_LARGE;
    const dim3 grid((unsigned)items);
    if (cudaFuncSetAttribute(attn_causal_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ATTN_SMEM) !=
        cudaSuccess)
        return GDN_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(ATTN_THREADS);
    cfg.dynamicSmemBytes = ATTN_SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, attn_causal_kernel, mq, mk, mv, p);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_CUDA;
}

}  // namespace gdn
