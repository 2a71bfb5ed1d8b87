// fp32-arithmetic chunked gated delta-rule prefill (plain FMA, no tensor cores).
//
// One cluster of eight CTAs walks the chunks of one (sequence, head) chain for a group of up to 128 value
// columns.  Per 64-token chunk it evaluates the chunked scan (Section "A chunked delta-rule scan for the
// recurrent layers") in fp32:
//   a   g_r = sum_{i<=r} log_alpha_i                       (warp scan)
//   b1  A[r,i] = beta_r e^{g_r-g_i} (k_r.k_i), i <  r
//       P[r,i] =        e^{g_r-g_i} (q_r.k_i), i <= r
//   b2  Tm = (I + A)^{-1}: forward substitution of the 16x16 diagonal blocks, then block merges
//   c   v_new = Tm diag(beta) (V - diag(e^g) K S) ;  S <- e^{g_C} S + sum_i e^{g_C-g_i} k_i v_new_i^T
//   d   O = diag(e^g) Q S + P v_new            (S = the chunk's incoming state)
// Steps a and b do not depend on the state, so the cluster does them for eight chunks at once, one chunk per
// CTA (the results stay in that CTA's shared memory).  Steps c and d then walk these chunks with the
// value columns split over the CTAs: a CTA keeps the state of its dv/8 columns in shared memory and fetches Tm, P
// and the gate vectors of each chunk from the CTA that made them, through distributed shared memory, one
// chunk ahead in registers.  No scratch in global memory is needed, which this entry point has none of.
//
// What bounds it: fp32 FMAs of one SM (about 460 k multiply-adds per chunk and CTA at d_k = d_v = 128, 3600
// cycles at full rate) and the shared-memory loads that feed them (six 16-byte loads per 32 FMAs).  The form
// v_new = Tm (V - K S) needs neither W nor U, so what a CTA fetches per chunk is 34 KiB instead of 66 KiB.
// Measured on a B200 (2048 tokens, 16 heads, d = 128): 324 us against 2480 us; 256 tokens, 2 heads, d = 64: 32 us against 256 us.  Before, one
// CTA per 32 value columns did every step of every chunk itself.
//
// Rows past the end of a sequence are identity tokens (beta = 0, log_alpha = 0,
// k = q = v = 0): they change nothing and are never stored.
//
// This kernel serves fp32 inputs (the paper's precision) and doubles as a slow
// cross-check of the tensor-core kernel for bf16 inputs.

#include <mutex>

#include "gdn_internal.h"
#include "sm100_ptx.cuh"

namespace gdn {
namespace {

constexpr int C = kChunk;   // 64
constexpr int NT = 256;     // threads per CTA
constexpr int LDT = C + 4;  // row stride of the 64x64 matrices and of the transposed slices (float4 reads without conflicts)

// What steps a, b leave behind for one chunk: Tm, P, then beta, e^g, e^{gC-g} and g.
constexpr int BK_T = 0, BK_P = C * LDT, BK_BETA = 2 * C * LDT, BK_EG = BK_BETA + C, BK_EC = BK_EG + C, BK_G = BK_EC + C;
constexpr int BK_FLOATS = BK_G + C;

struct SimtParams {
    const void* q;
    const void* k;
    const void* v;
    const float* a;
    const float* beta;
    const float* s0;
    void* out;
    float* sT;
    const int32_t* cu;
    int B, T, H, dk, dv;
};

// Two fp32 values in one 64-bit register; fma2 is two independent IEEE fused multiply-adds in one instruction (half the
// issue slots: this kernel issues as many loads and address steps as it issues FMAs).
typedef unsigned long long f2;
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ f2 pack2(float x, float y) {
    f2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
    return d;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
    float2 r;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
    return r;
}
__device__ __forceinline__ float sum2(f2 v) { const float2 r = unpack2(v); return r.x + r.y; }
// four consecutive elements of a shared-memory tile, widened
struct F4 { f2 lo, hi; };
__device__ __forceinline__ F4 load4(const float* p) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
    return F4{v.x, v.y};
}
__device__ __forceinline__ F4 load4(const __nv_bfloat16* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    return F4{pack2(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u)),
              pack2(__uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u))};
}
// dot product of four pairs onto a two-lane accumulator (its halves are added at the end)
__device__ __forceinline__ f2 dot4(const F4& a, const F4& b, f2 c) { return fma2(a.hi, b.hi, fma2(a.lo, b.lo, c)); }
__device__ __forceinline__ float load1(const float* p) { return *p; }
__device__ __forceinline__ float load1(const __nv_bfloat16* p) { return __bfloat162float(*p); }
__device__ __forceinline__ void store1(float* p, float x) { *p = x; }
__device__ __forceinline__ void store1(__nv_bfloat16* p, float x) { *p = __float2bfloat16_rn(x); }
// asynchronous copy global -> shared of BYTES (8 or 16); zero fill when !valid (the source is then not read)
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool valid) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(valid ? BYTES : 0) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void half_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the address, in CTA `rank` of the cluster, of this CTA's shared-memory location p
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(static_cast<uint32_t>(__cvta_generic_to_shared(p))), "r"(rank));
    return r;
}
__device__ __forceinline__ float4 load4_peer(uint32_t addr) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
    return v;
}

template <typename TIO>
__host__ __device__ constexpr int tile_ld(int dk) { return dk + 16 / (int)sizeof(TIO); }   // K, Q rows: 16 bytes of padding
template <typename TIO>
__host__ __device__ constexpr size_t tile_bytes(int dk) { return (size_t)C * tile_ld<TIO>(dk) * sizeof(TIO); }
template <typename TIO, int NC>
constexpr size_t simt_smem(int dk) {
    return 3 * tile_bytes<TIO>(dk) + 2 * BK_FLOATS * sizeof(float) + (size_t)NC * (dk + 4) * sizeof(float) +
           3 * (size_t)NC * LDT * sizeof(float) + 2 * (size_t)C * NC * sizeof(TIO);
}
static_assert(simt_smem<float, 16>(128) <= 232448, "shared memory per CTA");

// Steps a and b of one chunk by one CTA; K and Q tiles in shared memory, results in `blk`.  `tmp`: 1056 floats.
template <typename TIO>
__device__ __forceinline__ void prepare_chunk(const TIO* sK, const TIO* sQ, float* blk, float* tmp, const float* ga, const float* gb,
                                              size_t gstride, int R, int dk) {
    const int tid = threadIdx.x, lane = tid & 31;
    const int ld = tile_ld<TIO>(dk);
    if (tid < 32) {   // step a: chunk-local cumulative log gate
        const int r0 = lane, r1 = lane + 32;
        float x = 0.f, y = 0.f, b0 = 0.f, b1 = 0.f;
        if (r0 < R) { x = ga[r0 * gstride]; b0 = gb[r0 * gstride]; }
        if (r1 < R) { y = ga[r1 * gstride]; b1 = gb[r1 * gstride]; }
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const float xu = __shfl_up_sync(0xffffffffu, x, d);
            const float yu = __shfl_up_sync(0xffffffffu, y, d);
            if (lane >= d) { x += xu; y += yu; }
        }
        y += __shfl_sync(0xffffffffu, x, 31);
        const float gC = __shfl_sync(0xffffffffu, y, 31);
        blk[BK_G + r0] = x; blk[BK_G + r1] = y;
        blk[BK_BETA + r0] = b0; blk[BK_BETA + r1] = b1;
        blk[BK_EG + r0] = expf(x); blk[BK_EG + r1] = expf(y);
        blk[BK_EC + r0] = expf(gC - x); blk[BK_EC + r1] = expf(gC - y);
    }
    cp_async_wait();
    __syncthreads();
    float* sT = blk + BK_T;
    float* sP = blk + BK_P;
    {
        // step b1: thread (tr, ti) owns entries (tr + 16x, ti + 16y), y <= x: every thread has the same share of the
        // lower triangle, and neighbouring lanes read neighbouring rows (no bank conflicts)
        const int tr = tid >> 4, ti = tid & 15;
        f2 acc[4][4], accp[4][4];
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y < 4; ++y) { acc[x][y] = 0; accp[x][y] = 0; }
#pragma unroll 2
        for (int m = 0; m < dk; m += 4) {
            F4 kr[4], qr[4], ki[4];
#pragma unroll
            for (int x = 0; x < 4; ++x) {
                kr[x] = load4(sK + (tr + 16 * x) * ld + m);
                qr[x] = load4(sQ + (tr + 16 * x) * ld + m);
                ki[x] = load4(sK + (ti + 16 * x) * ld + m);
            }
#pragma unroll
            for (int x = 0; x < 4; ++x)
#pragma unroll
                for (int y = 0; y <= x; ++y) {
                    acc[x][y] = dot4(kr[x], ki[y], acc[x][y]);
                    accp[x][y] = dot4(qr[x], ki[y], accp[x][y]);
                }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
            for (int y = 0; y <= x; ++y) {
                const int r = tr + 16 * x, i = ti + 16 * y;
                const float e = (i <= r) ? expf(blk[BK_G + r] - blk[BK_G + i]) : 0.f;   // mask before exp is used
                sT[r * LDT + i] = (i < r) ? blk[BK_BETA + r] * e * sum2(acc[x][y]) : 0.f;
                sP[r * LDT + i] = (i <= r) ? e * sum2(accp[x][y]) : 0.f;
            }
        sT[tr * LDT + 16 + ti] = 0.f;                     // 16-blocks (0,1) and (2,3): the merges read them as part of a 32-block
        sT[(32 + tr) * LDT + 48 + ti] = 0.f;
    }
    __syncthreads();
    // step b2, level 0: the four 16x16 diagonal blocks, one column per thread
    float xs[16];
    if (tid < C) {
        const float* Ab = sT + (tid & 48) * LDT + (tid & 48);
        const int cc = tid & 15;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int i4 = 0; i4 < (r + 3) / 4; ++i4) {
                const float4 a4 = *reinterpret_cast<const float4*>(Ab + r * LDT + 4 * i4);
                if (4 * i4 + 0 < r) a0 = fmaf(a4.x, xs[4 * i4 + 0], a0);
                if (4 * i4 + 1 < r) a1 = fmaf(a4.y, xs[4 * i4 + 1], a1);
                if (4 * i4 + 2 < r) a0 = fmaf(a4.z, xs[4 * i4 + 2], a0);
                if (4 * i4 + 3 < r) a1 = fmaf(a4.w, xs[4 * i4 + 3], a1);
            }
            xs[r] = ((r == cc) ? 1.f : 0.f) - (a0 + a1);
        }
    }
    __syncthreads();
    if (tid < C) {
        float* Tb = sT + (tid & 48) * LDT + (tid & 48) + (tid & 15);
#pragma unroll
        for (int r = 0; r < 16; ++r) Tb[r * LDT] = xs[r];
    }
    __syncthreads();
    // level 1: blocks (1,0) and (3,2): T21 = -T22 (A21 T11), 16x16; two neighbouring columns per thread
    {
        const int lo = (tid >> 7) * 32, hi = lo + 16, r = (tid & 127) >> 3, c = (tid & 7) * 2;
        float* z = tmp + (tid >> 7) * 16 * 18;
        float2 s = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float a = sT[(hi + r) * LDT + lo + i];
            const float2 t = *reinterpret_cast<const float2*>(sT + (lo + i) * LDT + lo + c);
            s.x = fmaf(a, t.x, s.x); s.y = fmaf(a, t.y, s.y);
        }
        *reinterpret_cast<float2*>(z + r * 18 + c) = s;
        __syncthreads();
        s = make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const float a = sT[(hi + r) * LDT + hi + i];
            const float2 t = *reinterpret_cast<const float2*>(z + i * 18 + c);
            s.x = fmaf(a, t.x, s.x); s.y = fmaf(a, t.y, s.y);
        }
        *reinterpret_cast<float2*>(sT + (hi + r) * LDT + lo + c) = make_float2(-s.x, -s.y);
    }
    __syncthreads();
    // level 2: block (1,0) of the 32-blocks; four neighbouring columns per thread
    {
        const int r = tid >> 3, c = (tid & 7) * 4;
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
            const float a = sT[(32 + r) * LDT + i];
            const float4 t = *reinterpret_cast<const float4*>(sT + i * LDT + c);
            s.x = fmaf(a, t.x, s.x); s.y = fmaf(a, t.y, s.y); s.z = fmaf(a, t.z, s.z); s.w = fmaf(a, t.w, s.w);
        }
        __syncthreads();                                  // level 1's z is no longer read
        float* z = tmp + r * 33 + c;
        z[0] = s.x; z[1] = s.y; z[2] = s.z; z[3] = s.w;
        __syncthreads();
        s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
        for (int i = 0; i < 32; ++i) {
            const float a = sT[(32 + r) * LDT + 32 + i];
            const float* t = tmp + i * 33 + c;
            s.x = fmaf(a, t[0], s.x); s.y = fmaf(a, t[1], s.y); s.z = fmaf(a, t[2], s.z); s.w = fmaf(a, t[3], s.w);
        }
        *reinterpret_cast<float4*>(sT + (32 + r) * LDT + c) = make_float4(-s.x, -s.y, -s.z, -s.w);
    }
}

template <typename TIO, int NC>
__global__ void __launch_bounds__(NT, 1) gdn_simt_kernel(SimtParams p) {
    extern __shared__ __align__(16) uint8_t smem_raw[];
    constexpr int NQ = NC / 4;                 // value columns per thread in the row products
    constexpr int EB = 16 / (int)sizeof(TIO);  // elements per 16-byte piece
    const int dk = p.dk, dv = p.dv, H = p.H;
    const int ld = tile_ld<TIO>(dk), lds = dk + 4;
    const size_t tile = tile_bytes<TIO>(dk);
    TIO* const sK = reinterpret_cast<TIO*>(smem_raw);                    // two tiles: chunk c in tile c & 1
    TIO* const sQ = reinterpret_cast<TIO*>(smem_raw + 2 * tile);
    float* const own = reinterpret_cast<float*>(smem_raw + 3 * tile);    // steps a, b of the chunk this CTA prepared
    float* const loc = own + BK_FLOATS;                                  // the same of the chunk being walked
    float* const sS = loc + BK_FLOATS;                                   // state slice, transposed: [NC][dk + 4]
    float* const sR = sS + NC * lds;                                     // [NC][LDT] diag(beta) (V - diag(e^g) K S)
    float* const sD = sR + NC * LDT;                                     // [NC][LDT] v_new
    float* const sW = sD + NC * LDT;                                     // [NC][LDT] e^{gC-g} v_new
    TIO* const sV = reinterpret_cast<TIO*>(sW + NC * LDT);               // two slices [C][NC]

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    ptx::pdl_trigger();
    ptx::pdl_wait();                           // launched ahead of the previous kernel's end: nothing is read or written before it
    const uint32_t rank = cluster_rank();
    const int CS = (int)cluster_size();        // chunks prepared at a time, one per CTA
    const int h = blockIdx.y, n = blockIdx.z;
    const int j0 = (int)blockIdx.x * NC;       // a cluster's CTAs are neighbours in x: its groups of columns follow each other
    long tok0;
    int len;
    if (p.cu) { tok0 = p.cu[n]; len = p.cu[n + 1] - p.cu[n]; }
    else      { tok0 = (long)n * p.T; len = p.T; }
    const int nchunks = (len + C - 1) / C;

    const TIO* gq = static_cast<const TIO*>(p.q) + ((size_t)tok0 * H + h) * dk;
    const TIO* gk = static_cast<const TIO*>(p.k) + ((size_t)tok0 * H + h) * dk;
    const TIO* gv = static_cast<const TIO*>(p.v) + ((size_t)tok0 * H + h) * dv + j0;
    TIO* gout = static_cast<TIO*>(p.out) + ((size_t)tok0 * H + h) * dv + j0;
    const size_t state_off = ((size_t)n * H + h) * dk * dv + j0;

    // One 16-byte piece of a K or Q row per thread and step.  nt threads (t = 0 .. nt-1) share the copy: all of the
    // CTA at a group's start, half of it inside the walk, while the other half computes.
    const int ppr = dk / EB;
    auto load_tile = [&](TIO* dst, const TIO* src, int c, int t, int nt) {              // rows past the end are zero
        const int R = min(C, len - c * C), step = nt / ppr, r0 = t / ppr, m = (t - r0 * ppr) * EB;
        if (r0 >= step) return;
        const TIO* s = src + (size_t)(c * C + r0) * H * dk + m;
        TIO* d = dst + r0 * ld + m;
        for (int r = r0; r < C; r += step, s += (size_t)step * H * dk, d += step * ld) cp_async<16>(d, r < R ? s : src, r < R);
    };
    auto load_v = [&](int c, int t, int nt) {
        const int R = min(C, len - c * C);
        for (int x = t; x < C * NQ; x += nt) {
            const int r = x / NQ, m = (x - r * NQ) * 4;
            cp_async<4 * (int)sizeof(TIO)>(sV + (c & 1) * C * NC + r * NC + m, gv + (size_t)(c * C + (r < R ? r : 0)) * H * dv + m, r < R);
        }
    };

    for (int x = tid; x < dk * NC; x += NT) {
        const int m = x / NC, j = x - m * NC;
        sS[j * lds + m] = p.s0 ? p.s0[state_off + (size_t)m * dv + j] : 0.f;
    }

    const int l8 = lane & 7, cg = lane >> 3;          // row products: two rows (8 apart) x columns cg + 4y per thread
    const int wr = (warp & 3) * 16;                   // first of the 16 rows of this warp
    for (int c0 = 0; c0 < nchunks; c0 += CS) {
        const int mine = c0 + (int)rank, cend = min(c0 + CS, nchunks);
        if (mine < nchunks) {
            load_tile(sK + (size_t)(c0 & 1) * C * ld, gk, mine, tid, NT);
            load_tile(sQ, gq, mine, tid, NT);
            const size_t t0 = (size_t)(tok0 + (long)mine * C) * H + h;
            prepare_chunk<TIO>(sK + (size_t)(c0 & 1) * C * ld, sQ, own, reinterpret_cast<float*>(sQ), p.a + t0, p.beta + t0, H,
                               min(C, len - mine * C), dk);
            __syncthreads();
        }
        load_tile(sK + (size_t)(c0 & 1) * C * ld, gk, c0, tid, NT);
        load_tile(sQ, gq, c0, tid, NT);
        load_v(c0, tid, NT);
        cluster_sync();                               // every CTA's block is complete
        // the chunk's block travels in registers: threads 0-127 carry Tm and the gate vectors, 128-255 carry P
        constexpr int NF = (C * LDT / 4 + C + 127) / 128;
        float4 nxt[NF];
        auto fetch = [&](int c) {
            const uint32_t src = peer_addr(own + (tid < 128 ? BK_T : BK_P), (uint32_t)(c - c0));
            const uint32_t gat = peer_addr(own + BK_BETA, (uint32_t)(c - c0));
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const int x = i * 128 + (tid & 127), g = x - C * LDT / 4;
                if (g < 0) nxt[i] = load4_peer(src + x * 16);
                else if (tid < 128 && g < C) nxt[i] = load4_peer(gat + g * 16);
            }
        };
        auto put = [&]() {
            float4* dst = reinterpret_cast<float4*>(loc + (tid < 128 ? BK_T : BK_P));
            float4* gat = reinterpret_cast<float4*>(loc + BK_BETA);
#pragma unroll
            for (int i = 0; i < NF; ++i) {
                const int x = i * 128 + (tid & 127), g = x - C * LDT / 4;
                if (g < 0) dst[x] = nxt[i];
                else if (tid < 128 && g < C) gat[g] = nxt[i];
            }
        };
        fetch(c0);
        put();
        cp_async_wait();
        __syncthreads();
        for (int c = c0; c < cend; ++c) {
            const int R = min(C, len - c * C);
            const bool more = c + 1 < cend;
            const TIO* tK = sK + (size_t)(c & 1) * C * ld;
            if (more) fetch(c + 1);
            // ---- K S (warps 0-3) and Q S (warps 4-7) ----
            f2 acc[2][NQ];
#pragma unroll
            for (int x = 0; x < 2; ++x)
#pragma unroll
                for (int y = 0; y < NQ; ++y) acc[x][y] = 0;
            {
                const TIO* row = (warp < 4 ? tK : sQ) + (wr + l8) * ld;
                const float* col = sS + cg * lds;
#pragma unroll 4
                for (int m = 0; m < dk; m += 4) {
                    const F4 a0 = load4(row + m), a1 = load4(row + 8 * ld + m);
#pragma unroll
                    for (int y = 0; y < NQ; ++y) {
                        const F4 s4 = load4(col + 4 * y * lds + m);
                        acc[0][y] = dot4(a0, s4, acc[0][y]);
                        acc[1][y] = dot4(a1, s4, acc[1][y]);
                    }
                }
            }
            const float gamma = loc[BK_EG + C - 1];
            if (warp < 4) {
                // ---- v_new = Tm diag(beta) (V - diag(e^g) K S) ----
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int r = wr + l8 + 8 * x;
                    const float b = loc[BK_BETA + r], eg = loc[BK_EG + r];
#pragma unroll
                    for (int y = 0; y < NQ; ++y)
                        sR[(cg + 4 * y) * LDT + r] = b * (load1(sV + (c & 1) * C * NC + r * NC + cg + 4 * y) - eg * sum2(acc[x][y]));
                }
                half_sync(1);
#pragma unroll
                for (int x = 0; x < 2; ++x)
#pragma unroll
                    for (int y = 0; y < NQ; ++y) acc[x][y] = 0;
                const float* row = loc + BK_T + (wr + l8) * LDT;
#pragma unroll 4
                for (int i = 0; i < wr + 16; i += 4) {
                    const F4 a0 = load4(row + i), a1 = load4(row + 8 * LDT + i);
#pragma unroll
                    for (int y = 0; y < NQ; ++y) {
                        const F4 s4 = load4(sR + (cg + 4 * y) * LDT + i);
                        acc[0][y] = dot4(a0, s4, acc[0][y]);
                        acc[1][y] = dot4(a1, s4, acc[1][y]);
                    }
                }
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int r = wr + l8 + 8 * x;
                    const float ec = loc[BK_EC + r];
#pragma unroll
                    for (int y = 0; y < NQ; ++y) {
                        const float v = sum2(acc[x][y]);
                        sD[(cg + 4 * y) * LDT + r] = v;
                        sW[(cg + 4 * y) * LDT + r] = ec * v;
                    }
                }
            } else {
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const float eg = loc[BK_EG + wr + l8 + 8 * x];
#pragma unroll
                    for (int y = 0; y < NQ; ++y) acc[x][y] = pack2(eg * sum2(acc[x][y]), 0.f);
                }
                if (more) {
                    load_tile(sK + (size_t)((c + 1) & 1) * C * ld, gk, c + 1, tid - 128, 128);
                    load_v(c + 1, tid - 128, 128);
                }
            }
            __syncthreads();                          // v_new is complete; the incoming state and Q are no longer read
            if (warp < 4) {
                if (more) load_tile(sQ, gq, c + 1, tid, 128);
            } else {
                // ---- O = diag(e^g) Q S + P v_new ----
                const float* row = loc + BK_P + (wr + l8) * LDT;
#pragma unroll 4
                for (int i = 0; i < wr + 16; i += 4) {
                    const F4 a0 = load4(row + i), a1 = load4(row + 8 * LDT + i);
#pragma unroll
                    for (int y = 0; y < NQ; ++y) {
                        const F4 s4 = load4(sD + (cg + 4 * y) * LDT + i);
                        acc[0][y] = dot4(a0, s4, acc[0][y]);
                        acc[1][y] = dot4(a1, s4, acc[1][y]);
                    }
                }
#pragma unroll
                for (int x = 0; x < 2; ++x) {
                    const int r = wr + l8 + 8 * x;
                    if (r < R) {
                        TIO* o = gout + (size_t)(c * C + r) * H * dv + cg;
#pragma unroll
                        for (int y = 0; y < NQ; ++y) store1(o + 4 * y, sum2(acc[x][y]));
                    }
                }
                half_sync(2);                         // P is no longer read
            }
            // ---- S <- e^{gC} S + sum_i e^{gC-g_i} k_i v_new_i^T: four state rows of a column per thread ----
            // (the second column, G to the right, shares the K rows; G columns x dk/4 row groups fit the CTA at least
            //  half of NC at a time for every supported dk)
            const int mg = dk >> 2, G = NT / mg, j = tid / mg, m = (tid - j * mg) * 4;
            if (j < G && j < NC) {
                const bool two = j + G < NC;
                const int j2 = two ? j + G : j;
                F4 a{0, 0}, b{0, 0};
                const float* w1 = sW + j * LDT;
                const float* w2 = sW + j2 * LDT;
                const TIO* kp = tK + m;
#pragma unroll 4
                for (int i = 0; i < C; i += 4, kp += 4 * ld) {
                    const float4 x = *reinterpret_cast<const float4*>(w1 + i), y = *reinterpret_cast<const float4*>(w2 + i);
                    const float xv[4] = {x.x, x.y, x.z, x.w}, yv[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const F4 kk = load4(kp + e * ld);
                        const f2 xx = pack2(xv[e], xv[e]), yy = pack2(yv[e], yv[e]);
                        a.lo = fma2(kk.lo, xx, a.lo); a.hi = fma2(kk.hi, xx, a.hi);
                        b.lo = fma2(kk.lo, yy, b.lo); b.hi = fma2(kk.hi, yy, b.hi);
                    }
                }
                const f2 gg = pack2(gamma, gamma);
                ulonglong2* s1 = reinterpret_cast<ulonglong2*>(sS + j * lds + m);
                *s1 = make_ulonglong2(fma2(gg, s1->x, a.lo), fma2(gg, s1->y, a.hi));
                if (two) {
                    ulonglong2* s2 = reinterpret_cast<ulonglong2*>(sS + j2 * lds + m);
                    *s2 = make_ulonglong2(fma2(gg, s2->x, b.lo), fma2(gg, s2->y, b.hi));
                }
            }
            if (more) put();
            cp_async_wait();
            __syncthreads();
        }
        cluster_sync();                               // every CTA has read this one's block: it may be replaced (or go away)
    }
    if (p.sT)
        for (int x = tid; x < dk * NC; x += NT) {
            const int m = x / NC, j = x - m * NC;
            p.sT[state_off + (size_t)m * dv + j] = sS[j * lds + m];
        }
}

constexpr int kMaxDevices = 64;
// Time per chunk of the walk and of steps a, b in units of 10 ns (one B200, d = 128: 8.9 us a chunk in clusters of eight, which
// prepare eight chunks at a time, 9.75 us in clusters of four; the ratio is the same with d = 96 and 64)
constexpr long kWalk = 800, kPrep = 680;

template <typename TIO, int NC>
int launch_typed(const SimtParams& p, cudaStream_t stream) {
    // once per device: the dynamic shared-memory limit, and how many clusters of eight and of four run at once
    static std::mutex mu;
    static int active8[kMaxDevices] = {0}, active4[kMaxDevices] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return GDN_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return GDN_ERR_UNSUPPORTED;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cfg.blockDim = dim3(NT);
    {
        std::lock_guard<std::mutex> lock(mu);
        if (active4[dev] == 0) {
            cfg.dynamicSmemBytes = simt_smem<TIO, NC>(128);
            int n[2] = {0, 0};
            if (cudaFuncSetAttribute(gdn_simt_kernel<TIO, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.dynamicSmemBytes) != cudaSuccess)
                return GDN_ERR_CUDA;
            for (int i = 0; i < 2; ++i) {
                attr[0].val.clusterDim.x = i ? 4 : 8;
                cfg.gridDim = dim3(attr[0].val.clusterDim.x);
                if (cudaOccupancyMaxActiveClusters(&n[i], gdn_simt_kernel<TIO, NC>, &cfg) != cudaSuccess || n[i] <= 0) return GDN_ERR_CUDA;
            }
            active8[dev] = n[0];
            active4[dev] = n[1];
        }
    }
    // Cluster size: eight CTAs prepare eight chunks at a time for 8 NC columns; four prepare four for 4 NC columns, so
    // steps a and b cost twice as much per chunk of the walk, but more of the SMs can be covered (a B200 runs 15
    // clusters of eight or 33 of four of the largest shape).  Whichever ends first: rounds x time per chunk (512 tokens, d = 128,
    // eights / fours: 48 chains 291 / 240 us, 60 296 / 318, 64 365 / 320, 75 372 / 402, 80 441 / 405, 99 522 / 492, 120 601 / 648).
    const long groups = (long)p.B * p.H * (p.dv / NC);
    const long t8 = (groups / 8 + active8[dev] - 1) / active8[dev] * (kWalk + kPrep / 8);
    const long t4 = (groups / 4 + active4[dev] - 1) / active4[dev] * (kWalk + kPrep / 4);
    const int cs = t8 <= t4 ? 8 : 4;
    attr[0].val.clusterDim.x = cs;
    cfg.gridDim = dim3(p.dv / NC, p.H, p.B);
    cfg.dynamicSmemBytes = simt_smem<TIO, NC>(p.dk);
    cfg.stream = stream;
    cfg.numAttrs = 2;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gdn_simt_kernel<TIO, NC>, p);
    count_launch();
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_CUDA;
}

// Columns per CTA: the widest group (8 CTAs x 16, 12, 8 or 4 columns) that divides d_v.  Wider slices share each K
// and Q row read from shared memory among more columns.
template <typename TIO>
int launch_columns(const SimtParams& p, cudaStream_t stream) {
    if (p.dv % 128 == 0) return launch_typed<TIO, 16>(p, stream);
    if (p.dv % 96 == 0) return launch_typed<TIO, 12>(p, stream);
    if (p.dv % 64 == 0) return launch_typed<TIO, 8>(p, stream);
    return launch_typed<TIO, 4>(p, stream);
}

}  // namespace

bool simt_supported(int d_k, int d_v) {
    return d_k > 0 && d_v > 0 && d_k % 32 == 0 && d_k <= 128 && d_v % 32 == 0;
}

int launch_simt(const PrefillArgs& a, bool io_bf16, cudaStream_t stream) {
    if (!simt_supported(a.d_k, a.d_v)) return GDN_ERR_UNSUPPORTED;
    if (a.H > 65535 || a.B > 65535) return GDN_ERR_UNSUPPORTED;
    SimtParams p{a.q, a.k, a.v, a.log_alpha, a.beta, a.initial_state, a.out, a.final_state,
                 a.cu_seqlens, a.B, a.T, a.H, a.d_k, a.d_v};
    return io_bf16 ? launch_columns<__nv_bfloat16>(p, stream) : launch_columns<float>(p, stream);
}

}  // namespace gdn
