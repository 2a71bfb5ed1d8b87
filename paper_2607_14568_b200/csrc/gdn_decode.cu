// Single-token decode step of the gated delta rule (the recurrence advanced by one token,
// Section "The model"; decode is bandwidth-bound, Section "Decode, and why 4-bit is slower").
//
// Per (sequence, head), state S in R^{d_k x d_v} (fp32, updated in place), one token:
//     S <- alpha S ;  delta <- beta (v - S^T k) ;  S <- S + k delta^T ;  o <- S^T q
// Every value column j is independent.  With u_j = sum_m S[m][j] k[m] and w_j = sum_m S[m][j] q[m]
// taken from the OLD state, delta_j = beta (v_j - alpha u_j) and o_j = alpha w_j + (k.q) delta_j,
// so the state is read once and written once: 8 d_k d_v bytes per (sequence, head), the floor.
//
// One CTA per (sequence, head, COLS value columns); the CTA's warps share the d_k rows, all of a thread's loads are issued
// before any is used, the column sums are reduced across lanes and warps, and the updated rows are written back from
// registers.  COLS = 128 (a row is 512 contiguous bytes, one float4 per lane) moves the state at the memory's rate;
// with so few (sequence, head) pairs that most SMs would idle, a call is one round trip to memory, and 32 columns per
// CTA shorten it: four times the CTAs, a quarter of the loads per thread (one sequence, 16 heads: 6.2 -> 4.1 us a call).
// Launched ahead of the previous kernel's end (programmatic launch): back-to-back steps overlap launch and set-up.

#include "gdn_internal.h"
#include "sm100_ptx.cuh"

namespace gdn {
namespace {

constexpr int DVB = 128;          // granularity of d_v
constexpr int NW = 8;             // warps per CTA
constexpr int MAX_ROWS = 16;      // rows per warp (d_k <= 128)

struct DecodeParams {
    const __nv_bfloat16* q;
    const __nv_bfloat16* k;
    const __nv_bfloat16* v;
    const float* a;
    const float* beta;
    float* state;
    __nv_bfloat16* out;
    int H, dk, dv;
};

template <int COLS>
__global__ void __launch_bounds__(NW * 32, 2) gdn_decode_kernel(DecodeParams p) {
    constexpr int LC = COLS / 4;                              // lanes per row
    constexpr int RG = 32 / LC;                               // rows per load instruction of a warp
    constexpr int NL = MAX_ROWS / RG;                         // loads per thread
    __shared__ float sk[128], sq[128];
    __shared__ float4 su[NW][LC], sw[NW][LC];
    __shared__ float skq[NW];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int rg = lane / LC, lc = lane % LC;
    const int h = blockIdx.y, n = blockIdx.z;
    const int dk = p.dk, dv = p.dv;
    const size_t nh = (size_t)n * p.H + h;
    const int rows = dk / NW;                                 // rows of this warp: warp * rows ...
    const size_t col = (size_t)blockIdx.x * COLS + 4 * lc;
    float* S = p.state + nh * dk * dv + col;
    ptx::pdl_trigger();
    ptx::pdl_wait();                                          // the state comes from the previous step

    // the state first: every load in flight before anything else is touched
    float4 s[NL];
#pragma unroll
    for (int i = 0; i < NL; ++i)
        if (RG * i + rg < rows) s[i] = *reinterpret_cast<const float4*>(S + (size_t)(warp * rows + RG * i + rg) * dv);
    if (tid < dk) {
        sk[tid] = __bfloat162float(p.k[nh * dk + tid]);
        sq[tid] = __bfloat162float(p.q[nh * dk + tid]);
    }
    const float alpha = expf(p.a[nh]), beta = p.beta[nh];
    const uint2 vb = *reinterpret_cast<const uint2*>(p.v + nh * dv + col);
    const float v0 = __uint_as_float(vb.x << 16), v1 = __uint_as_float(vb.x & 0xffff0000u);
    const float v2 = __uint_as_float(vb.y << 16), v3 = __uint_as_float(vb.y & 0xffff0000u);
    __syncthreads();

    float4 u = make_float4(0.f, 0.f, 0.f, 0.f), wq = u;
    float kq = 0.f;
#pragma unroll
    for (int i = 0; i < NL; ++i)
        if (RG * i + rg < rows) {
            const float km = sk[warp * rows + RG * i + rg], qm = sq[warp * rows + RG * i + rg];
            u.x = fmaf(s[i].x, km, u.x); u.y = fmaf(s[i].y, km, u.y); u.z = fmaf(s[i].z, km, u.z); u.w = fmaf(s[i].w, km, u.w);
            wq.x = fmaf(s[i].x, qm, wq.x); wq.y = fmaf(s[i].y, qm, wq.y); wq.z = fmaf(s[i].z, qm, wq.z); wq.w = fmaf(s[i].w, qm, wq.w);
            kq = fmaf(km, qm, kq);
        }
#pragma unroll
    for (int d = LC; d < 32; d <<= 1) {                       // rows of the same columns in other lanes
        u.x += __shfl_xor_sync(0xffffffffu, u.x, d); u.y += __shfl_xor_sync(0xffffffffu, u.y, d);
        u.z += __shfl_xor_sync(0xffffffffu, u.z, d); u.w += __shfl_xor_sync(0xffffffffu, u.w, d);
        wq.x += __shfl_xor_sync(0xffffffffu, wq.x, d); wq.y += __shfl_xor_sync(0xffffffffu, wq.y, d);
        wq.z += __shfl_xor_sync(0xffffffffu, wq.z, d); wq.w += __shfl_xor_sync(0xffffffffu, wq.w, d);
        kq += __shfl_xor_sync(0xffffffffu, kq, d);
    }
    if (rg == 0) {
        su[warp][lc] = u;
        sw[warp][lc] = wq;
    }
    if (lane == 0) skq[warp] = kq;
    __syncthreads();
    u = su[0][lc]; wq = sw[0][lc]; kq = skq[0];
#pragma unroll
    for (int x = 1; x < NW; ++x) {                            // fixed order: deterministic
        const float4 a4 = su[x][lc], b4 = sw[x][lc];
        u.x += a4.x; u.y += a4.y; u.z += a4.z; u.w += a4.w;
        wq.x += b4.x; wq.y += b4.y; wq.z += b4.z; wq.w += b4.w;
        kq += skq[x];
    }
    float4 d;
    d.x = beta * (v0 - alpha * u.x); d.y = beta * (v1 - alpha * u.y);
    d.z = beta * (v2 - alpha * u.z); d.w = beta * (v3 - alpha * u.w);
#pragma unroll
    for (int i = 0; i < NL; ++i)
        if (RG * i + rg < rows) {
            const int m = warp * rows + RG * i + rg;
            const float km = sk[m];
            float4 o;
            o.x = fmaf(alpha, s[i].x, km * d.x); o.y = fmaf(alpha, s[i].y, km * d.y);
            o.z = fmaf(alpha, s[i].z, km * d.z); o.w = fmaf(alpha, s[i].w, km * d.w);
            *reinterpret_cast<float4*>(S + (size_t)m * dv) = o;
        }
    if (warp == 0 && rg == 0) {
        __nv_bfloat16* op = p.out + nh * dv + col;
        const __nv_bfloat162 o01 = __floats2bfloat162_rn(fmaf(alpha, wq.x, kq * d.x), fmaf(alpha, wq.y, kq * d.y));
        const __nv_bfloat162 o23 = __floats2bfloat162_rn(fmaf(alpha, wq.z, kq * d.z), fmaf(alpha, wq.w, kq * d.w));
        *reinterpret_cast<__nv_bfloat162*>(op) = o01;
        *reinterpret_cast<__nv_bfloat162*>(op + 2) = o23;
    }
}

}  // namespace

bool decode_supported(int d_k, int d_v) { return d_k > 0 && d_k % NW == 0 && d_k <= NW * MAX_ROWS && d_v > 0 && d_v % DVB == 0; }

int launch_decode(const void* q, const void* k, const void* v, const float* log_alpha, const float* beta,
                  float* state, void* out, int B, int H, int d_k, int d_v, cudaStream_t stream) {
    if (!decode_supported(d_k, d_v)) return GDN_ERR_UNSUPPORTED;
    if (H > 65535 || B > 65535) return GDN_ERR_UNSUPPORTED;
    DecodeParams p{static_cast<const __nv_bfloat16*>(q), static_cast<const __nv_bfloat16*>(k),
                   static_cast<const __nv_bfloat16*>(v), log_alpha, beta, state, static_cast<__nv_bfloat16*>(out), H, d_k, d_v};
    // 32 columns per CTA while the CTAs of 128 would not give every SM one (148 on a B200): 64 of them 5.0 -> 3.4 us, 80 6.0 -> 4.7 us,
    // 128 6.0 -> 5.3 us, but 256 6.4 -> 9 us (one B200, back to back)
    const int sms = sm_count();
    if (sms <= 0) return GDN_ERR_CUDA;
    const bool narrow = (long)B * H * (d_v / DVB) <= sms;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(d_v / (narrow ? 32 : DVB), H, B);
    cfg.blockDim = dim3(NW * 32);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, narrow ? gdn_decode_kernel<32> : gdn_decode_kernel<DVB>, p);
    count_launch();
    return cudaGetLastError() == cudaSuccess ? GDN_OK : GDN_ERR_CUDA;
}

}  // namespace gdn
