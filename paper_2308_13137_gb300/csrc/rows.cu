// Per-token row kernels with the row held in registers: the activation quantizer Q_a (Eq. 2 with
// gamma = beta = 1, one group per token, Sec. 4.1) fused with its producers (LET of Eq. 3,
// RMSNorm, SwiGLU), the RoPE + [Q,K] LET (Eq. 5) + Q_a chain of q, k, v, and the straight-through
// backward of each.  One CTA walks one token row at a time; each thread owns fixed float4 vectors
// of the row (vector j*NT + tid), so a row needs only its block reductions (long forward rows wait in
// shared memory between their passes), and the LET column sums of a thread's columns accumulate in registers across rows.
#include "attn.cuh"
#include "quant.cuh"

#include <algorithm>

namespace {

__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float f4get(const float4& v, int e) { return e == 0 ? v.x : (e == 1 ? v.y : (e == 2 ? v.z : v.w)); }
// silu(g) = g sigmoid(g); the quotient by the correctly rounded reciprocal (one rounding more than
// an IEEE division: within 1 ulp of g / (1 + e^-g)); the forward and the backward's recomputation of
// the quantizer input both use this form
__device__ __forceinline__ float silu(float g) { return g * __frcp_rn(1.f + expf(-g)); }

__device__ __forceinline__ void st_bf16x4(__nv_bfloat16* p, const float* v) {
  uint2 u;
  __nv_bfloat162* q = reinterpret_cast<__nv_bfloat162*>(&u);
  q[0] = __floats2bfloat162_rn(v[0], v[1]);
  q[1] = __floats2bfloat162_rn(v[2], v[3]);
  *reinterpret_cast<uint2*>(p) = u;
}

}  // namespace

// fake quantization of four elements; SMALL: the row's quotients are inside omq_rint2_small's range
template <bool SMALL>
__device__ __forceinline__ void quant4(float (&v)[4], const QState& qs, float Q, float (&cd)[4]) {
#pragma unroll
  for (int e = 0; e < 4; e += 2) {
    float2 c2;
    const float2 w = make_float2(v[e], v[e + 1]);
    const float2 r = SMALL ? omq_fakequant2_small(w, qs, Q, &c2) : omq_fakequant2(w, qs, Q, &c2);
    v[e] = r.x; v[e + 1] = r.y; cd[e] = c2.x; cd[e + 1] = c2.y;
  }
}

__device__ __forceinline__ uint32_t pack_codes4(const float (&cd)[4]) {
  return (uint32_t)cd[0] | ((uint32_t)cd[1] << 8) | ((uint32_t)cd[2] << 16) | ((uint32_t)cd[3] << 24);
}

// one float4 of a quantized row: fake-quantized, stored as bf16, codes where wanted
__device__ __forceinline__ void act_store4(const ActFwdArgs& a, int64_t t, int64_t vi, float (&v)[4], const QState& qs,
                                           float Q, bool quant, bool small) {
  float cd[4];
  if (quant) {
    if (small) quant4<true>(v, qs, Q, cd);
    else quant4<false>(v, qs, Q, cd);
  }
  st_bf16x4(a.Xq + t * a.ldq + 4 * vi, v);
  if (a.codes && quant) *reinterpret_cast<uint32_t*>(a.codes + t * a.C + 4 * vi) = pack_codes4(cd);
}

// v -= delta (one float4 of a LET producer)
__device__ __forceinline__ void let_sub4(float (&v)[4], const ActFwdArgs& a, int64_t vi) {
  if (!a.delta) return;
  const float4 dl = ld4(a.delta + 4 * vi);
#pragma unroll
  for (int e = 0; e < 4; ++e) v[e] = v[e] - f4get(dl, e);
}

// ================================================================================================
// activation quantizer forward: producer -> (LET) -> Q_a -> bf16
// ================================================================================================
// Rows of up to 4 K columns, one CTA a row, held in the registers of 128 threads (32 values each).  Two block
// barriers (three with RMSNorm): the extremes are combined from per-warp values by every thread, and the first
// indices are found by the holders of an extreme alone, in shared memory.  What bounds it is the latency of
// its phases, so many short CTAs beat fewer with several rows each: 2048 x 4096 takes 25 us with LET and 13 without,
// and with two, three, four and seven rows a CTA 14, 7, 14 and 38 % more (12 - 35 % without LET).  The rounding
// stays off the conversion pipe.
template <int P, int NT, int VPT, int MINB>
__global__ void __launch_bounds__(NT, MINB) act_fwd_rows(ActFwdArgs a) {
  constexpr int NE = 4 * VPT, NW = NT / 32;
  constexpr bool LETP = P == AP_LET || P == AP_RMS_LET;
  static_assert(P != AP_SWIGLU, "the SwiGLU row is staged in shared memory (act_fwd_smem)");
  __shared__ float red[3][NW];
  __shared__ int sidx[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t nv = a.C / 4;
  const int64_t t = blockIdx.x;
  const bool quant = a.abits < 16;
  const float Q = (float)((1 << (quant ? a.abits : 1)) - 1);
  if (tid == 0) { sidx[0] = OMQ_NO_INDEX; sidx[1] = OMQ_NO_INDEX; }
  float4 raw[VPT];
#pragma unroll
  for (int j = 0; j < VPT; ++j) {                   // every load of the row first
    const int64_t vi = (int64_t)j * NT + tid;
    raw[j] = vi < nv ? ld4(a.X + t * a.ldx + 4 * vi) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float val[VPT][4];
  float ss = 0.f;
#pragma unroll
  for (int j = 0; j < VPT; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      val[j][e] = f4get(raw[j], e);
      if (P == AP_RMS_LET) ss = fmaf(val[j][e], val[j][e], ss);
    }
  if (P == AP_RMS_LET) {                            // the summation tree of block_sum2
    ss = warp_sum(ss);
    if (lane == 0) red[2][warp] = ss;
    __syncthreads();
    const float tot = NW == 4 ? (red[2][0] + red[2][2]) + (red[2][1] + red[2][3]) : warp_sum(lane < NW ? red[2][lane] : 0.f);
    const float rstd = 1.0f / sqrtf(tot / (float)a.C + a.rms_eps);
    if (tid == 0 && a.rstd) a.rstd[t] = rstd;
#pragma unroll
    for (int j = 0; j < VPT; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) val[j][e] = __fmul_rn(val[j][e], rstd);   // rounded before delta is taken off
  }
  if (LETP) {
#pragma unroll
    for (int j = 0; j < VPT; ++j) {
      const int64_t vi = (int64_t)j * NT + tid;
      if (vi < nv) {
        let_sub4(val[j], a, vi);
        if (a.s) {
          const float4 sv = ld4(a.s + 4 * vi);
#pragma unroll
          for (int e = 0; e < 4; ++e) val[j][e] = __fdiv_rn(val[j][e], f4get(sv, e));
        }
      }
    }
  }
  QState qs{};
  bool small = false;
  if (quant) {
    float lM = -INFINITY, lm = INFINITY;             // this thread's own extremes
#pragma unroll
    for (int j = 0; j < VPT; ++j)
      if ((int64_t)j * NT + tid < nv)
#pragma unroll
        for (int e = 0; e < 4; ++e) { lM = fmaxf(lM, val[j][e]); lm = fminf(lm, val[j][e]); }
    float M = lM, m = lm;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
      m = fminf(m, __shfl_xor_sync(0xffffffffu, m, off));
    }
    if (lane == 0) { red[0][warp] = M; red[1][warp] = m; }
    __syncthreads();
    M = red[0][0]; m = red[1][0];
#pragma unroll
    for (int w = 1; w < NW; ++w) { M = fmaxf(M, red[0][w]); m = fminf(m, red[1][w]); }
    if (lM == M || lm == m) {
      int iM = OMQ_NO_INDEX, im = OMQ_NO_INDEX;
#pragma unroll
      for (int k = NE - 1; k >= 0; --k) {
        const int64_t vi = (int64_t)(k >> 2) * NT + tid;
        if (vi < nv) {
          if (val[k >> 2][k & 3] == M) iM = (int)(4 * vi) + (k & 3);
          if (val[k >> 2][k & 3] == m) im = (int)(4 * vi) + (k & 3);
        }
      }
      if (iM != OMQ_NO_INDEX) atomicMin(&sidx[0], iM);
      if (im != OMQ_NO_INDEX) atomicMin(&sidx[1], im);
    }
    qs = omq_qstate(M, m, 1.f, 1.f, Q, a.eps);
    small = omq_small_quot(qs);
  }
#pragma unroll
  for (int j = 0; j < VPT; ++j) {
    const int64_t vi = (int64_t)j * NT + tid;
    if (vi < nv) act_store4(a, t, vi, val[j], qs, Q, quant, small);
  }
  if (!quant) return;
  __syncthreads();                                  // first indices final
  if (tid == 0) {
    a.h[t] = qs.h; a.z[t] = (int32_t)qs.z;
    a.imax[t] = omq_saved_index(sidx[0], 0); a.imin[t] = omq_saved_index(sidx[1], 0);
  }
}

// Longer rows, and the SwiGLU row: the CTA's one row goes through shared memory.  Pass 1 forms the quantizer
// input (loads four float4 ahead) and the extremes, pass 2 quantizes it from there, so a thread needs few
// registers whatever the row's length and several CTAs a SM overlap one's loads with another's arithmetic.
// 2048 x 11008 SwiGLU rows in registers (48 values a thread, one CTA a SM) took 98 us.
template <int P, int NT>
__global__ void __launch_bounds__(NT) act_fwd_smem(ActFwdArgs a) {
  constexpr int NW = NT / 32;
  static_assert(P != AP_RMS_LET, "RMSNorm rows keep the summation order of the register form");
  extern __shared__ float4 row4[];                    // [C / 4]
  __shared__ float red[2][NW];
  __shared__ int sidx[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nv = (int)(a.C / 4);
  const int64_t t = blockIdx.x;
  const bool quant = a.abits < 16;
  const float Q = (float)((1 << (quant ? a.abits : 1)) - 1);
  const float* xr = a.X + t * a.ldx;
  const float* ur = P == AP_SWIGLU ? a.U + t * a.ldu : nullptr;
  if (tid == 0) { sidx[0] = OMQ_NO_INDEX; sidx[1] = OMQ_NO_INDEX; }
  QState qs{};
  float lM = -INFINITY, lm = INFINITY;
  for (int i0 = tid; i0 < nv; i0 += 4 * NT) {
    float4 x4[4], u4[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int vi = i0 + k * NT;
      x4[k] = vi < nv ? ld4(xr + 4 * vi) : make_float4(0.f, 0.f, 0.f, 0.f);
      if (P == AP_SWIGLU) u4[k] = vi < nv ? ld4(ur + 4 * vi) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int vi = i0 + k * NT;
      if (vi >= nv) break;
      float v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = P == AP_SWIGLU ? silu(f4get(x4[k], e)) * f4get(u4[k], e) : f4get(x4[k], e);
      if (P == AP_LET) {
        let_sub4(v, a, vi);
        if (a.s) {
          const float4 sv = ld4(a.s + 4 * vi);
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = __fdiv_rn(v[e], f4get(sv, e));
        }
      }
      if (!quant) {
        act_store4(a, t, vi, v, qs, Q, false, false);
        continue;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) { lM = fmaxf(lM, v[e]); lm = fminf(lm, v[e]); }
      row4[vi] = make_float4(v[0], v[1], v[2], v[3]);
    }
  }
  if (!quant) return;
  float M = lM, m = lm;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    m = fminf(m, __shfl_xor_sync(0xffffffffu, m, off));
  }
  if (lane == 0) { red[0][warp] = M; red[1][warp] = m; }
  __syncthreads();
  M = red[0][lane % NW]; m = red[1][lane % NW];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
    m = fminf(m, __shfl_xor_sync(0xffffffffu, m, off));
  }
  qs = omq_qstate(M, m, 1.f, 1.f, Q, a.eps);
  const bool small = omq_small_quot(qs);
  int iM = OMQ_NO_INDEX, im = OMQ_NO_INDEX;
  const bool holder = lM == M || lm == m;
  for (int vi = tid; vi < nv; vi += NT) {
    const float4 r = row4[vi];
    float v[4] = {r.x, r.y, r.z, r.w};
    if (holder) {
#pragma unroll
      for (int e = 3; e >= 0; --e) {
        if (v[e] == M) iM = min(iM, 4 * vi + e);
        if (v[e] == m) im = min(im, 4 * vi + e);
      }
    }
    act_store4(a, t, vi, v, qs, Q, true, small);
  }
  if (iM != OMQ_NO_INDEX) atomicMin(&sidx[0], iM);
  if (im != OMQ_NO_INDEX) atomicMin(&sidx[1], im);
  __syncthreads();
  if (tid == 0) {
    a.h[t] = qs.h; a.z[t] = (int32_t)qs.z;
    a.imax[t] = omq_saved_index(sidx[0], 0); a.imin[t] = omq_saved_index(sidx[1], 0);
  }
}

// ================================================================================================
// activation quantizer backward: STE of Q_a, then the producer's backward, streamed.
// The STE gradient of a token is the in-range mask times the incoming gradient everywhere except
// at the first max / min, which also receive the h-path routing (a row sum).  So one streaming
// pass writes every output with the masked gradient and accumulates the row sums; after one block
// reduction the owners of the two routed elements rewrite them.  Only RMSNorm, whose backward
// needs the row dot product of the final gradient, streams the row a second time (from L2).
// 256 threads, low register count: several CTAs (rows) per SM hide the load latency (512 threads where
// the LET column sums of a longer row would take more than 32 registers a thread).  CTA p
// handles rows [p * rows_per_cta, ...) and writes LET column partial p.  A row's quantizer state and the
// inputs at its max and min hang on a chain of three dependent loads: they are formed for eight
// rows at a time, one warp each, before the rows are walked.
// ================================================================================================

__device__ __forceinline__ float3 block_sum3(float a, float b, float c, float* smem) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  a = warp_sum(a); b = warp_sum(b); c = warp_sum(c);
  __syncthreads();
  if (lane == 0) { smem[wid] = a; smem[32 + wid] = b; smem[64 + wid] = c; }
  __syncthreads();
  float x = lane < nw ? smem[lane] : 0.f, y = lane < nw ? smem[32 + lane] : 0.f, z = lane < nw ? smem[64 + lane] : 0.f;
  return make_float3(warp_sum(x), warp_sum(y), warp_sum(z));
}

// o . d over one float4 group, in the order of the attention backward's own row dot
__device__ __forceinline__ float rowdot4(const float4 o, const float (&d)[4]) {
  return o.x * d[0] + o.y * d[1] + o.z * d[2] + o.w * d[3];
}

// X~ of one element from the producer's inputs (exactly as the forward formed it)
template <int P>
__device__ __forceinline__ float act_xt(const ActBwdArgs& a, float x, float u, float dl, float sv, float rstd) {
  float v;
  if (P == AP_SWIGLU) v = silu(x) * u;
  else if (P == AP_RMS_LET) v = __fmul_rn(x, rstd);   // rounded before delta is taken off, as in the forward
  else v = x;
  if (P == AP_LET || P == AP_RMS_LET) {
    if (a.delta) v = v - dl;
    if (a.s) v = __fdiv_rn(v, sv);
  }
  return v;
}

// What a token row's backward needs besides the row itself: the quantizer state, re-formed once per row, and the
// values at its max (r = 0) and min (r = 1), whose gradient receives the routing.
struct ActBwdRowState {
  float h, z, rh, u, rstd;
  int floored, small;
  int idx[2];
  float x[2], up[2], g[2], v[2], s[2];
};
constexpr int kStateRows = 8;          // rows whose states are formed together, one warp each

// One warp forms row t's state: lane 0 the max, lane 1 the min, then the state from both.
template <int P>
__device__ __forceinline__ void act_row_state(const ActBwdArgs& a, int64_t t, float Q, int lane, ActBwdRowState& o) {
  constexpr bool LETP = (P == AP_LET || P == AP_RMS_LET);
  const float rstd = P == AP_RMS_LET ? a.rstd[t] : 1.f;
  if (a.abits >= 16) {
    if (lane == 0) o.rstd = rstd;
    return;
  }
  const int r = lane & 1;
  const int c = r == 0 ? a.imax[t] : a.imin[t];
  const float x = a.X[t * a.ldx + c];
  const float up = P == AP_SWIGLU ? a.U[t * a.ldu + c] : 0.f;
  const float dl = (LETP && a.delta) ? a.delta[c] : 0.f;
  const float sv = (LETP && a.s) ? a.s[c] : 1.f;
  const float g = a.dXq[t * a.lddq + c];
  const float v = act_xt<P>(a, x, up, dl, sv, rstd);
  const float M = __shfl_sync(0xffffffffu, v, 0), m = __shfl_sync(0xffffffffu, v, 1);
  if (lane < 2) { o.idx[r] = c; o.x[r] = x; o.up[r] = up; o.g[r] = g; o.v[r] = v; o.s[r] = sv; }
  if (lane == 0) {
    QState qs = omq_qstate(M, m, 1.f, 1.f, Q, a.eps);
    qs.h = a.h[t]; qs.z = (float)a.z[t]; qs.rh = __frcp_rn(qs.h);
    o.h = qs.h; o.z = qs.z; o.rh = qs.rh; o.u = __fmul_rn(m, qs.rh); o.rstd = rstd;
    o.floored = qs.floored; o.small = omq_small_quot(qs) ? 1 : 0;
  }
}

template <int P, int NT, int VPT, int JB, int MINB, bool SUMS, bool RD = false>
__global__ void __launch_bounds__(NT, MINB) act_bwd_stream(ActBwdArgs a) {
  constexpr bool LETP = (P == AP_LET || P == AP_RMS_LET);
  static_assert(!SUMS || LETP, "only the LET producers have column sums");
  static_assert(VPT % JB == 0, "whole batches");
  constexpr int NE = SUMS ? 4 * VPT : 1;
  // the SwiGLU body is long: the batches of a long row, unrolled, overflow the instruction cache (2048 x 28672:
  // 377 us unrolled, 211 not; 2048 x 11008 81 and 76).  The others gain 3% by unrolling, or index registers
  constexpr int UNR = P == AP_SWIGLU ? 1 : VPT / JB;
  __shared__ float fsm[96];
  __shared__ ActBwdRowState rows_sm[kStateRows];
  const int tid = threadIdx.x, lane = tid & 31;
  const int nv = (int)(a.C / 4);
  const bool quant = a.abits < 16;
  const float Q = (float)((1 << (quant ? a.abits : 1)) - 1);
  const bool want_out = a.dX != nullptr || a.dXb != nullptr;
  const int64_t nparts = (a.T + a.rows_per_cta - 1) / a.rows_per_cta;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f), o4 = make_float4(1.f, 1.f, 1.f, 1.f);
  // the inputs come into L2 ahead of their use: whole rows, the next one's while this one is worked on; with column
  // sums (one CTA a SM) and long rows a window instead, spread over the row (1531 x 11008 91 -> 83 us, 1024 x 14336
  // 88 -> 78; without sums, several CTAs a SM, the window is 3 - 15% slower)
  constexpr bool WIN = SUMS && NT * VPT * 16 > 32 * 1024;
  constexpr int WINB = 16 * 1024;
  const int row_bytes = (int)(a.C * 4);
  auto fetch = [&](int64_t t, int b0, int b1) {      // bytes [b0, b1) of row t
    if (b0 >= b1) return;
    omq_l2_prefetch(a.X + t * a.ldx + b0 / 4, (uint64_t)(b1 - b0));
    omq_l2_prefetch(a.dXq + t * a.lddq + b0 / 4, (uint64_t)(b1 - b0));
    if (P == AP_SWIGLU) omq_l2_prefetch(a.U + t * a.ldu + b0 / 4, (uint64_t)(b1 - b0));
  };
  float acc_s[NE], acc_d[NE];
  // with column sums: 1/s of the thread's columns in shared memory (each thread reads back only its own
  // slots), computed once; the exact division of the quantizer input takes it too (omq_div2).  The RMSNorm
  // backward also keeps x * rstd and the masked gradient of its elements in registers for pass 2
  constexpr bool RS = SUMS;
  constexpr bool KEEP = RS && P == AP_RMS_LET && VPT <= 8;   // a longer row's would spill
  // the plain form with a.rowdot: D[head, t] = the sum of bf16(dX) X over each 128-column head (the
  // attention backward's rowsum(dO * O)), taken while the row is here; the float4 group j of a warp
  // is one head (lane L holds its columns 4L .. 4L + 3)
  static_assert(!RD || (P == AP_PLAIN && !SUMS), "the row dot is a form of the plain producer");
  float dpart[RD ? VPT : 1];
  __shared__ float4 rs_sm[RS ? VPT * NT : 1];
  float xk[KEEP ? NE : 1], dk[KEEP ? NE : 1];
  bool s_ok = LETP && RS && a.s != nullptr;
#pragma unroll
  for (int j = 0; j < (RS ? VPT : 0); ++j) {
    const int vi = j * NT + tid;
    const float4 sv = (LETP && a.s && vi < nv) ? ld4(a.s + 4 * vi) : o4;
    s_ok = s_ok && omq_div_ok(sv.x) && omq_div_ok(sv.y) && omq_div_ok(sv.z) && omq_div_ok(sv.w);
    rs_sm[j * NT + tid] = make_float4(__frcp_rn(sv.x), __frcp_rn(sv.y), __frcp_rn(sv.z), __frcp_rn(sv.w));
  }
  for (int64_t p = blockIdx.x; p < nparts; p += gridDim.x) {
#pragma unroll
    for (int k = 0; k < NE; ++k) { acc_s[k] = 0.f; acc_d[k] = 0.f; }
    const int64_t t0 = p * a.rows_per_cta, t1 = min(a.T, t0 + a.rows_per_cta);
    if (tid == 0) fetch(t0, 0, WIN ? WINB : row_bytes);   // the first row on its way while the states are formed
    for (int64_t t = t0; t < t1; ++t) {
      if (tid == 0) {                          // the next row's inputs (and this row's residual) into L2
        if (P == AP_RMS_LET && a.resid) omq_l2_prefetch(a.resid + t * a.lddx, row_bytes);
        if (!WIN && t + 1 < t1) {
          fetch(t + 1, 0, row_bytes);
          if (P == AP_RMS_LET && a.resid) omq_l2_prefetch(a.resid + (t + 1) * a.lddx, row_bytes);
        }
      }
      if ((t - t0) % kStateRows == 0) {        // the states of the next rows, off each row's own chain of loads
        __syncthreads();
        for (int w = tid >> 5; w < kStateRows && t + w < t1; w += NT / 32)
          act_row_state<P>(a, t + w, Q, lane, rows_sm[w]);
        __syncthreads();
      }
      const ActBwdRowState& S = rows_sm[(t - t0) % kStateRows];
      const float rstd = S.rstd;
      const float* xr = a.X + t * a.ldx;
      const float* gr = a.dXq + t * a.lddq;
      const float* ur = (P == AP_SWIGLU) ? a.U + t * a.ldu : nullptr;
      QState qs{};
      int iM = -1, im = -1;
      bool small = false;
      if (quant) {
        iM = S.idx[0]; im = S.idx[1];
        qs.h = S.h; qs.z = S.z; qs.rh = S.rh; qs.u = S.u; qs.floored = S.floored;
        small = S.small != 0;
      }
      float Gh = 0.f, Gbm = 0.f, dot = 0.f;
      // ---- pass 1: masked gradient through the producer, row sums ----
#pragma unroll UNR
      for (int jb = 0; jb < VPT; jb += JB) {
        if (UNR == 1 && jb * NT >= nv) break;
        if (WIN && tid == 0) {                          // the window moves on, into the next row at its end
          const int b0 = WINB + jb * NT * 16, b1 = b0 + JB * NT * 16;
          if (b0 < row_bytes) fetch(t, b0, min(b1, row_bytes));
          if (b1 > row_bytes && t + 1 < t1) fetch(t + 1, max(b0 - row_bytes, 0), min(b1 - row_bytes, WINB));
        }
        float4 x4[JB], g4[JB], u4[JB];
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {               // every load of the batch first
          const int vi = (jb + jj) * NT + tid;
          const bool ok = vi < nv;
          x4[jj] = ok ? ld4(xr + 4 * vi) : z4;
          g4[jj] = ok ? ld4(gr + 4 * vi) : z4;
          u4[jj] = (P == AP_SWIGLU && ok) ? ld4(ur + 4 * vi) : z4;
        }
#pragma unroll
        for (int jj = 0; jj < JB; ++jj) {
          const int j = jb + jj;
          const int vi = j * NT + tid;
          if (vi >= nv) continue;
          const float4 rs4 = RS ? rs_sm[j * NT + tid] : o4;
          float4 sv = o4;
          if (LETP && a.s) sv = ld4(a.s + 4 * vi);
          // the quantizer input, as the forward formed it
          float v[4], sg[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float x = f4get(x4[jj], e);
            if (P == AP_SWIGLU) {
              sg[e] = __frcp_rn(1.f + expf(-x));
              v[e] = (x * sg[e]) * f4get(u4[jj], e);
            } else {
              v[e] = P == AP_RMS_LET ? __fmul_rn(x, rstd) : x;
            }
          }
          if (LETP) {
            if (a.delta) {
              const float4 dl = ld4(a.delta + 4 * vi);
#pragma unroll
              for (int e = 0; e < 4; ++e) v[e] = v[e] - f4get(dl, e);
            }
            if (a.s) {
              const uint32_t key = max(max(omq_div_key(v[0]), omq_div_key(v[1])), max(omq_div_key(v[2]), omq_div_key(v[3])));
              if (RS && s_ok && key < OMQ_DIV_KEYS) {
                const float2 q0 = omq_div2(make_float2(v[0], v[1]), make_float2(sv.x, sv.y), make_float2(rs4.x, rs4.y));
                const float2 q1 = omq_div2(make_float2(v[2], v[3]), make_float2(sv.z, sv.w), make_float2(rs4.z, rs4.w));
                v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
              } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) v[e] = __fdiv_rn(v[e], f4get(sv, e));
              }
            }
          }
          float dh[4];
          int in[4] = {1, 1, 1, 1};
          if (quant) {
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
              const float2 w = make_float2(v[e], v[e + 1]);
              const float2 r = small ? omq_ste_dh2_small(w, qs, Q, &in[e], &in[e + 1]) : omq_ste_dh2(w, qs, Q, &in[e], &in[e + 1]);
              dh[e] = r.x; dh[e + 1] = r.y;
            }
          }
          float o1[4], o2[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float x = f4get(x4[jj], e), g = f4get(g4[jj], e);
            float d = g;
            if (quant) {
              Gh = fmaf(g, dh[e], Gh);
              if (!in[e]) { Gbm += g; d = 0.f; }
            }
            if (P == AP_SWIGLU) {
              const float uu = f4get(u4[jj], e);
              o1[e] = d * uu * sg[e] * (1.f + x * (1.f - sg[e]));
              o2[e] = d * x * sg[e];
            } else {
              if (SUMS) {                        // divided by s once, when the partial is written
                const int k = (4 * j + e) % NE;
                acc_s[k] = fmaf(d, v[e], acc_s[k]);
                acc_d[k] += d;
              }
              const int k = (4 * j + e) % NE;
              const float rcp = RS ? f4get(rs4, e) : ((LETP && a.s) ? __frcp_rn(f4get(sv, e)) : 1.f);
              const float dn = (LETP && a.s) ? d * rcp : d;
              if (P == AP_RMS_LET) dot = fmaf(dn, x * rstd, dot);
              if (KEEP) { xk[k] = x * rstd; dk[k] = dn; }
              o1[e] = dn;
            }
          }
          if (P == AP_SWIGLU) {
            if (a.dX) {
              *reinterpret_cast<float4*>(a.dX + t * a.lddx + 4 * vi) = make_float4(o1[0], o1[1], o1[2], o1[3]);
              *reinterpret_cast<float4*>(a.dU + t * a.lddx + 4 * vi) = make_float4(o2[0], o2[1], o2[2], o2[3]);
            }
            if (a.dXb) { st_bf16x4(a.dXb + t * a.lddxb + 4 * vi, o1); st_bf16x4(a.dUb + t * a.lddxb + 4 * vi, o2); }
          } else if (P == AP_PLAIN || P == AP_LET) {
            if (a.dX) *reinterpret_cast<float4*>(a.dX + t * a.lddx + 4 * vi) = make_float4(o1[0], o1[1], o1[2], o1[3]);
            if (a.dXb) st_bf16x4(a.dXb + t * a.lddxb + 4 * vi, o1);
            if constexpr (RD) {   // C % 128 == 0: the whole warp is here
              float b4[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) b4[e] = __bfloat162float(__float2bfloat16_rn(o1[e]));
              dpart[j] = rowdot4(x4[jj], b4);
            }
          }
        }
      }
      if constexpr (RD) {
#pragma unroll
        for (int j = 0; j < VPT; ++j) {
          const int v0 = j * NT + (tid & ~31);   // the head's first float4 (warp-uniform)
          if (v0 >= nv) break;
          const float sd = warp_sum(dpart[j]);
          if (lane == 0) a.rowdot[(v0 >> 5) * a.ldrow + t] = sd;
        }
      }
      if (!quant && !(P == AP_RMS_LET && want_out)) continue;
      const float3 tot = block_sum3(Gh, Gbm, dot, fsm);
      float GaM = 0.f, Gbt = 0.f;
      if (quant) {
        const float Gh_t = qs.floored ? 0.f : tot.x;
        GaM = Gh_t / Q;
        Gbt = tot.y - Gh_t / Q;
      }
      // ---- the routed elements: their owners rewrite them ----
      float dot_t = tot.z;
      if (quant) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int c = r == 0 ? iM : im;
          if (r == 1 && im == iM) break;
          const float route = (im == iM) ? GaM + Gbt : (r == 0 ? GaM : Gbt);
          const float x = S.x[r], se = S.s[r];
          if (P == AP_RMS_LET) dot_t = fmaf((a.s ? __fdiv_rn(route, se) : route), x * rstd, dot_t);
          if ((c >> 2) % NT != tid) continue;
          const float v = S.v[r];
          int in = 0;
          omq_ste_dh(v, qs, Q, &in);
          const float d = (in ? S.g[r] : 0.f) + route;
          if (P == AP_SWIGLU) {
            const float uu = S.up[r];
            const float sg = __frcp_rn(1.f + expf(-x));
            const float v1 = d * uu * sg * (1.f + x * (1.f - sg)), v2 = d * x * sg;
            if (a.dX) { a.dX[t * a.lddx + c] = v1; a.dU[t * a.lddx + c] = v2; }
            if (a.dXb) { a.dXb[t * a.lddxb + c] = f_to_bf16(v1); a.dUb[t * a.lddxb + c] = f_to_bf16(v2); }
          } else {
            if (SUMS) {
#pragma unroll
              for (int k = 0; k < NE; ++k)
                if (4 * ((k >> 2) * NT + tid) + (k & 3) == c) {
                  acc_s[k] = fmaf(route, v, acc_s[k]);
                  acc_d[k] += route;
                }
            }
            if (P == AP_PLAIN || P == AP_LET) {
              const float dn = (LETP && a.s) ? __fdiv_rn(d, se) : d;
              if (a.dX) a.dX[t * a.lddx + c] = dn;
              if (a.dXb) a.dXb[t * a.lddxb + c] = f_to_bf16(dn);
            }
          }
        }
        if constexpr (RD) {     // the heads of the routed elements, summed again
          __syncwarp();                                  // the owner's rewrite, seen by its warp
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int c = r == 0 ? iM : im;
            if (r == 1 && (im >> 7) == (iM >> 7)) break;
            const int v0 = (c >> 2) & ~31;                 // the head's first float4
            if (((v0 % NT) >> 5) != (tid >> 5)) continue;
            const int vi = v0 + lane;
            const uint2 u = *reinterpret_cast<const uint2*>(a.dXb + t * a.lddxb + 4 * vi);
            const float2 b01 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
            const float2 b23 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
            const float b4[4] = {b01.x, b01.y, b23.x, b23.y};
            const float sd = warp_sum(rowdot4(ld4(xr + 4 * vi), b4));
            if (lane == 0) a.rowdot[(v0 >> 5) * a.ldrow + t] = sd;
          }
        }
      }
      // ---- RMSNorm backward: second pass over the row ----
      if (KEEP && want_out) {                    // x * rstd and dn kept from pass 1: only resid is read
        const float mean_dot = dot_t / (float)a.C;
#pragma unroll
        for (int jb = 0; jb < VPT; jb += JB) {
          float4 r4[JB];
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const int vi = (jb + jj) * NT + tid;
            r4[jj] = (vi < nv && a.resid) ? ld4(a.resid + t * a.lddx + 4 * vi) : z4;
          }
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const int j = jb + jj;
            const int vi = j * NT + tid;
            if (vi >= nv) continue;
            float o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int k = (4 * j + e) % NE;
              const int c = 4 * vi + e;
              float dn = dk[k];
              if (c == iM || c == im) {
                const float rc = f4get(rs_sm[j * NT + tid], e);
                if (c == iM) dn = fmaf(GaM, rc, dn);
                if (c == im) dn = fmaf(Gbt, rc, dn);
              }
              o[e] = rstd * (dn - xk[k] * mean_dot) + f4get(r4[jj], e);
            }
            if (a.dX) *reinterpret_cast<float4*>(a.dX + t * a.lddx + 4 * vi) = make_float4(o[0], o[1], o[2], o[3]);
            if (a.dXb) st_bf16x4(a.dXb + t * a.lddxb + 4 * vi, o);
          }
        }
      } else if (P == AP_RMS_LET && want_out) {
        const float mean_dot = dot_t / (float)a.C;
#pragma unroll
        for (int jb = 0; jb < VPT; jb += JB) {
          float4 x4[JB], g4[JB], r4[JB];
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const int vi = (jb + jj) * NT + tid;
            const bool ok = vi < nv;
            x4[jj] = ok ? ld4(xr + 4 * vi) : z4;
            g4[jj] = ok ? ld4(gr + 4 * vi) : z4;
            r4[jj] = (ok && a.resid) ? ld4(a.resid + t * a.lddx + 4 * vi) : z4;
          }
#pragma unroll
          for (int jj = 0; jj < JB; ++jj) {
            const int vi = (jb + jj) * NT + tid;
            if (vi >= nv) continue;
            float4 dl = z4, sv = o4;
            if (a.delta) dl = ld4(a.delta + 4 * vi);
            if (a.s) sv = ld4(a.s + 4 * vi);
            float o[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int c = 4 * vi + e;
              const float x = f4get(x4[jj], e), g = f4get(g4[jj], e), se = f4get(sv, e);
              float d = g;
              if (quant) {
                const float v = act_xt<P>(a, x, 0.f, f4get(dl, e), se, rstd);
                int in = 0;
                omq_ste_dh(v, qs, Q, &in);
                d = in ? g : 0.f;
                if (c == iM) d += GaM;
                if (c == im) d += Gbt;
              }
              const float dn = a.s ? __fdiv_rn(d, se) : d;
              o[e] = rstd * (dn - x * rstd * mean_dot) + f4get(r4[jj], e);
            }
            if (a.dX) *reinterpret_cast<float4*>(a.dX + t * a.lddx + 4 * vi) = make_float4(o[0], o[1], o[2], o[3]);
            if (a.dXb) st_bf16x4(a.dXb + t * a.lddxb + 4 * vi, o);
          }
        }
      }
    }
    if (SUMS) {                                  // ds partial -sum(d X~) / s, ddelta partial -sum(d) / s
#pragma unroll
      for (int j = 0; j < VPT; ++j) {
        const int vi = j * NT + tid;
        if (vi < nv) {
          const float4 sv = (LETP && a.s) ? ld4(a.s + 4 * vi) : o4;
          float* ps = a.part_s + p * a.C + 4 * vi;
          float* pd = a.part_d + p * a.C + 4 * vi;
          float os[4], od[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            os[e] = -acc_s[(4 * j + e) % NE] / f4get(sv, e);
            od[e] = -acc_d[(4 * j + e) % NE] / f4get(sv, e);
          }
          *reinterpret_cast<float4*>(ps) = make_float4(os[0], os[1], os[2], os[3]);
          *reinterpret_cast<float4*>(pd) = make_float4(od[0], od[1], od[2], od[3]);
        }
      }
    }
  }
}

// ---- launchers ---------------------------------------------------------------------------------
template <int P, int NT>
static omq_status act_fwd_smem_go(cudaStream_t st, const ActFwdArgs& a) {
  auto kern = act_fwd_smem<P, NT>;
  const size_t smem = a.abits < 16 ? (size_t)a.C * 4 : 0;
  // With its static part a CTA has 48 KB without asking.  What is asked for is the longest row's, on every call: the
  // limit belongs to the current device, and one that followed the rows seen so far could be lowered by another
  // host thread between a call and its launch
  if (smem > 40 * 1024 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * 32 * 1024) != cudaSuccess)
    return OMQ_ERR_CUDA;
  kern<<<(unsigned)a.T, NT, smem, st>>>(a);
  OMQ_LAUNCH_CHECK();
  return OMQ_OK;
}

// Rows of up to 4 K columns and RMSNorm rows in registers, every other row of up to 32 K columns
// through shared memory: 256 threads while several rows fit an SM, 512 beyond, which overlap a row's own phases.
// 2048 rows with LET of 5120 columns 29 against 31 us, of 8192 44 and 40, of 16000 91 and 66; plain of 8192 31 and
// 27, of 28672 102 and 89 (1024 threads: 52, 58, 88, 38, 89).  SwiGLU rows, heavier an element, change later: of
// 11008 49 and 55 us, of 28672 129 with 512 and 136 with 1024.
template <int PRODUCER>
static omq_status act_fwd_dispatch(cudaStream_t st, const ActFwdArgs& a) {
  const int64_t nv = a.C / 4;
  if (nv > 1024 * 8) return OMQ_ERR_UNSUPPORTED;
  if constexpr (PRODUCER != AP_SWIGLU) {
    if (nv <= 128 * 8) {
      act_fwd_rows<PRODUCER, 128, 8, 8><<<(unsigned)a.T, 128, 0, st>>>(a);
      OMQ_LAUNCH_CHECK();
      return OMQ_OK;
    }
  }
  if constexpr (PRODUCER == AP_RMS_LET) {
    if (a.ldx % 4 != 0 || !omq_aligned16(a.X)) return OMQ_ERR_ALIGN;
    // the row-to-thread mapping fixes the RMS sum's order.  A CTA a row: persistent CTAs with a bulk-copied ring of
    // rows took 42 us for 2048 x 8192 with LET, a 70B block with this form 13 us less in each of its two
    if (nv <= 512 * 4) act_fwd_rows<PRODUCER, 512, 4, 3><<<(unsigned)a.T, 512, 0, st>>>(a);
    else if (nv <= 1024 * 4) act_fwd_rows<PRODUCER, 1024, 4, 1><<<(unsigned)a.T, 1024, 0, st>>>(a);
    else act_fwd_rows<PRODUCER, 1024, 8, 1><<<(unsigned)a.T, 1024, 0, st>>>(a);
    OMQ_LAUNCH_CHECK();
    return OMQ_OK;
  } else {
    if (a.C <= (PRODUCER == AP_SWIGLU ? 16 : 6) * 1024) return act_fwd_smem_go<PRODUCER, 256>(st, a);
    return act_fwd_smem_go<PRODUCER, 512>(st, a);
  }
}

template <int PRODUCER, int NT, int VPT, int JB, int MINB, bool SUMS, bool RD = false>
static omq_status act_bwd_go(cudaStream_t st, const ActBwdArgs& a0) {
  ActBwdArgs a = a0;
  // without column partials the rows per CTA are free: one wave of the CTAs that fit (SwiGLU rows, the longest,
  // one at a time: 16 us slower with four)
  if (!SUMS && PRODUCER != AP_SWIGLU) {
    const int64_t slots = (int64_t)MINB * omq_num_sms();
    a.rows_per_cta = (int)std::min<int64_t>(VPT > 12 ? 4 : VPT > 8 ? 2 : 8, (a.T + slots - 1) / slots);
  }
  const int64_t nparts = (a.T + a.rows_per_cta - 1) / a.rows_per_cta;
  act_bwd_stream<PRODUCER, NT, VPT, JB, MINB, SUMS, RD><<<(unsigned)nparts, NT, 0, st>>>(a);
  OMQ_LAUNCH_CHECK();
  return OMQ_OK;
}

// Row length -> threads and vectors per thread, up to 28 K columns.  Without LET column sums a row streams in
// batches of four vectors; the column sums keep 8 VPT accumulators per thread in registers (past 16 K columns
// 112 of them, of which 30 spill: 1531 x 28672 takes 334 us forward and backward, 1531 x 16384 160).
template <int PRODUCER>
static omq_status act_bwd_dispatch(cudaStream_t st, const ActBwdArgs& a) {
  const int64_t vpt = (a.C / 4 + 255) / 256;
  const bool sums = a.part_s != nullptr;
  if constexpr (PRODUCER == AP_PLAIN) {
    if (a.rowdot) {   // the row dot's partials take registers: loads in pairs to keep four CTAs per SM (two for longer rows)
      if (sums) return OMQ_ERR_UNSUPPORTED;
      if (vpt <= 4) return act_bwd_go<PRODUCER, 256, 4, 2, 4, false, true>(st, a);
      if (vpt <= 8) return act_bwd_go<PRODUCER, 256, 8, 4, 2, false, true>(st, a);
      if (vpt <= 16) return act_bwd_go<PRODUCER, 256, 16, 4, 2, false, true>(st, a);
      if (vpt <= 28) return act_bwd_go<PRODUCER, 256, 28, 4, 2, false, true>(st, a);
      return OMQ_ERR_UNSUPPORTED;
    }
  }
  if constexpr (PRODUCER == AP_SWIGLU) {
    return vpt <= 28 ? act_bwd_go<PRODUCER, 256, 28, 2, 4, false>(st, a) : OMQ_ERR_UNSUPPORTED;
  }
  if (!sums) {
    // four vectors' loads ahead with three CTAs a SM, which does not spill; the longest rows two with four
    if constexpr (PRODUCER == AP_PLAIN || PRODUCER == AP_LET)
      if (vpt > 12 && vpt <= 28) return act_bwd_go<PRODUCER, 256, 28, 2, 4, false>(st, a);
    if (vpt <= 4) return act_bwd_go<PRODUCER, 256, 4, 4, 3, false>(st, a);
    if (vpt <= 8) return act_bwd_go<PRODUCER, 256, 8, 4, 3, false>(st, a);
    if (vpt <= 12) return act_bwd_go<PRODUCER, 256, 12, 4, 3, false>(st, a);
    if constexpr (PRODUCER == AP_RMS_LET) {
      if (vpt <= 16) return act_bwd_go<PRODUCER, 256, 16, 4, 3, false>(st, a);
      if (vpt <= 28) return act_bwd_go<PRODUCER, 256, 28, 4, 3, false>(st, a);
    }
    return OMQ_ERR_UNSUPPORTED;
  }
  if constexpr (PRODUCER == AP_LET || PRODUCER == AP_RMS_LET) {
    if (vpt <= 4) return act_bwd_go<PRODUCER, 256, 4, 4, 2, true>(st, a);
    if (vpt <= 8) return act_bwd_go<PRODUCER, 512, 4, 4, 1, true>(st, a);
    if (vpt <= 12) return act_bwd_go<PRODUCER, 512, 6, 2, 1, true>(st, a);
    if (vpt <= 16) return act_bwd_go<PRODUCER, 512, 8, 2, 1, true>(st, a);
    if (vpt <= 28) return act_bwd_go<PRODUCER, 512, 14, 2, 1, true>(st, a);
  }
  return OMQ_ERR_UNSUPPORTED;
}

int act_bwd_rows(int64_t T, int64_t C, int at_least, int at_most) {
  const int64_t slots = (C <= 4096 ? 2 : 1) * (int64_t)omq_num_sms();
  return (int)std::min<int64_t>(at_most, std::max<int64_t>(at_least, (T + slots - 1) / slots));
}

omq_status act_fwd_launch(cudaStream_t st, const ActFwdArgs& a) {
  OMQ_REQUIRE(a.C % 8 == 0 && a.T > 0, OMQ_ERR_SHAPE);
  switch (a.producer) {
    case AP_PLAIN: return act_fwd_dispatch<AP_PLAIN>(st, a);
    case AP_LET: return act_fwd_dispatch<AP_LET>(st, a);
    case AP_RMS_LET: return act_fwd_dispatch<AP_RMS_LET>(st, a);
    case AP_SWIGLU: return act_fwd_dispatch<AP_SWIGLU>(st, a);
  }
  return OMQ_ERR_INVALID_ARG;
}

omq_status act_bwd_launch(cudaStream_t st, const ActBwdArgs& a0) {
  ActBwdArgs a = a0;
  OMQ_REQUIRE(a.C % 8 == 0 && a.T > 0, OMQ_ERR_SHAPE);
  OMQ_REQUIRE(!a.rowdot || (a.producer == AP_PLAIN && a.dXb && a.C % 128 == 0 && a.ldrow >= a.T), OMQ_ERR_INVALID_ARG);
  if (a.rows_per_cta <= 0) a.rows_per_cta = 4;
  switch (a.producer) {
    case AP_PLAIN: return act_bwd_dispatch<AP_PLAIN>(st, a);
    case AP_LET: return act_bwd_dispatch<AP_LET>(st, a);
    case AP_RMS_LET: return act_bwd_dispatch<AP_RMS_LET>(st, a);
    case AP_SWIGLU: return act_bwd_dispatch<AP_SWIGLU>(st, a);
  }
  return OMQ_ERR_INVALID_ARG;
}

// ================================================================================================
// q, k, v: RoPE (rotate-half pairs), [Q, K] LET (Eq. 5: Q~ = q / s_a, K~ = k * s_a), per-token Q_a
// A pair is float4 p % 16 of the first half of head p / 16 and its partner 64 elements later, so the
// rotation and its transpose stay in registers.  Thread tid owns the pairs j*NT + tid; NT is a multiple
// of 16, so all of them turn by the same four angles.
// ================================================================================================
__device__ __forceinline__ int pair_elem(int p) { return (p >> 4) * 128 + 4 * (p & 15); }   // its first element
// the rounding is spelled out, so that the backward re-forms the forward's values bit for bit
__device__ __forceinline__ void rope_pair(float a1, float a2, float c, float s, float& r1, float& r2) {
  r1 = fmaf(a1, c, -__fmul_rn(a2, s));
  r2 = fmaf(a2, c, __fmul_rn(a1, s));
}

// One CTA per (token, q | k | v), the segment in registers: bound by the row's own latency (loads, two
// barriers), hence few registers, every load in float4s and the rounding off the conversion pipe.  The
// exact division stays the IEEE one: with one row a CTA a reciprocal of s_a would serve only once.  2048 rows of
// 3 x 32 heads with LET take 32 us, of 64 + 8 + 8 heads 42 (55 and 93 with scalar s_a loads and six barriers).
template <int NT, int PPT>
__global__ void __launch_bounds__(NT) qkv_fwd_rows(QkvArgs a) {
  constexpr int NW = NT / 32;
  __shared__ float red[2][NW];
  __shared__ int sidx[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t = blockIdx.x, seg = blockIdx.y;
  const int dq = a.H * a.hd, dkv = a.Hkv * a.hd;
  const int np = (seg == 0 ? a.H : a.Hkv) * 16;
  const float* base = a.Y + (int64_t)t * a.ldy + (seg == 0 ? 0 : (seg == 1 ? dq : dq + dkv));
  const float* sa = seg == 0 ? a.sa_exp : a.sa;
  const bool let = seg < 2 && a.sa_exp != nullptr;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  if (tid == 0) { sidx[0] = OMQ_NO_INDEX; sidx[1] = OMQ_NO_INDEX; }
  float4 ca = z4, cb = z4, x1[PPT], x2[PPT];
  if (seg < 2) {                                       // (cos, sin) of the four frequencies
    const float* cs = a.cs + (int64_t)t * 128 + 8 * (tid & 15);
    ca = ld4(cs); cb = ld4(cs + 4);
  }
#pragma unroll
  for (int j = 0; j < PPT; ++j) {                      // every load first
    const int p = j * NT + tid;
    x1[j] = p < np ? ld4(base + pair_elem(p)) : z4;
    x2[j] = p < np ? ld4(base + pair_elem(p) + 64) : z4;
  }
  const float cv[4] = {ca.x, ca.z, cb.x, cb.z}, sv[4] = {ca.y, ca.w, cb.y, cb.w};
  float v1[PPT][4], v2[PPT][4];
  float lM = -INFINITY, lm = INFINITY;                 // this thread's own extremes
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int p = j * NT + tid;
    if (p >= np) continue;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      v1[j][e] = f4get(x1[j], e);
      v2[j][e] = f4get(x2[j], e);
      if (seg < 2) rope_pair(f4get(x1[j], e), f4get(x2[j], e), cv[e], sv[e], v1[j][e], v2[j][e]);
    }
    if (let) {
      const float4 s1 = ld4(sa + pair_elem(p)), s2 = ld4(sa + pair_elem(p) + 64);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v1[j][e] = seg == 0 ? __fdiv_rn(v1[j][e], f4get(s1, e)) : __fmul_rn(v1[j][e], f4get(s1, e));
        v2[j][e] = seg == 0 ? __fdiv_rn(v2[j][e], f4get(s2, e)) : __fmul_rn(v2[j][e], f4get(s2, e));
      }
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      lM = fmaxf(lM, fmaxf(v1[j][e], v2[j][e]));
      lm = fminf(lm, fminf(v1[j][e], v2[j][e]));
    }
  }
  const bool quant = a.abits < 16;
  const float Q = (float)((1 << (quant ? a.abits : 1)) - 1);
  QState qs{};
  bool small = false;
  if (quant) {
    float M = lM, m = lm;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
      m = fminf(m, __shfl_xor_sync(0xffffffffu, m, off));
    }
    if (lane == 0) { red[0][warp] = M; red[1][warp] = m; }
    __syncthreads();
    M = red[0][0]; m = red[1][0];
#pragma unroll
    for (int w = 1; w < NW; ++w) { M = fmaxf(M, red[0][w]); m = fminf(m, red[1][w]); }
    if (lM == M || lm == m) {                          // only the holders of an extreme search its first index
      int iM = OMQ_NO_INDEX, im = OMQ_NO_INDEX;
#pragma unroll
      for (int j = 0; j < PPT; ++j) {
        const int p = j * NT + tid;
        if (p >= np) continue;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (v1[j][e] == M) iM = min(iM, pair_elem(p) + e);
          if (v2[j][e] == M) iM = min(iM, pair_elem(p) + 64 + e);
          if (v1[j][e] == m) im = min(im, pair_elem(p) + e);
          if (v2[j][e] == m) im = min(im, pair_elem(p) + 64 + e);
        }
      }
      if (iM != OMQ_NO_INDEX) atomicMin(&sidx[0], iM);
      if (im != OMQ_NO_INDEX) atomicMin(&sidx[1], im);
    }
    qs = omq_qstate(M, m, 1.f, 1.f, Q, a.eps);
    small = omq_small_quot(qs);
  }
  __nv_bfloat16* out = seg == 0 ? a.Qh + (int64_t)t * dq : (seg == 1 ? a.Kh : a.Vh) + (int64_t)t * dkv;
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int p = j * NT + tid;
    if (p >= np) continue;
    if (quant) {
      float cd[4];
      if (small) { quant4<true>(v1[j], qs, Q, cd); quant4<true>(v2[j], qs, Q, cd); }
      else { quant4<false>(v1[j], qs, Q, cd); quant4<false>(v2[j], qs, Q, cd); }
    }
    st_bf16x4(out + pair_elem(p), v1[j]);
    st_bf16x4(out + pair_elem(p) + 64, v2[j]);
  }
  if (!quant) return;
  __syncthreads();                                     // first indices final
  if (tid == 0) {
    const int64_t k = (int64_t)seg * a.T + t;
    a.h[k] = qs.h; a.z[k] = (int32_t)qs.z;
    a.imax[k] = omq_saved_index(sidx[0], 0); a.imin[k] = omq_saved_index(sidx[1], 0);
  }
}

// Backward of the q, k, v chain: one pass over a row writes the gradient with the in-range mask applied
// and sums the h path; the owner of each routed pair (the first max / min and its RoPE partner) then
// rewrites that pair with the routing added.
//
// A CTA owns the pairs of all three segments (q | k | v; with odd head counts a warp holds some of two), or of one where
// three do not fit 512 threads x 4 pairs, and walks a slab of rows, the next one prefetched into L2.  The
// quantizer states and the routed pairs of several rows are formed together, one warp each, so a row has no
// chain of dependent loads and one barrier.  1/s_a of the thread's query columns is formed once a CTA: it
// scales the gradient and gives the exact division of the quantizer input (omq_div2).  2048 rows of 3 x 32 heads
// 71 us, of 64 + 8 + 8 heads 71 (83 and 198 with the chain and two barriers in each row); half of what is left
// is issue slots (50 instructions an element), the rest the latency of the loads at 16 warps a SM.
struct QkvRowState {
  float h, z, rh, u;
  int floored, small, iM, im;
  int first[2];              // the routed pair's element in the first half-head, within its segment
  float r1[2], r2[2], v1[2], v2[2], g1[2], g2[2], c[2], s[2], s1[2], s2[2];
};
constexpr int kQkvGroup = 16;          // rows whose states are formed, and whose routed pairs are rewritten, together

// Two lanes form the state of segment seg of row t: the even one the max's pair, the odd one the min's.
__device__ __forceinline__ void qkv_row_state(const QkvArgs& a, int seg, int t, float Q, int r, uint32_t lanes, QkvRowState& o) {
  const int dq = a.H * a.hd, dkv = a.Hkv * a.hd;
  const int off = seg == 0 ? 0 : (seg == 1 ? dq : dq + dkv);
  const bool rope = seg < 2, let = rope && a.sa_exp != nullptr;
  const float* sa = seg == 0 ? a.sa_exp : a.sa;
  const int64_t kq = (int64_t)seg * a.T + t;
  const int c = r == 0 ? a.imax[kq] : a.imin[kq];
  const int first = (c & ~127) + (c & 63), f = first & 63;
  const float* y = a.Y + (int64_t)t * a.ldy + off + first;
  const float* g = a.dQKV + (int64_t)t * a.ldd + off + first;
  const float y1 = y[0], y2 = y[64], g1 = g[0], g2 = g[64];
  const float cv = rope ? a.cs[(int64_t)t * 128 + 2 * f] : 1.f, sv = rope ? a.cs[(int64_t)t * 128 + 2 * f + 1] : 0.f;
  const float s1 = let ? sa[first] : 1.f, s2 = let ? sa[first + 64] : 1.f;
  float r1 = y1, r2 = y2;
  if (rope) rope_pair(y1, y2, cv, sv, r1, r2);
  float v1 = r1, v2 = r2;
  if (let) {
    v1 = seg == 0 ? __fdiv_rn(r1, s1) : __fmul_rn(r1, s1);
    v2 = seg == 0 ? __fdiv_rn(r2, s2) : __fmul_rn(r2, s2);
  }
  const float v = (c & 64) ? v2 : v1;
  const float w = __shfl_xor_sync(lanes, v, 1);
  o.first[r] = first; o.r1[r] = r1; o.r2[r] = r2; o.v1[r] = v1; o.v2[r] = v2; o.g1[r] = g1; o.g2[r] = g2;
  o.c[r] = cv; o.s[r] = sv; o.s1[r] = s1; o.s2[r] = s2;
  if (r == 1) {
    o.im = c;
    return;
  }
  o.iM = c;
  QState qs = omq_qstate(v, w, 1.f, 1.f, Q, a.eps);
  qs.h = a.h[kq]; qs.z = (float)a.z[kq]; qs.rh = __frcp_rn(qs.h);
  o.h = qs.h; o.z = qs.z; o.rh = qs.rh; o.u = __fmul_rn(w, qs.rh);
  o.floored = qs.floored; o.small = omq_small_quot(qs) ? 1 : 0;
}

template <int NT, int PPT, int MINB>
__global__ void __launch_bounds__(NT, MINB) qkv_bwd_rows(QkvArgs a) {
  constexpr int NW = NT / 32, JB = PPT % 3 == 0 ? 3 : PPT < 2 ? 1 : 2;
  static_assert(PPT % JB == 0, "whole batches");
  extern __shared__ float4 rs_sm[];                    // [PPT][2][NT]: 1/s_a of the thread's own columns
  __shared__ QkvRowState rows_sm[kQkvGroup][3];
  __shared__ float2 red[kQkvGroup][3][NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int dq = a.H * a.hd, dkv = a.Hkv * a.hd;
  const int b0 = a.H * 16, b1 = b0 + a.Hkv * 16, b2 = b1 + a.Hkv * 16;   // the segments' ends, in pairs
  const int seg0 = gridDim.y == 1 ? 0 : (int)blockIdx.y, nseg = gridDim.y == 1 ? 3 : 1;
  const int lo = seg0 == 0 ? 0 : (seg0 == 1 ? b0 : b1);
  const int hi = nseg == 3 ? b2 : (seg0 == 0 ? b0 : (seg0 == 1 ? b1 : b2));
  const bool sums = a.part_q != nullptr;
  const bool quant = a.abits < 16;
  const float Q = (float)((1 << (quant ? a.abits : 1)) - 1);
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  const int t0 = blockIdx.x * a.rows_per_cta, t1 = min(a.T, t0 + a.rows_per_cta);
  auto prefetch = [&](int t) {
    omq_l2_prefetch(a.Y + (int64_t)t * a.ldy + 8 * lo, (uint64_t)(hi - lo) * 32);
    omq_l2_prefetch(a.dQKV + (int64_t)t * a.ldd + 8 * lo, (uint64_t)(hi - lo) * 32);
  };
  if (tid == 0) {
    prefetch(t0);
    if (t0 + 1 < t1) prefetch(t0 + 1);
  }
  float acc1[PPT][4], acc2[PPT][4];
  bool s_ok = a.sa_exp != nullptr;
#pragma unroll
  for (int j = 0; j < PPT; ++j) {
    const int g = lo + j * NT + tid;
#pragma unroll
    for (int e = 0; e < 4; ++e) { acc1[j][e] = 0.f; acc2[j][e] = 0.f; }
    if (a.sa_exp && g < b0) {
      const float4 s1 = ld4(a.sa_exp + pair_elem(g)), s2 = ld4(a.sa_exp + pair_elem(g) + 64);
      s_ok = s_ok && omq_div_ok(s1.x) && omq_div_ok(s1.y) && omq_div_ok(s1.z) && omq_div_ok(s1.w);
      s_ok = s_ok && omq_div_ok(s2.x) && omq_div_ok(s2.y) && omq_div_ok(s2.z) && omq_div_ok(s2.w);
      rs_sm[(2 * j) * NT + tid] = make_float4(__frcp_rn(s1.x), __frcp_rn(s1.y), __frcp_rn(s1.z), __frcp_rn(s1.w));
      rs_sm[(2 * j + 1) * NT + tid] = make_float4(__frcp_rn(s2.x), __frcp_rn(s2.y), __frcp_rn(s2.z), __frcp_rn(s2.w));
    }
  }
  // X~ of four query elements from their rotated values, as the forward formed them
  auto div4 = [&](const float (&r)[4], const float4 s, const float4 rs, float (&v)[4]) {
    const uint32_t key = max(max(omq_div_key(r[0]), omq_div_key(r[1])), max(omq_div_key(r[2]), omq_div_key(r[3])));
    if (s_ok && key < OMQ_DIV_KEYS) {
      const float2 q0 = omq_div2(make_float2(r[0], r[1]), make_float2(s.x, s.y), make_float2(rs.x, rs.y));
      const float2 q1 = omq_div2(make_float2(r[2], r[3]), make_float2(s.z, s.w), make_float2(rs.z, rs.w));
      v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = __fdiv_rn(r[e], f4get(s, e));
    }
  };
  for (int tg = t0; tg < t1; tg += kQkvGroup) {
  const int n = min(kQkvGroup, t1 - tg);
  if (quant) {
    __syncthreads();                                    // the previous group's states and sums have been used
    const int k = tid >> 1;                             // two lanes a state
    const uint32_t lanes = __ballot_sync(0xffffffffu, k < n * nseg);
    if (k < n * nseg) {
      const int seg = nseg == 3 ? k % 3 : seg0, i = k / nseg;
      qkv_row_state(a, seg, tg + i, Q, tid & 1, lanes, rows_sm[i][seg]);
    }
    __syncthreads();
  }
  for (int t = tg; t < tg + n; ++t) {                   // no barrier between rows: the warps drift apart
    if (tid == 0 && t + 2 < t1) prefetch(t + 2);
    const QkvRowState* S3 = rows_sm[t - tg];
    const float* yr = a.Y + (int64_t)t * a.ldy;
    const float* gr = a.dQKV + (int64_t)t * a.ldd;
    __nv_bfloat16* dyb = a.dYb + (int64_t)t * a.ldy;
    const float* csr = a.cs + (int64_t)t * 128 + 8 * (tid & 15);
    const float4 ca = ld4(csr), cb = ld4(csr + 4);
    const float cv[4] = {ca.x, ca.z, cb.x, cb.z}, sv[4] = {ca.y, ca.w, cb.y, cb.w};
    float Gh0 = 0.f, Gh1 = 0.f, Gh2 = 0.f, Gb0 = 0.f, Gb1 = 0.f, Gb2 = 0.f;
#pragma unroll
    for (int jb = 0; jb < PPT; jb += JB) {
      float4 x1[JB], x2[JB], g1[JB], g2[JB];
#pragma unroll
      for (int jj = 0; jj < JB; ++jj) {                 // every load of the batch first
        const int g = lo + (jb + jj) * NT + tid;
        const bool ok = g < hi;
        x1[jj] = ok ? ld4(yr + pair_elem(g)) : z4;
        x2[jj] = ok ? ld4(yr + pair_elem(g) + 64) : z4;
        g1[jj] = ok ? ld4(gr + pair_elem(g)) : z4;
        g2[jj] = ok ? ld4(gr + pair_elem(g) + 64) : z4;
      }
#pragma unroll
      for (int jj = 0; jj < JB; ++jj) {
        const int j = jb + jj;
        const int g = lo + j * NT + tid;
        if (g >= hi) continue;
        const int seg = g < b0 ? 0 : (g < b1 ? 1 : 2);
        const bool rope = seg < 2, let = rope && a.sa_exp != nullptr;
        float r1[4], r2[4], v1[4], v2[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          r1[e] = f4get(x1[jj], e);
          r2[e] = f4get(x2[jj], e);
          if (rope) rope_pair(f4get(x1[jj], e), f4get(x2[jj], e), cv[e], sv[e], r1[e], r2[e]);
          v1[e] = r1[e]; v2[e] = r2[e];
        }
        float4 m1 = z4, m2 = z4;                        // what the gradient is multiplied by: 1/s_a (q), s_a (k)
        if (let && seg == 0) {
          m1 = rs_sm[(2 * j) * NT + tid]; m2 = rs_sm[(2 * j + 1) * NT + tid];
          div4(r1, ld4(a.sa_exp + pair_elem(g)), m1, v1);
          div4(r2, ld4(a.sa_exp + pair_elem(g) + 64), m2, v2);
        } else if (let) {
          m1 = ld4(a.sa + pair_elem(g - b0)); m2 = ld4(a.sa + pair_elem(g - b0) + 64);
#pragma unroll
          for (int e = 0; e < 4; ++e) { v1[e] = __fmul_rn(r1[e], f4get(m1, e)); v2[e] = __fmul_rn(r2[e], f4get(m2, e)); }
        }
        float d1[4] = {g1[jj].x, g1[jj].y, g1[jj].z, g1[jj].w}, d2[4] = {g2[jj].x, g2[jj].y, g2[jj].z, g2[jj].w};
        if (quant) {
          const QkvRowState& S = S3[seg];
          QState qs{};
          qs.h = S.h; qs.z = S.z; qs.rh = S.rh; qs.u = S.u;
          const bool small = S.small != 0;
          float gh = 0.f, gb = 0.f;
          auto ste = [&](const float (&v)[4], float (&d)[4]) {
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
              int i0 = 0, i1 = 0;
              const float2 w = make_float2(v[e], v[e + 1]);
              const float2 dh = small ? omq_ste_dh2_small(w, qs, Q, &i0, &i1) : omq_ste_dh2(w, qs, Q, &i0, &i1);
              gh = fmaf(d[e], dh.x, gh);
              gh = fmaf(d[e + 1], dh.y, gh);
              if (!i0) { gb += d[e]; d[e] = 0.f; }
              if (!i1) { gb += d[e + 1]; d[e + 1] = 0.f; }
            }
          };
          ste(v1, d1);
          ste(v2, d2);
          if (seg == 0) { Gh0 += gh; Gb0 += gb; }
          else if (seg == 1) { Gh1 += gh; Gb1 += gb; }
          else { Gh2 += gh; Gb2 += gb; }
        }
        if (let) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            // q: the 1/s_a of the ds_a terms is applied once, at the end
            const float w1 = seg == 0 ? -v1[e] : r1[e], w2 = seg == 0 ? -v2[e] : r2[e];
            acc1[j][e] = fmaf(d1[e], w1, acc1[j][e]);
            acc2[j][e] = fmaf(d2[e], w2, acc2[j][e]);
            d1[e] = __fmul_rn(d1[e], f4get(m1, e));
            d2[e] = __fmul_rn(d2[e], f4get(m2, e));
          }
        }
        float o1[4], o2[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          o1[e] = rope ? d1[e] * cv[e] + d2[e] * sv[e] : d1[e];
          o2[e] = rope ? d2[e] * cv[e] - d1[e] * sv[e] : d2[e];
        }
        st_bf16x4(dyb + pair_elem(g), o1);
        st_bf16x4(dyb + pair_elem(g) + 64, o2);
      }
    }
    if (!quant) continue;
#pragma unroll
    for (int sg = 0; sg < 3; ++sg) {
      if (sg < seg0 || sg >= seg0 + nseg) continue;
      const float h = warp_sum(sg == 0 ? Gh0 : (sg == 1 ? Gh1 : Gh2)), b = warp_sum(sg == 0 ? Gb0 : (sg == 1 ? Gb1 : Gb2));
      if (lane == 0) red[t - tg][sg][warp] = make_float2(h, b);
    }
  }
  if (!quant) continue;
  __syncthreads();
  // ---- the routed pairs, rewritten with the routing by their owners ----
  for (int i = 0; i < n; ++i) {
    const int t = tg + i;
    for (int sg = seg0; sg < seg0 + nseg; ++sg) {
      const QkvRowState& S = rows_sm[i][sg];
      const int sb = sg == 0 ? 0 : (sg == 1 ? b0 : b1);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int first = S.first[r];
        if (r == 1 && S.first[0] == first) break;        // same pair: already done
        const int g = sb + (first >> 7) * 16 + ((first & 63) >> 2);
        if ((g - lo) % NT != tid) continue;
        float h = 0.f, b = 0.f;
#pragma unroll
        for (int w = 0; w < NW; ++w) { h += red[i][sg][w].x; b += red[i][sg][w].y; }
        const float GaM = (S.floored ? 0.f : h) / Q, Gbt = b - GaM;
        float ro1 = 0.f, ro2 = 0.f;                      // routing of each element of the pair
        if (first == S.iM) ro1 += GaM;
        if (first == S.im) ro1 += Gbt;
        if (first + 64 == S.iM) ro2 += GaM;
        if (first + 64 == S.im) ro2 += Gbt;
        QState qs{};
        qs.h = S.h; qs.z = S.z; qs.rh = S.rh; qs.u = S.u;
        int in1 = 0, in2 = 0;
        omq_ste_dh(S.v1[r], qs, Q, &in1);
        omq_ste_dh(S.v2[r], qs, Q, &in2);
        float d1 = (in1 ? S.g1[r] : 0.f) + ro1, d2 = (in2 ? S.g2[r] : 0.f) + ro2;
        const bool rope = sg < 2, let = rope && a.sa_exp != nullptr;
        if (let) {
          const int jr = (g - lo) / NT, er = first & 3;
          const float w1 = sg == 0 ? -S.v1[r] : S.r1[r], w2 = sg == 0 ? -S.v2[r] : S.r2[r];
#pragma unroll
          for (int j = 0; j < PPT; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e)
              if (j == jr && e == er) {
                acc1[j][e] = fmaf(ro1, w1, acc1[j][e]);
                acc2[j][e] = fmaf(ro2, w2, acc2[j][e]);
              }
          d1 = sg == 0 ? __fdiv_rn(d1, S.s1[r]) : __fmul_rn(d1, S.s1[r]);
          d2 = sg == 0 ? __fdiv_rn(d2, S.s2[r]) : __fmul_rn(d2, S.s2[r]);
        }
        const float cr = S.c[r], sr = S.s[r];
        __nv_bfloat16* o = a.dYb + (int64_t)t * a.ldy + 8 * sb + first;
        o[0] = f_to_bf16(rope ? d1 * cr + d2 * sr : d1);
        o[64] = f_to_bf16(rope ? d2 * cr - d1 * sr : d2);
      }
    }
  }
  }
  if (sums) {
#pragma unroll
    for (int j = 0; j < PPT; ++j) {
      const int g = lo + j * NT + tid;
      if (g >= hi || g >= b1) continue;
      if (g < b0) {
        const float4 m1 = rs_sm[(2 * j) * NT + tid], m2 = rs_sm[(2 * j + 1) * NT + tid];
#pragma unroll
        for (int e = 0; e < 4; ++e) { acc1[j][e] *= f4get(m1, e); acc2[j][e] *= f4get(m2, e); }
      }
      float* o = g < b0 ? a.part_q + (int64_t)blockIdx.x * dq + pair_elem(g) : a.part_k + (int64_t)blockIdx.x * dkv + pair_elem(g - b0);
      *reinterpret_cast<float4*>(o) = make_float4(acc1[j][0], acc1[j][1], acc1[j][2], acc1[j][3]);
      *reinterpret_cast<float4*>(o + 64) = make_float4(acc2[j][0], acc2[j][1], acc2[j][2], acc2[j][3]);
    }
  }
}

// The pairs of a CTA: one segment's where the three are equally long, else all of them up to 2048 (a CTA for each
// of a grouped-query row's segments would leave most threads of two of them idle: 2048 x (64 + 8 + 8 heads) 95 us
// against 79; 2048 x 3 x 32 heads 76 and 80).
static bool qkv_bwd_split(int H, int Hkv) { return H == Hkv || (H + 2 * Hkv) * 16 > 2048; }
static int qkv_bwd_pairs(int H, int Hkv) { return (qkv_bwd_split(H, Hkv) ? H : H + 2 * Hkv) * 16; }
static int qkv_bwd_rows_per_cta(int T, int H, int Hkv) {
  const int n = qkv_bwd_pairs(H, Hkv);
  const int slots = (n <= 256 ? 4 : n <= 768 ? 2 : 1) * omq_num_sms() / (qkv_bwd_split(H, Hkv) ? 3 : 1);
  return std::min(32, std::max(2, (T + slots - 1) / slots));
}
// token rows per CTA: one wave; the ds_a partials have one row per CTA
int64_t qkv_bwd_nslab(int T, int H, int Hkv) {
  const int r = qkv_bwd_rows_per_cta(T, H, Hkv);
  return (T + r - 1) / r;
}

omq_status qkv_fwd_launch(cudaStream_t st, const QkvArgs& a) {
  OMQ_REQUIRE(a.hd == 128, OMQ_ERR_UNSUPPORTED);
  const int np = a.H * 16;
  const dim3 grid((unsigned)a.T, 3);
  if (np <= 512) qkv_fwd_rows<128, 4><<<grid, 128, 0, st>>>(a);
  else if (np <= 1024) qkv_fwd_rows<256, 4><<<grid, 256, 0, st>>>(a);
  else if (np <= 2048) qkv_fwd_rows<512, 4><<<grid, 512, 0, st>>>(a);
  else return OMQ_ERR_UNSUPPORTED;
  OMQ_LAUNCH_CHECK();
  return OMQ_OK;
}

template <int NT, int PPT, int MINB>
static omq_status qkv_bwd_go(cudaStream_t st, const QkvArgs& a) {
  auto kern = qkv_bwd_rows<NT, PPT, MINB>;
  const size_t smem = a.sa_exp ? (size_t)PPT * 2 * NT * sizeof(float4) : 0;
  if (smem > 24 * 1024 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return OMQ_ERR_CUDA;
  const unsigned y = qkv_bwd_split(a.H, a.Hkv) ? 3 : 1;
  kern<<<dim3((unsigned)qkv_bwd_nslab(a.T, a.H, a.Hkv), y), NT, smem, st>>>(a);
  OMQ_LAUNCH_CHECK();
  return OMQ_OK;
}

omq_status qkv_bwd_launch(cudaStream_t st, const QkvArgs& a0) {
  QkvArgs a = a0;
  OMQ_REQUIRE(a.hd == 128, OMQ_ERR_UNSUPPORTED);
  a.rows_per_cta = qkv_bwd_rows_per_cta(a.T, a.H, a.Hkv);
  const int n = qkv_bwd_pairs(a.H, a.Hkv);
  if (n <= 256) return qkv_bwd_go<256, 1, 4>(st, a);
  if (n <= 512) return qkv_bwd_go<256, 2, 2>(st, a);
  if (n <= 768) return qkv_bwd_go<256, 3, 2>(st, a);
  if (n <= 1024) return qkv_bwd_go<512, 2, 1>(st, a);
  if (n <= 1536) return qkv_bwd_go<512, 3, 1>(st, a);
  if (n <= 2048) return qkv_bwd_go<512, 4, 1>(st, a);
  return OMQ_ERR_UNSUPPORTED;
}
