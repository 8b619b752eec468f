// Input-dependent gate (paper Eq. 18 with a one-layer F_o) on the tensor-core attention kernels.
//
// alpha_t = sigmoid(<w_lt, O_lt,t> + <w_st, O_st,t> + b), O_t = alpha_t O_lt,t + (1 - alpha_t) O_st,t.
// The attention kernels themselves know a gate weight per row only through the per-row records of
// the backward pre-pass; everything else the gate needs is row-local or can be put into the
// tensors those kernels read:
//   forward   the attention kernel produces O_lt, O_st (and the log-sum-exps) as in training mode;
//             a row-wise kernel here forms alpha_t from them and writes O.
//   backward  with c_t = alpha_t (1 - alpha_t) <G_t, O_lt,t - O_st,t> the upstream gradients of the
//             two branches are alpha_t (G_t + kL_t w_lt) and (1 - alpha_t) (G_t + kS_t w_st) with
//             kL_t = c_t / alpha_t, kS_t = c_t / (1 - alpha_t).  They differ by more than a factor,
//             so the backward kernels run once per branch: pass 1 with the tensor G + kL w_lt in
//             place of dO, tile lists of the long-term branch only and records that carry alpha_t
//             in the exponent and switch the short-term branch off; pass 2 likewise for the
//             short-term branch, adding to the first pass's gradients as it writes them.  The
//             gradient of F_o's parameters is row-local (dw_lt = sum_t c_t O_lt,t, dw_st likewise,
//             db = sum_t c_t) and is accumulated here in double precision, per query block, for the
//             fixed-order reduction of gate_param_grad_kernel.
// The branch outputs entering F_o are the stored (bf16) rows.
#include "tc_common.cuh"

namespace blossom {
namespace tc {
namespace {

typedef __nv_bfloat16 bf;

__device__ __forceinline__ void unpack8(const uint4 &v, float (&x)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    x[2 * e] = __uint_as_float(w[e] << 16);
    x[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
  }
}
__device__ __forceinline__ uint4 pack8(const float (&x)[8]) {
  return make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]), pack_bf16(x[6], x[7]));
}
// sum over the LPR lanes that share a row (LPR a power of two, rows aligned in the warp)
template <int LPR>
__device__ __forceinline__ float row_sum(float a) {
#pragma unroll
  for (int o = LPR / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  return a;
}
// F_o's parameters of head h are 2 D + 1 floats: an odd count, so rows of it are not 16-byte aligned
__device__ __forceinline__ void load_w8(const float *p, float (&w)[8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) w[e] = p[e];
}
__device__ __forceinline__ void gate_of_row(float a, float &alpha, float &beta) {
  // both from the same exponential, so that alpha + beta = 1 to rounding and neither underflows first
  const float e = __expf(-fabsf(a));
  const float big = 1.f / (1.f + e), small = e / (1.f + e);
  alpha = a >= 0.f ? big : small;
  beta = a >= 0.f ? small : big;
}

// ---- forward: O = alpha_t O_lt + (1 - alpha_t) O_st -------------------------------------------
// D / 8 lanes per row, one 16-byte chunk each.  Padded rows hold zeros in both branches.
template <int D>
__global__ void __launch_bounds__(256) gate_mix_kernel(Shape s, const float *__restrict__ gate,
                                                       const bf *__restrict__ out_lt, const bf *__restrict__ out_st,
                                                       bf *__restrict__ out) {
  grid_chain_enter();
  constexpr int LPR = D / 8, RPB = 256 / LPR;
  const int blocks_per_unit = (s.L + RPB - 1) / RPB;
  const int u = blockIdx.x / blocks_per_unit, n = u / s.H, h = u % s.H;
  const int t = (blockIdx.x % blocks_per_unit) * RPB + threadIdx.x / LPR, ch = threadIdx.x % LPR;
  const float *gw = gate + (int64_t)h * (2 * D + 1);
  float wl[8], wsv[8], ol[8] = {0, 0, 0, 0, 0, 0, 0, 0}, os[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  load_w8(gw + ch * 8, wl);
  load_w8(gw + D + ch * 8, wsv);
  const bool row = t < s.L;
  const int64_t off = row ? row_offset(s, n, h, t) + ch * 8 : 0;
  if (row) {
    unpack8(*reinterpret_cast<const uint4 *>(out_lt + off), ol);
    unpack8(*reinterpret_cast<const uint4 *>(out_st + off), os);
  }
  float a = 0.f;
#pragma unroll
  for (int e = 0; e < 8; ++e) a = fmaf(wl[e], ol[e], fmaf(wsv[e], os[e], a));
  a = row_sum<LPR>(a) + gw[2 * D];
  float alpha, beta;
  gate_of_row(a, alpha, beta);
  if (row) {
    float o[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) o[e] = alpha * ol[e] + beta * os[e];
    *reinterpret_cast<uint4 *>(out + off) = pack8(o);
  }
}

// ---- backward pre-pass --------------------------------------------------------------------------
// One CTA per (batch, head, gate_prep_rows rows).  Bound by the tail of a CTA (the double-precision sums of the
// parameters' gradient, 2 D + 1 of them, over lanes and warps) and then by memory: with a CTA per query block a thread
// had one row for each such tail, and 129 partial sums per 32 rows went to memory and back (B 16, H 4, L 900, D 64
// 19.0 us and 8.5 in the kernel that adds the partials; four rows a thread, the next loaded ahead, 13.3 and 4.2; B 64
// 72 and 40 -> 43 and 13; three CTAs an SM instead of two spill: 19.1).  Per row: alpha_t, c_t, the two upstream tensors (bf16,
// zeros in padded rows: the attention kernels multiply them by exact zeros, which must stay
// zeros), the records of the two passes (layout of bwd_prep_kernel; Delta of a pass is taken with
// the rounded tensor the pass multiplies with, and the branch a pass leaves out gets the exponent
// offset -1e30, i.e. probability 0), and the partial sums of the parameter gradient.
template <int D>
__global__ void __launch_bounds__(256) gate_prep_kernel(Shape s, const float *__restrict__ gate,
                                                        const int32_t *__restrict__ seq_lens,
                                                        const bf *__restrict__ out_lt, const bf *__restrict__ out_st,
                                                        const float *__restrict__ lse, const bf *__restrict__ dout,
                                                        bf *__restrict__ g_lt, bf *__restrict__ g_st,
                                                        float4 *__restrict__ rec_lt, float4 *__restrict__ rec_st,
                                                        double *__restrict__ dgate_part, int Lpad, int rows, int parts,
                                                        int32_t *__restrict__ status) {
  grid_release();  // (no wait here: the tile lists' kernel before it, of which it needs nothing, waits first and lets it start then)
  if (blockIdx.x == 0 && threadIdx.x < 4) status[threadIdx.x] = 0;  // the backward's status words
  constexpr int LPR = D / 8, RPB = 256 / LPR, GW = 2 * D + 1;
  __shared__ double red[8][GW];
  const int u = blockIdx.x / parts, qb = blockIdx.x % parts, n = u / s.H, h = u % s.H;
  const int lr = threadIdx.x / LPR, ch = threadIdx.x % LPR;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len;
  const float *gw = gate + (int64_t)h * GW;
  float wl[8], wsv[8];
  load_w8(gw + ch * 8, wl);
  load_w8(gw + D + ch * 8, wsv);
  const float bias = gw[2 * D];
  const int64_t BHL = (int64_t)s.B * s.H * s.L;
  double acc[16], accB = 0.0;  // eight columns of O_lt, eight of O_st
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e] = 0.0;
  // the last CTA of a head also writes the (zero) records of the rows that pad L to a multiple of 64
  const int t_end = qb == parts - 1 ? Lpad : (qb + 1) * rows;
  uint4 next[3];  // the next row's pieces of dO, O_lt, O_st, loaded a row ahead
  auto load = [&](int t) {
    next[0] = next[1] = next[2] = make_uint4(0u, 0u, 0u, 0u);
    if (t >= pad0 && t < min(t_end, s.L)) {
      const int64_t off = row_offset(s, n, h, t) + ch * 8;
      next[0] = *reinterpret_cast<const uint4 *>(dout + off);
      next[1] = *reinterpret_cast<const uint4 *>(out_lt + off);
      next[2] = *reinterpret_cast<const uint4 *>(out_st + off);
    }
  };
  load(qb * rows + lr);
#pragma unroll 1
  for (int t0 = qb * rows; t0 < t_end; t0 += RPB) {
    const int t = t0 + lr;
    const bool in_rec = t < t_end, row = in_rec && t < s.L, valid = row && t >= pad0;
    const int64_t off = row ? row_offset(s, n, h, t) + ch * 8 : 0;
    float g[8], ol[8], os[8];
    unpack8(next[0], g);
    unpack8(next[1], ol);
    unpack8(next[2], os);
    load(t + RPB);
    float aL = 0.f, aS = 0.f, woL = 0.f, woS = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      aL = fmaf(g[e], ol[e], aL);
      aS = fmaf(g[e], os[e], aS);
      woL = fmaf(wl[e], ol[e], woL);
      woS = fmaf(wsv[e], os[e], woS);
    }
    aL = row_sum<LPR>(aL);
    aS = row_sum<LPR>(aS);
    woL = row_sum<LPR>(woL);
    woS = row_sum<LPR>(woS);
    float alpha, beta;
    gate_of_row(woL + woS + bias, alpha, beta);
    const float diff = aL - aS, c = alpha * beta * diff, kL = beta * diff, kS = alpha * diff;
    float gl[8], gs[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      gl[e] = valid ? fmaf(kL, wl[e], g[e]) : 0.f;
      gs[e] = valid ? fmaf(kS, wsv[e], g[e]) : 0.f;
    }
    const uint4 pl = pack8(gl), ps = pack8(gs);
    if (row) {
      *reinterpret_cast<uint4 *>(g_lt + off) = pl;
      *reinterpret_cast<uint4 *>(g_st + off) = ps;
    }
    unpack8(pl, gl);  // as the attention kernels will read them
    unpack8(ps, gs);
    float dL = 0.f, dS = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      dL = fmaf(gl[e], ol[e], dL);
      dS = fmaf(gs[e], os[e], dS);
    }
    dL = row_sum<LPR>(dL);
    dS = row_sum<LPR>(dS);
    if (ch == 0 && in_rec) {
      float l0 = 0.f, l2 = 0.f, l4 = 0.f, s0 = 0.f, s4 = 0.f, s6 = 0.f;
      if (valid) {
        l0 = -(lse[(int64_t)u * s.L + t] * kLog2e - log2f(fmaxf(alpha, 1e-37f)));
        l2 = -dL;
        l4 = -1e30f;
        s0 = -1e30f;
        s4 = -(lse[BHL + (int64_t)u * s.L + t] * kLog2e - log2f(fmaxf(beta, 1e-37f)));
        s6 = -dS;
      }
      const int64_t ro = ((int64_t)u * Lpad + (t & ~1)) * 4 + (t & 1);
      float *rl = reinterpret_cast<float *>(rec_lt) + ro, *rs = reinterpret_cast<float *>(rec_st) + ro;
      rl[0] = l0; rl[2] = l2; rl[4] = l4; rl[6] = 0.f;
      rs[0] = s0; rs[2] = 0.f; rs[4] = s4; rs[6] = s6;
    }
    if (valid) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        acc[e] += (double)c * (double)ol[e];
        acc[8 + e] += (double)c * (double)os[e];
      }
      if (ch == 0) accB += (double)c;
    }
  }
  // The warp's rows: lanes that share columns exchange halves, each ends with 16 LPR / 32 sums (all of every
  // row's in shared memory and added there: 33 KB a CTA).
  int at = ch * 8;
#pragma unroll
  for (int o = LPR, m = 8; o < 32; o <<= 1, m >>= 1) {
    const bool up = threadIdx.x & o;
#pragma unroll
    for (int e = 0; e < m; ++e) {
      const double send = up ? acc[e] : acc[e + m], keep = up ? acc[e + m] : acc[e];
      acc[e] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    at += up ? (m == 8 ? D : m) : 0;
    accB += __shfl_xor_sync(0xffffffffu, accB, o);
  }
  const int warp = threadIdx.x >> 5;
#pragma unroll
  for (int e = 0; e < LPR / 2; ++e) red[warp][at + e] = acc[e];
  if ((threadIdx.x & 31) == 0) red[warp][2 * D] = accB;
  __syncthreads();
  for (int d = threadIdx.x; d < GW; d += 256) {
    double a = 0.0;
#pragma unroll
    for (int r = 0; r < 8; ++r) a += red[r][d];  // fixed order
    dgate_part[((int64_t)u * s.M + qb) * GW + d] = a;
  }
  if (threadIdx.x == 0) grid_wait();  // who waits for this kernel has then waited for the lists too
}

}  // namespace

int launch_fwd_tc_gate(const Shape &s, const void *q, const void *k, const void *v, const float *gate,
                       const int32_t *seq_lens, const int32_t *idx, void *out, void *out_lt, void *out_st,
                       float *lse, const Workspace &ws, cudaStream_t st) {
  void *olt = out_lt ? out_lt : ws.gate_olt, *ost = out_st ? out_st : ws.gate_ost;
  // (the attention kernel also writes `out`, mixed with a per-head weight it reads from the first
  // floats of F_o's parameters: finite numbers, overwritten below)
  if (int rc = launch_fwd_tc(s, q, k, v, gate, seq_lens, idx, out, olt, ost, lse, ws, st)) return rc;
  const int rpb = 256 / (s.D / 8);
  const unsigned grid = (unsigned)(s.B * s.H) * (unsigned)((s.L + rpb - 1) / rpb);
  LaunchScope ls(K_GATE_GRAD, st);
  launch_chained(s.D == 32 ? gate_mix_kernel<32> : gate_mix_kernel<64>, dim3(grid), dim3(256), 0, st, s, gate,
                 (const bf *)olt, (const bf *)ost, (bf *)out);
  return cudaGetLastError() == cudaSuccess ? BLOSSOM_OK : BLOSSOM_ERR_CUDA;
}

int launch_bwd_tc_gate(const Shape &s, const void *q, const void *k, const void *v, const float *gate,
                       const int32_t *seq_lens, const int32_t *idx, const void *out_lt, const void *out_st,
                       const float *lse, const void *dout, void *dq, void *dk, void *dv, float *dgate,
                       const Workspace &ws, cudaStream_t st) {
  const int Lpad = (s.L + 63) / 64 * 64;
  // The lists of both passes in one launch; the second pass adds to the first one's gradients as it writes them
  // (three scratch tensors, an addition kernel and a launch of lists less: 234 -> 204 us for a step of B 16,
  // H 4, L 900, D 64 with rotary positions), and beside the pre-pass, which needs none of it: one behind the other, and key-major
  // lists of both branches from the forward that nobody read, 165.5 us, now 160.1.
  int rc = launch_tc_meta(s, seq_lens, idx, ws.qmeta, ws.kmeta, st, ws.status + kTicketWord, 3, 0, ws.qmeta2, ws.kmeta2, true);
  if (rc) return rc;
  {
    LaunchScope ls(K_BWD_PREP, st);
    const int prows = gate_prep_rows(s), parts = (s.L + prows - 1) / prows;
    const unsigned grid = (unsigned)(s.B * s.H) * (unsigned)parts;
    launch_chained(s.D == 32 ? gate_prep_kernel<32> : gate_prep_kernel<64>, dim3(grid), dim3(256), 0, st, s, gate, seq_lens,
                   (const bf *)out_lt, (const bf *)out_st, lse, (const bf *)dout, (bf *)ws.gate_glt, (bf *)ws.gate_gst,
                   ws.qstats, ws.qstats2, ws.dgate_part, Lpad, prows, parts, ws.status_bwd);
    if (cudaGetLastError() != cudaSuccess) return BLOSSOM_ERR_CUDA;
  }
  rc = launch_bwd_tc(s, q, k, v, gate, seq_lens, idx, out_lt, out_st, lse, ws.gate_glt, dq, dk, dv, dgate, ws, st, 1,
                     ws.qstats);
  if (rc) return rc;
  Workspace second = ws;
  second.qmeta = ws.qmeta2;
  second.kmeta = ws.kmeta2;
  return launch_bwd_tc(s, q, k, v, gate, seq_lens, idx, out_lt, out_st, lse, ws.gate_gst, dq, dk, dv, nullptr, second, st, 2,
                       ws.qstats2);
}

}  // namespace tc
}  // namespace blossom
