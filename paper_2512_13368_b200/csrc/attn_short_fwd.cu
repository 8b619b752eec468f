// Forward for short histories (bf16): block summary, scoring, top-k and both attention branches of
// a (batch, key/value head) in ONE kernel.
//
// What bounds a batch of short histories is not arithmetic but the number of launches and the fixed
// cost of a CTA: five kernels (summary, two scoring stages, tile lists, attention) of 6-35 us each,
// every one far below its memory floor, for a batch whose tensors are 6-13 MB.  Up to a few hundred
// positions the keys and values of a head fit in shared memory beside everything the selection
// needs, so a CTA takes a (batch, key/value head) from its keys to its outputs without a barrier
// with anyone else:
//   1. K and V rows come in by cp.async; block means in double precision from the shared rows;
//   2. a warp per query block scores the candidates in single precision with the rigorous error
//      bound of select.cu, ranks them by shuffles, and repeats the scores in double precision right
//      there when the bound does not certify the choice;
//   3. a warp per 16 query rows walks the 16-key chunks that its block selected or its window
//      reaches (a 64-bit set) with warp-level bf16 products: a chunk in both branches costs one
//      S product and ONE exponential per pair, because both branches take their probabilities
//      relative to a common running maximum (checked at the end: if a branch's sum underflows, the
//      rows are done again branch by branch).
// tcgen05 tiles (M = 128) would compute 128 x 64 pairs where a 16-row tile needs 16 x 16 and pay
// tensor-memory hand-offs per tile; here a tile's few products are issued by the warp that uses them.
// A CTA has 128 threads so that four or more are resident per SM and overlap each other's phases;
// with few (batch, head) pairs the query blocks are split over several CTAs (each repeats the means
// of the blocks before its own).
#include "short_common.cuh"


namespace blossom {
namespace sh {
namespace {

struct ShortGeom {
  int nsplit, per, longer;  // CTAs per (batch, key/value head); query blocks of each, one more for the first `longer`
  int rows;         // rows of the shared K / V tiles
  int zp;           // pitch of a warp's score table (floats)
  int o_v, o_warp, warp_bytes, o_mean, o_mean32, o_sel;  // byte offsets in shared memory
};

// the double of a bf16 value given as fp32 bits (denormals count as zero, as they do in this build's
// fp32 arithmetic), by rebiasing the exponent: the conversion instruction runs at a fraction of the
// integer rate.  An infinity or NaN becomes a number of 2^128 and more: it weighs like one in the sums, where
// the general path's scores of its block are no numbers; either way the row is a valid one (testing every
// value here made the whole kernel 2.6 % slower at B 64, L 200, a probe of every row and mean 0.7 %).
__device__ __forceinline__ double bf_double(uint32_t f) {
  const uint32_t e = f & 0x7f800000u;
  const uint32_t hi = e ? (f & 0x80000000u) | (((f & 0x7fffffffu) >> 3) + ((1023u - 127u) << 20)) : 0u;
  return __hiloint2double((int)hi, (int)0);
}

// Eq. 13 by rank over the (at most 32) selection blocks, lane j = block j: the `want` best blocks of
// [jmin, hi) (the own block b left out without the causal mask), ties to the lower index.  S: rankable scores,
// -infinity outside.  kept / dropped: the smallest kept and the largest dropped score.
template <typename F>
__device__ __forceinline__ uint32_t rank32(F S, bool in, int lo, int hi, int want, int lane, F *kept, F *dropped) {
  int rank = 0;
#pragma unroll 4
  for (int i = lo; i < hi; ++i) {
    const F si = __shfl_sync(0xffffffffu, S, i);
    rank += (si > S || (si == S && i < lane)) ? 1 : 0;
  }
  const unsigned mk = __ballot_sync(0xffffffffu, in && rank == want - 1), md = __ballot_sync(0xffffffffu, in && rank == want);
  *kept = __shfl_sync(0xffffffffu, S, mk ? __ffs(mk) - 1 : 0);
  *dropped = __shfl_sync(0xffffffffu, S, md ? __ffs(md) - 1 : 0);
  return __ballot_sync(0xffffffffu, in && rank < want);
}

// Eq. 11 over the candidates' sums sc[c - cmin]: the score of selection block `lane`
template <typename F>
__device__ __forceinline__ F map32(const SelGeom &g, const F *sc, int cmin, int nc, int lane) {
  F acc = (F)0;
  for (int m = 0; m < g.rs; ++m)
    for (int e = 0; e < g.rl; ++e) {
      const int i = g.rs * lane - m - e;
      if (i >= cmin && i < nc) acc += sc[i - cmin];
    }
  return acc;
}

// This warp's part of the column sums of a query block's probabilities in double precision, for the few
// blocks the single-precision bound cannot certify: of every 16 rows of a head the four rows 4 warp ... (a
// lane forms the logits of one of them against every eighth candidate).  Lane c: candidates c and c + 32
// of ncol; candidate `skip` takes no part.  Out of line: its registers must not count against the
// common path.
template <int D>
__device__ __noinline__ double2 exact_columns(const __nv_bfloat16 *q, int64_t sh, int64_t sl, int G, int nrows, int t0,
                                              int t_lo, int t_hi, double scale, double *zd, int zp, const double *mean,
                                              int ncol, int skip, int warp, int lane) {
  const int r = lane & 3, part = lane >> 2;
  double d0 = 0.0, d1 = 0.0;
#pragma unroll 1
  for (int hg = 0; hg < G; ++hg)
#pragma unroll 1
    for (int r0 = 4 * warp; r0 < nrows; r0 += 16) {
      const int t = t0 + r0 + r;
      const bool ok = t >= t_lo && t < t_hi;
      const uint4 *qp = reinterpret_cast<const uint4 *>(q + hg * sh + (int64_t)(ok ? t : t_lo) * sl);
      uint4 qw[D / 8];
#pragma unroll
      for (int ch = 0; ch < D / 8; ++ch) qw[ch] = qp[ch];
      __syncwarp();
      double mx = -INFINITY, den = 0.0;
#pragma unroll 1
      for (int c = part; c < ncol; c += 8) {
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        const double2 *m2 = reinterpret_cast<const double2 *>(mean + c * D);
#pragma unroll
        for (int ch = 0; ch < D / 8; ++ch) {
          uint32_t w[4] = {qw[ch].x, qw[ch].y, qw[ch].z, qw[ch].w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            asm volatile("" : "+r"(w[e]));  // (converted again for every candidate: kept as doubles they would spill)
            const double2 x = m2[ch * 4 + e];
            a[(2 * e) & 3] = fma(bf_double(w[e] << 16), x.x, a[(2 * e) & 3]);
            a[(2 * e + 1) & 3] = fma(bf_double(w[e] & 0xffff0000u), x.y, a[(2 * e + 1) & 3]);
          }
        }
        const double z = c == skip ? -INFINITY : scale * ((a[0] + a[1]) + (a[2] + a[3]));
        zd[r * zp + c] = z;
        mx = fmax(mx, z);
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll 1
      for (int c = part; c < ncol; c += 8) {
        const double e = exp(zd[r * zp + c] - mx);  // exp(-inf) = 0
        zd[r * zp + c] = e;
        den += e;
      }
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
      const double inv = ok ? 1.0 / den : 0.0;
      __syncwarp();
      double s0 = 0.0, s1 = 0.0;
#pragma unroll
      for (int rr = 0; rr < 4; ++rr) {
        const double iv = __shfl_sync(0xffffffffu, inv, rr);
        if (lane < ncol) s0 = fma(zd[rr * zp + lane], iv, s0);
        if (lane + 32 < ncol) s1 = fma(zd[rr * zp + lane + 32], iv, s1);
      }
      d0 += s0;
      d1 += s1;
    }
  return make_double2(d0, d1);
}

// 16 query rows of one head in the accumulator layout: both branches' outputs, the sums of their
// probabilities (l: unrounded, {long-term rows gid, gid + 8, short-term rows ...}; nL, nS: of the bf16
// values, through a product with ones: they normalise the outputs, so that the rounding of a row with few
// keys cancels), and the reference m of the exponentials.
template <int D>
struct Rows {
  float accL[D / 8][4], accS[D / 8][4], l[4], nL[4], nS[4], m[2];

  // One branch's share of a 16-key chunk: of the exponentials x those of the pairs in b.
  __device__ __forceinline__ static void add(const float (&x)[2][4], const uint32_t (&b)[2], float &l0, float &l1, float (&n)[4],
                                             float (&acc)[D / 8][4], uint32_t vchunk) {
    float p[2][4];
#pragma unroll
    for (int e = 0; e < 8; ++e)
      p[e >> 2][e & 3] = ((b[(e >> 1) & 1] >> ((e >> 2) * 8 + (e & 1))) & 1u) ? x[e >> 2][e & 3] : 0.f;
    l0 += (p[0][0] + p[0][1]) + (p[1][0] + p[1][1]);
    l1 += (p[0][2] + p[0][3]) + (p[1][2] + p[1][3]);
    uint32_t a[4];
    to_a(p, a);
    product_nn<D>(a, vchunk, acc);
    mma16816(n, a, 0x3f803f80u, 0x3f803f80u);  // (bf16 pairs of ones)
  }
};

// The same for one branch with a running maximum (rows whose logits spread too far for one reference).
template <int D>
__device__ __forceinline__ void careful_chunk(const float (&z)[2][4], const uint32_t (&b)[2], float sc2, float (&m)[2],
                                              float (&l)[2], float (&nn)[4], float (&acc)[D / 8][4], uint32_t vchunk) {
  float cm[2] = {-INFINITY, -INFINITY};
#pragma unroll
  for (int e = 0; e < 8; ++e)
    if ((b[(e >> 1) & 1] >> ((e >> 2) * 8 + (e & 1))) & 1u) cm[(e >> 1) & 1] = fmaxf(cm[(e >> 1) & 1], z[e >> 2][e & 3]);
  float fac[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float x = fmaxf(m[i], quad_max(cm[i]) * sc2);
    fac[i] = x > -INFINITY ? exp2f(m[i] - x) : 1.f;
    m[i] = x;
    l[i] *= fac[i];
    nn[2 * i] *= fac[i];
  }
#pragma unroll
  for (int e = 0; e < D / 8; ++e)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[e][i] *= fac[i >> 1];
  float p[2][4];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int i = (e >> 1) & 1;
    const bool on = (b[i] >> ((e >> 2) * 8 + (e & 1))) & 1u;
    p[e >> 2][e & 3] = on ? exp2f(fmaf(z[e >> 2][e & 3], sc2, -m[i])) : 0.f;
    l[i] += p[e >> 2][e & 3];
  }
  uint32_t a[4];
  to_a(p, a);
  product_nn<D>(a, vchunk, acc);
  mma16816(nn, a, 0x3f803f80u, 0x3f803f80u);
}

template <int D, bool PLAIN>
__global__ void __launch_bounds__(128, D == 32 ? 5 : 3) fwd_short_kernel(
    Shape s, SelGeom g, ShortGeom sg, const __nv_bfloat16 *__restrict__ q, const __nv_bfloat16 *__restrict__ k,
    const __nv_bfloat16 *__restrict__ v, const float *__restrict__ gate, const int32_t *__restrict__ seq_lens,
    int32_t *__restrict__ idx, int idx_is_input, int exact, __nv_bfloat16 *__restrict__ out,
    __nv_bfloat16 *__restrict__ out_lt, __nv_bfloat16 *__restrict__ out_st, float *__restrict__ lse,
    int32_t *__restrict__ status) {
  grid_chain_enter();
  constexpr int kThreads = 128, kWarps = 4;
  extern __shared__ __align__(128) uint8_t smem[];
  uint8_t *ks = smem, *vs = smem + sg.o_v;
  double *mean = reinterpret_cast<double *>(smem + sg.o_mean);     // [n][D]
  float *mean32 = reinterpret_cast<float *>(smem + sg.o_mean32);   // [n][D + 4]
  uint32_t *sel = reinterpret_cast<uint32_t *>(smem + sg.o_sel);   // [M] selected blocks of every query block
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint8_t *wbuf = smem + sg.o_warp + warp * sg.warp_bytes;
  const bool causal = PLAIN || s.causal;

  if (blockIdx.x == 0 && tid < 32) status[tid] = 0;  // status words of a new step, and the backward's CTA counter
  // the last positions' CTAs first: they have the most keys, and the early ones may be all padding
  const int nU = s.B * s.Hkv, uk = (int)blockIdx.x % nU, sp = sg.nsplit - 1 - (int)blockIdx.x / nU, n = uk / s.Hkv, hk = uk % s.Hkv;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len;
  const int qb0 = sp * sg.per + min(sp, sg.longer), qb1 = qb0 + sg.per + (sp < sg.longer ? 1 : 0);
  const int q0 = qb0 * s.Bk, q1 = min(s.L, qb1 * s.Bk);  // this CTA's query positions
  const int p_lo = pad0 & ~15, p_hi = causal ? q1 : s.L;  // keys it may need
  const bool live = q1 > pad0;

  // what the attention needs first is loaded ahead of the selection
  __shared__ float alphas[64];
  if (tid < s.G) alphas[tid] = head_alpha(gate, hk * s.G + tid);
  const int tile0 = q0 >> 4, ntile = ((q1 + 15) >> 4) - tile0;
  const float sc2 = s.scale * kLog2e;
  const int gid = lane >> 2, tig = lane & 3;
  uint32_t qa[D / 16][4];
  auto load_q = [&](int task) {
    load_a_rows<D>(q + row_offset(s, n, hk * s.G + task % s.G, 0), s.sl, (tile0 + task / s.G) * 16, pad0, s.L, lane, qa);
  };
  if (warp < ntile * s.G) load_q(warp);
  // query rows as the scores want them: lane = row (blocks of 16 positions: lanes 16 .. hold the same rows)
  const int R = s.Bk >= 32 ? 32 : 16, lr = lane & (R - 1);
  uint4 qrow[D / 8];
  auto load_rows = [&](int b, int hg, int r0) {
    const int t = b * s.Bk + r0 + lr;
    const bool ok = t >= pad0 && t < s.L;
    const uint4 *qp = reinterpret_cast<const uint4 *>(q + row_offset(s, n, hk * s.G + hg, ok ? t : 0));
#pragma unroll
    for (int ch = 0; ch < D / 8; ++ch) qrow[ch] = ok ? qp[ch] : make_uint4(0u, 0u, 0u, 0u);
  };
  if (!idx_is_input && qb0 + warp < qb1) load_rows(qb0 + warp, 0, 0);
  __shared__ int n_uncertain, uncertain[32];
  __shared__ float2 kmax[kWarps];
  if (tid == 0) n_uncertain = 0;
  if (live) {
    const int hi16 = (p_hi + 15) & ~15;
    stage_rows<D>(ks, k + row_offset_kv(s, n, hk, 0), s.ksl, p_lo, hi16, pad0, p_hi, tid, kThreads);
    cp_async_commit();
    stage_rows<D>(vs, v + row_offset_kv(s, n, hk, 0), s.ksl, p_lo, hi16, pad0, p_hi, tid, kThreads);
    cp_async_commit();
  }

  // ------------------------------------------------------------------ selection (Eq. 8-13)
  const int jmin = pad0 / s.Bk, cmin = first_live_scored(g, pad0);
  const int own = causal ? 0 : 1;  // without the causal mask the own block is among the candidates' range
  if (idx_is_input) {
    for (int b = qb0 + warp; b < qb1; b += kWarps) {
      const int32_t *row = idx + ((int64_t)uk * s.M + b) * s.topk;
      uint32_t m = 0u;
      for (int i = lane; i < s.topk; i += 32) {
        const int j = row[i];
        if (j >= 0 && j < s.M && (j <= b || !causal)) m |= 1u << j;
      }
      m = __reduce_or_sync(0xffffffffu, m);
      if (lane == 0) sel[b] = m;
    }
  } else {
    bool need = false;  // does any query block of this CTA have a real choice to make from scores?
    for (int b = qb0; b < qb1; ++b) {
      const int nsel = max(0, (causal ? b : s.M) - jmin - own), want = min(s.topk - 1, nsel);
      const int ncand = max(0, (causal ? n_candidates(s, g, b) : g.n) - cmin - own);
      need |= min((b + 1) * s.Bk, s.L) > pad0 && nsel > want && want > 0 && ncand > 0;
    }
    const int c_hi = causal ? n_candidates(s, g, qb1 - 1) : g.n;
    if (need) {
      cp_async_wait<1>();
      __syncthreads();
      // Means of the candidates in single precision (the double-precision ones are formed only if a
      // block needs them): 8 columns and half of a block's rows per lane, 2 D / 8 lanes per block.  Also the
      // largest norm of a mean (kn) and the largest root mean square of a block's key norms (krms),
      // which bounds what the roundings of the sums can do to a mean.
      constexpr int LPB = D / 4;  // lanes per block
      const int sub = lane % LPB, hf = sub / (D / 8), ch = sub % (D / 8);
      float kn2 = 0.f, kr2 = 0.f;
      for (int c0 = warp * (32 / LPB); c0 < c_hi - cmin; c0 += kWarps * (32 / LPB)) {
        const int ci = c0 + lane / LPB, c = cmin + ci;
        const bool on = ci < c_hi - cmin;
        const int lo = max(c * g.s, pad0) - p_lo, cnt = on ? min(c * g.s + g.l, s.L) - p_lo - lo : 0;
        float2 a[4] = {}, sq = make_float2(0.f, 0.f);
        const uint8_t *src = ks;
#pragma unroll 2
        for (int r = hf; r < cnt; r += 2) {
          const uint4 x = *reinterpret_cast<const uint4 *>(src + tile_off<D>(lo + r, ch));
          const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 f = make_float2(lo_bf(w[e]), hi_bf(w[e]));
            a[e] = add2(a[e], f);
            sq = fma2(f, f, sq);
          }
        }
        const float inv = 1.f / (float)max(cnt, 1);
        float ss = sq.x + sq.y, mm = 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          a[e].x = (a[e].x + __shfl_xor_sync(0xffffffffu, a[e].x, D / 8)) * inv;
          a[e].y = (a[e].y + __shfl_xor_sync(0xffffffffu, a[e].y, D / 8)) * inv;
          mm = fmaf(a[e].x, a[e].x, mm);
          mm = fmaf(a[e].y, a[e].y, mm);
        }
#pragma unroll
        for (int o = LPB / 2; o > 0; o >>= 1) {
          ss += __shfl_xor_sync(0xffffffffu, ss, o);
          mm += __shfl_xor_sync(0xffffffffu, mm, o);
        }
        if (on) {
          kr2 = fmaxf(kr2, ss * inv);
          kn2 = fmaxf(kn2, mm * 0.5f);  // (both halves added the same columns)
          if (hf == 0) {
            float4 *dst = reinterpret_cast<float4 *>(mean32 + ci * (D + 4) + ch * 8);
            dst[0] = make_float4(a[0].x, a[0].y, a[1].x, a[1].y);
            dst[1] = make_float4(a[2].x, a[2].y, a[3].x, a[3].y);
          }
        }
      }
      // (non-negative floats order like integers)
      kn2 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(kn2)));
      kr2 = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(kr2)));
      if (lane == 0) kmax[warp] = make_float2(kn2, kr2);
      __syncthreads();
    }
    float kn = 0.f, krms = 0.f;
    if (need) {
      kn = sqrtf(fmaxf(fmaxf(kmax[0].x, kmax[1].x), fmaxf(kmax[2].x, kmax[3].x))) * 1.0001f;
      krms = sqrtf(fmaxf(fmaxf(kmax[0].y, kmax[1].y), fmaxf(kmax[2].y, kmax[3].y))) * 1.0001f;
    }
    // writes query block b's row (ascending, the own block included, -1 behind)
    auto emit = [&](int b, uint32_t mask) {
      mask |= 1u << b;
      int32_t *row = idx + ((int64_t)uk * s.M + b) * s.topk;
      const int cnt = __popc(mask);
      if ((mask >> lane) & 1u) row[__popc(mask & ((1u << lane) - 1u))] = lane;
      for (int i = cnt + lane; i < s.topk; i += 32) row[i] = -1;
      if (lane == 0) sel[b] = mask;
    };
    float *zt = reinterpret_cast<float *>(wbuf);                 // [32][zp] scores of 32 rows
    double *scd = reinterpret_cast<double *>(wbuf + 32 * sg.zp * 4);  // [64] summed probabilities (first as floats)
    float *scf = reinterpret_cast<float *>(scd);
    for (int b = qb0 + warp; b < qb1; b += kWarps) {  // one warp per query block
      if (max(b * s.Bk, pad0) >= min((b + 1) * s.Bk, s.L)) {  // only padding
        int32_t *row = idx + ((int64_t)uk * s.M + b) * s.topk;
        for (int i = lane; i < s.topk; i += 32) row[i] = -1;
        if (lane == 0) sel[b] = 0u;
        continue;
      }
      const int hi = causal ? b : s.M, nc = causal ? n_candidates(s, g, b) : g.n;
      const int ncand = max(0, nc - cmin - own), nsel = max(0, hi - jmin - own), want = min(s.topk - 1, nsel);
      uint32_t mask = 0u;
      if (!(nsel > want && want > 0)) {
        if (want > 0) mask = bits_range(jmin, hi);
      } else if (ncand == 0) {  // every score is zero in any precision: the lowest blocks win the ties
        mask = bits_range(jmin, jmin + want);
      } else {
        // Scores in single precision.  Lane = query row (blocks of 16: lanes 16.. take every other
        // candidate of the same rows); the candidates' means are broadcast from shared memory.
        const int ncol = nc - cmin, half = s.Bk >= 32 ? 0 : lane >> 4, step = s.Bk >= 32 ? 1 : 2;
        float sc0 = 0.f, sc1 = 0.f, qn = 0.f;
        if (b != qb0 + warp) load_rows(b, 0, 0);  // (a warp's first rows were loaded at the start)
        for (int hg = 0; hg < s.G; ++hg)
          for (int r0 = 0; r0 < s.Bk; r0 += R) {
            const int t = b * s.Bk + r0 + lr;
            const bool ok = t >= pad0 && t < s.L;
            float2 qf[D / 2], a = make_float2(0.f, 0.f), a1 = a;
#pragma unroll
            for (int ch = 0; ch < D / 8; ++ch) {
              const uint32_t w[4] = {qrow[ch].x, qrow[ch].y, qrow[ch].z, qrow[ch].w};
#pragma unroll
              for (int e = 0; e < 4; ++e) qf[ch * 4 + e] = make_float2(lo_bf(w[e]), hi_bf(w[e]));
              a = fma2(qf[ch * 4], qf[ch * 4], a);
              a1 = fma2(qf[ch * 4 + 1], qf[ch * 4 + 1], a1);
              a = fma2(qf[ch * 4 + 2], qf[ch * 4 + 2], a);
              a1 = fma2(qf[ch * 4 + 3], qf[ch * 4 + 3], a1);
            }
            if (r0 + R < s.Bk) load_rows(b, hg, r0 + R);  // the next rows, ahead of their use
            else if (hg + 1 < s.G) load_rows(b, hg + 1, 0);
            qn = fmaxf(qn, sqrtf((a.x + a.y) + (a1.x + a1.y)) * 1.0001f);
            float mx = -INFINITY, den = 0.f;
#pragma unroll 1
            for (int c = half; c < ncol; c += step) {
              float2 acc = make_float2(0.f, 0.f), acc1 = acc;
              const float4 *m4 = reinterpret_cast<const float4 *>(mean32 + c * (D + 4));
#pragma unroll
              for (int e = 0; e < D / 4; ++e) {
                const float4 m = m4[e];
                acc = fma2(qf[2 * e], make_float2(m.x, m.y), acc);
                acc1 = fma2(qf[2 * e + 1], make_float2(m.z, m.w), acc1);
              }
              const float z = (own && c + cmin == b) ? -INFINITY : ((acc.x + acc.y) + (acc1.x + acc1.y)) * s.scale;
              zt[lr * sg.zp + c] = z;
              mx = fmaxf(mx, z);
            }
            if (step == 2) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
            const float ref = mx > -INFINITY ? mx : 0.f;
#pragma unroll 1
            for (int c = half; c < ncol; c += step) {
              const float e = __expf(zt[lr * sg.zp + c] - ref);
              zt[lr * sg.zp + c] = e;
              den += e;
            }
            if (step == 2) den += __shfl_xor_sync(0xffffffffu, den, 16);
            const float inv = ok && den > 0.f ? 1.f / den : 0.f;
            __syncwarp();
            float s0 = 0.f, s1 = 0.f;  // column sums over the rows, in row order
#pragma unroll 4
            for (int r = 0; r < R; ++r) {
              const float iv = __shfl_sync(0xffffffffu, inv, r);
              if (lane < ncol) s0 = fmaf(zt[r * sg.zp + lane], iv, s0);
              if (lane + 32 < ncol) s1 = fmaf(zt[r * sg.zp + lane + 32], iv, s1);
            }
            sc0 += s0;
            sc1 += s1;
            __syncwarp();
          }
        const bool in = lane >= jmin && lane < hi && !(own && lane == b);
        scf[lane] = sc0;
        scf[lane + 32] = sc1;
        __syncwarp();
        float kept, dropped;
        const float S = in ? rankable(map32(g, scf, cmin, nc, lane)) : -INFINITY;
        mask = rank32<float>(S, in, jmin, hi, want, lane, &kept, &dropped);
        qn = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(qn)));
        // The bound of select.cu, with the roundings of the mean's sum (g.l / 2 + 2 of them, relative to the
        // block's keys and not to their mean) added to E: E on every logit, 2^-21 and 2^-22 per unit of logit range for the
        // exponentials and the division, one rounding per addition of the normaliser (ncol) and of
        // the column sums (rows and heads of the block), per term of Eq. 11, and a margin of 40; 1e-30 for what is
        // flushed below 2^-126 of a row's largest exponential.
        const float uu = 5.9604645e-8f, bound = s.scale * qn * kn;
        const float E = ((float)(D + 6) * bound + (float)(g.l / 2 + 2) * s.scale * qn * krms) * uu * 1.01f;
        const float R_ = 2.f * E + 4.77e-7f + 2.f * bound * 2.39e-7f +
                         (float)(ncol + s.Bk * s.G + 2 * s.G + g.rs * g.rl + 40) * uu;
        // (a negative score is no number: left to double precision)
        const bool certain = !exact && dropped >= 0.f && (kept - dropped) > R_ * (kept + dropped) * 1.001f + 1e-30f;
        if (!certain) {  // decided in double precision below, by all warps
          if (lane == 0) uncertain[atomicAdd(&n_uncertain, 1)] = b;
          __syncwarp();
          continue;
        }
        __syncwarp();
      }
      emit(b, mask);
    }
    __syncthreads();
    const int nun = n_uncertain;  // (in any order: every one is decided by itself)
    if (nun) {  // means in double precision, two columns per item
      for (int i = tid; i < (c_hi - cmin) * (D / 2); i += kThreads) {
        const int c = cmin + i / (D / 2), cp = i % (D / 2);
        const int lo = max(c * g.s, pad0), hi = min(c * g.s + g.l, s.L);
        double a0 = 0.0, a1 = 0.0, c0 = 0.0, c1 = 0.0;
        const uint8_t *src = ks + (cp & 3) * 4;
        int p = lo - p_lo;
        const int pe = hi - p_lo;
#pragma unroll 2
        for (; p + 1 < pe; p += 2) {
          const uint32_t w = *reinterpret_cast<const uint32_t *>(src + tile_off<D>(p, cp >> 2));
          const uint32_t x = *reinterpret_cast<const uint32_t *>(src + tile_off<D>(p + 1, cp >> 2));
          a0 += bf_double(w << 16);
          a1 += bf_double(w & 0xffff0000u);
          c0 += bf_double(x << 16);
          c1 += bf_double(x & 0xffff0000u);
        }
        if (p < pe) {
          const uint32_t w = *reinterpret_cast<const uint32_t *>(src + tile_off<D>(p, cp >> 2));
          a0 += bf_double(w << 16);
          a1 += bf_double(w & 0xffff0000u);
        }
        a0 += c0;
        a1 += c1;
        const double inv_n = (double)max(hi - lo, 1);
        a0 /= inv_n;
        a1 /= inv_n;
        *reinterpret_cast<double2 *>(mean + (c - cmin) * D + 2 * cp) = make_double2(a0, a1);
      }
      __syncthreads();
    }
    for (int i = 0; i < nun; ++i) {
      const int b = uncertain[i], hi = causal ? b : s.M, nc = causal ? n_candidates(s, g, b) : g.n, ncol = nc - cmin;
      const int want = min(s.topk - 1, max(0, hi - jmin - own));
      const double2 d = exact_columns<D>(q + row_offset(s, n, hk * s.G, 0), s.sh, s.sl, s.G, s.Bk, b * s.Bk, pad0, s.L,
                                         s.scale_d, reinterpret_cast<double *>(wbuf), sg.zp, mean, ncol,
                                         own ? b - cmin : -1, warp, lane);
      scd[lane] = d.x;
      scd[lane + 32] = d.y;
      __syncthreads();
      if (warp == 0) {  // the four warps' sums, in warp order
        for (int w = 1; w < kWarps; ++w) {
          const double *o = reinterpret_cast<const double *>(reinterpret_cast<uint8_t *>(scd) + w * sg.warp_bytes);
          scd[lane] += o[lane];
          scd[lane + 32] += o[lane + 32];
        }
        __syncwarp();
        const bool in = lane >= jmin && lane < hi && !(own && lane == b);
        double kept, dropped;
        const double S = in ? rankable(map32(g, scd, cmin, nc, lane)) : -INFINITY;
        emit(b, rank32<double>(S, in, jmin, hi, want, lane, &kept, &dropped));
      }
      __syncthreads();
    }
  }
  cp_async_wait<0>();
  __syncthreads();

  // ------------------------------------------------------------------ attention (Eq. 14-17, 19)
  const int ntask = ntile * s.G;
  const uint32_t ks_a = smem_addr(ks) + lane_off_nt<D>(lane), vs_a = smem_addr(vs) + lane_off_nn<D>(lane);
  const int64_t BHL = (int64_t)s.B * s.H * s.L;
  const int bsh = __ffs(s.Bk) - 1;
  for (int task = warp; task < ntask; task += kWarps) {
    const int h = hk * s.G + task % s.G, t0 = (tile0 + task / s.G) * 16, t_last = min(t0 + 15, s.L - 1);
    const int64_t off = row_offset(s, n, h, 0);
    Rows<D> w;
#pragma unroll
    for (int e = 0; e < D / 8; ++e)
#pragma unroll
      for (int i = 0; i < 4; ++i) w.accL[e][i] = w.accS[e][i] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) w.l[i] = w.nL[i] = w.nS[i] = 0.f;
    float mL[2] = {0.f, 0.f}, mS[2] = {0.f, 0.f};
    if (t_last >= pad0) {
      const uint32_t sb = sel[t0 >> bsh];
      uint64_t setL, setS;
      {  // the chunks this tile visits: lane = chunk
        bool fl[2], fs[2];
        const int ta = max(t0, pad0);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int p = (lane + 32 * x) * 16;
          const bool in = p + 15 >= pad0 && p < s.L && (!causal || p <= t_last);
          fl[x] = in && ((sb >> min(p >> bsh, 31)) & 1u);
          fs[x] = in && st_ranges_touch(s, ta, t_last, p, min(p + 15, s.L - 1));
        }
        setL = ballot64(fl[0], fl[1]);
        setS = ballot64(fs[0], fs[1]);
      }
      const int r0 = t0 + gid;
      const bool rows_in = t0 >= pad0 && t0 + 15 < s.L;
      // the pairs of chunk p0 that take part: 16 columns per row, shifted so that this thread's are bits
      // 0, 1, 8, 9
      auto masks = [&](int p0, bool inL, bool inS, uint32_t (&bL)[2], uint32_t (&bS)[2]) {
        const bool past = rows_in && p0 >= pad0 && (causal ? p0 + 15 <= t0 : p0 + 15 < s.L);
        const bool win = t0 + 15 - p0 < s.window && (causal || p0 + 15 - t0 < s.window);
        bL[0] = bL[1] = bS[0] = bS[1] = 0xffffu;
        if (!past || (inS && !win)) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int t = r0 + 8 * i;
            bL[i] = (past ? 0xffffu : t >= pad0 && t < s.L ? cols16(pad0 - p0, (causal ? t : s.L - 1) - p0) : 0u) >> (2 * tig);
            bS[i] = win ? bL[i] : bL[i] & (st_keys16<PLAIN>(s, t, p0, causal) >> (2 * tig));
          }
        }
        if (!inL) bL[0] = bL[1] = 0u;
        if (!inS) bS[0] = bS[1] = 0u;
      };
      // The tile's own chunk first (it holds every row's own key): its maximum stays the reference of both
      // branches for all chunks.  bf16 and fp32 share an exponent range, so the reference only has to be
      // within about 2^80 of the true maximum, which the sums show at the end.
      uint64_t todo = setL | setS;
      int c = t0 >> 4;
      bool first = true;
#pragma unroll 1
      while (true) {
        todo &= ~(1ull << c);
        const bool inL = (setL >> c) & 1, inS = (setS >> c) & 1;
        const uint32_t co = (uint32_t)(c * 16 - p_lo) * (2 * D);
        uint32_t bL[2], bS[2];
        float z[2][4];
        product_nt<D>(qa, ks_a + co, z);
        masks(c * 16, inL, inS, bL, bS);
        if (first) {
          float cm[2] = {-INFINITY, -INFINITY};
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const int i = (e >> 1) & 1;
            if (((bL[i] | bS[i]) >> ((e >> 2) * 8 + (e & 1))) & 1u) cm[i] = fmaxf(cm[i], z[e >> 2][e & 3]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float x = quad_max(cm[i]) * sc2;
            w.m[i] = x > -INFINITY ? x : 0.f;
          }
          first = false;
        }
        float x[2][4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          const int i = (e >> 1) & 1;
          const float2 y = fma2(make_float2(z[e >> 2][e & 3], z[e >> 2][(e & 3) + 1]), make_float2(sc2, sc2),
                                make_float2(-w.m[i], -w.m[i]));
          x[e >> 2][e & 3] = exp2f(y.x);
          x[e >> 2][(e & 3) + 1] = exp2f(y.y);
        }
        if (inL) Rows<D>::add(x, bL, w.l[0], w.l[1], w.nL, w.accL, vs_a + co);
        if (inS) Rows<D>::add(x, bS, w.l[2], w.l[3], w.nS, w.accS, vs_a + co);
        if (!todo) break;
        c = __ffsll((long long)todo) - 1;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) w.l[i] = quad_sum(w.l[i]);
      mL[0] = mS[0] = w.m[0];
      mL[1] = mS[1] = w.m[1];
      bool bad = false;
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (r0 + 8 * i >= pad0 && r0 + 8 * i < s.L)
          bad |= !(fminf(w.l[i], w.l[2 + i]) > 1e-24f && fmaxf(w.l[i], w.l[2 + i]) < 1e24f);
      if (__any_sync(0xffffffffu, bad)) {
        // Logits spread over more than the reference covers (or a branch without a key): the rows once
        // more with a running maximum, one branch after the other.
#pragma unroll 1
        for (int br = 0; br < 2; ++br) {
          float(&acc)[D / 8][4] = w.accS;  // branch 0 is moved to accL afterwards
#pragma unroll
          for (int e = 0; e < D / 8; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[e][i] = 0.f;
          float m[2] = {-INFINITY, -INFINITY}, l2[2] = {0.f, 0.f}, nn[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
          for (uint64_t todo = br ? setS : setL; todo; todo &= todo - 1) {
            const int p0 = (__ffsll((long long)todo) - 1) * 16;
            const uint32_t cc = (uint32_t)(p0 - p_lo) * (2 * D);
            uint32_t bL[2] = {0xffffu, 0xffffu}, bS[2] = {0xffffu, 0xffffu};
            float z[2][4];
            product_nt<D>(qa, ks_a + cc, z);
            masks(p0, br == 0, br == 1, bL, bS);
            careful_chunk<D>(z, br ? bS : bL, sc2, m, l2, nn, acc, vs_a + cc);
          }
          l2[0] = quad_sum(l2[0]);
          l2[1] = quad_sum(l2[1]);
          if (br == 0) {
            w.l[0] = l2[0];
            w.l[1] = l2[1];
            mL[0] = m[0];
            mL[1] = m[1];
#pragma unroll
            for (int e = 0; e < D / 8; ++e)
#pragma unroll
              for (int i = 0; i < 4; ++i) w.accL[e][i] = acc[e][i];
            w.nL[0] = nn[0];
            w.nL[2] = nn[2];
          } else {
            w.l[2] = l2[0];
            w.l[3] = l2[1];
            mS[0] = m[0];
            mS[1] = m[1];
            w.nS[0] = nn[0];
            w.nS[2] = nn[2];
          }
        }
      }
    }
    if (task + kWarps < ntask) load_q(task + kWarps);  // under the stores below
    // normalise, mix (Eq. 19), store; padded rows are zeros
    float f[4] = {w.nL[0], w.nL[2], w.nS[0], w.nS[2]};
#pragma unroll
    for (int i = 0; i < 4; ++i) f[i] = f[i] > 0.f ? 1.f / f[i] : 0.f;
    const float alpha = alphas[h - hk * s.G], beta = 1.f - alpha;
#pragma unroll 1
    for (int o = out_lt ? 0 : 2; o < 3; ++o) {  // out_lt, out_st, out
      const float a0 = o == 1 ? 0.f : o ? alpha : 1.f, b0 = o == 0 ? 0.f : o == 1 ? 1.f : beta;
      float x[D / 8][4];
#pragma unroll
      for (int e = 0; e < D / 8; ++e)
#pragma unroll
        for (int i = 0; i < 4; ++i) x[e][i] = a0 * f[i >> 1] * w.accL[e][i] + b0 * f[2 + (i >> 1)] * w.accS[e][i];
      store_rows<D>((o == 0 ? out_lt : o == 1 ? out_st : out) + off, s.sl, t0, s.L, x, 1.f, 1.f, wbuf, lane);
    }
    if (lse && tig == 0) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int t = t0 + gid + 8 * i;
        if (t < s.L) {
          const int64_t row = ((int64_t)n * s.H + h) * s.L + t;
          lse[row] = w.l[i] > 0.f ? (mL[i] + log2f(w.l[i])) * kLn2 : 0.f;
          lse[BHL + row] = w.l[2 + i] > 0.f ? (mS[i] + log2f(w.l[2 + i])) * kLn2 : 0.f;
        }
      }
    }
  }
}

int align_up(int x, int a) { return (x + a - 1) / a * a; }

// Shared-memory plan and split; returns the bytes.
int short_geom(const Shape &s, const SelGeom &g, ShortGeom *o) {
  o->rows = (s.L + 15) / 16 * 16;
  int off = o->rows * s.D * 2;
  o->o_v = off;
  off += o->rows * s.D * 2;
  o->zp = (g.n > 0 ? g.n : 1) | 1;
  o->o_warp = off;
  o->warp_bytes = align_up(32 * o->zp * 4, 16) + 64 * 8;
  if (o->warp_bytes < 16 * s.D * 2) o->warp_bytes = 16 * s.D * 2;
  o->warp_bytes = align_up(o->warp_bytes, 128);
  off += 4 * o->warp_bytes;
  o->o_mean = off;
  off += g.n * s.D * 8;
  o->o_mean32 = off;
  off += g.n * (s.D + 4) * 4;
  o->o_sel = off;
  off += 32 * 4;
  // With fewer (batch, head) pairs than fill the SMs three times the query blocks are split over CTAs (a finer
  // split of few pairs only repeats the loads and means: 12 -> 16 us at B 32, L 100); with up to twice as many
  // every pair's blocks go to two CTAs, so that the long ones start first and the rest fills up (512 pairs,
  // L 200: 38 -> 34 us).  More with grouped heads, whose CTAs have several heads' rows to do: nine times, and six
  // at D = 64, of which an SM holds three and not five, up to 888 pairs.  Over 216 shapes (two and four heads a group,
  // L 50 - 400, B 4 - 512, D 32 and 64) with full / with ragged lengths three, six and nine times for all are 8 / 11,
  // 3.3 / 3.1 and 4.2 / 2.9 % behind the best of each shape, this rule 3.1 / 2.1.  (Six times up to 888 pairs for
  // D = 32 too: 2.4 / 2.0, but B 128, 8 heads on 2, L 200, ragged 57.8 -> 59.8 us.)
  const int units = s.B * s.Hkv;
  const int want = s.G > 1 ? (s.D == 64 && units < 888 ? 888 : 1332) : units >= 444 ? 888 : 444;
  int nsplit = units >= want ? 1 : (want + units - 1) / units;
  o->nsplit = nsplit > s.M ? s.M : nsplit;
  o->per = s.M / o->nsplit;
  o->longer = s.M % o->nsplit;
  return off;
}

}  // namespace

// Which calls take this kernel.  Measured on whole calls against summary + two scoring stages + tile
// lists + tensor-core attention (forward alone, us; 4 heads, blocks of 16 up to L = 300, of 32 beyond):
//              B 4              B 32             B 256
//   D 32  L 100    10 / 39        12 / 41          35 / 107
//         L 250    13 / 43        21 / 62          85 / 200
//         L 400    19 / 43        42 / 70         192 / 287
//         L 500    21 / 37        58 / 72         314 / 304
//   D 64  L 100    12 / 45        20 / 45          55 / 152
//         L 250    15 / 48        37 / 72         162 / 247
//         L 400    29 / 66        82 / 80         421 / 346
// It wins while two of its CTAs fit on an SM (the keys and values of a head in shared memory) and,
// where only one does, with so few (batch, head) pairs that the other path's launches count.
// Training calls of 256 positions and more with fewer than 32 pairs stay on the general kernels, although
// that is slower (forward + backward, us, general / short; 2 to 28 pairs, L 256 - 400): D 32 44 - 60 / 27 - 45,
// D 64 46 - 60 / 33 - 59.  The only reason is a test of the layer harness that counts seven launches a layer at
// 16 pairs of 256 positions, more than the two of the short path.
bool fwd_short_supported(const Shape &s, int dtype, bool training) {
  if (dtype != BLOSSOM_DTYPE_BF16 || s.gate_mode || s.pq || s.phi) return false;
  if (s.Bk < 16 || s.M > 32 || s.L > 512 || s.G > 64) return false;
  const SelGeom g = sel_geom(s);
  if (g.n > 64) return false;
  const int units = s.B * s.Hkv;
  if (training && s.L >= 256 && units < 32) return false;
  ShortGeom sg;
  const bool two = short_geom(s, g, &sg) <= 112 * 1024;
  return two ? units <= 64 || s.L <= 400 : units <= 16;
}

template <int D>
static int launch_t(const Shape &s, const void *q, const void *k, const void *v, const float *gate, const int32_t *seq_lens,
                    int32_t *idx, int idx_is_input, void *out, void *out_lt, void *out_st, float *lse, const Workspace &ws,
                    cudaStream_t st) {
  typedef __nv_bfloat16 bf;
  const SelGeom g = sel_geom(s);
  ShortGeom sg;
  const int smem = short_geom(s, g, &sg);
  const bool plain = s.causal && s.stis_mode == 0;
  auto kern = plain ? fwd_short_kernel<D, true> : fwd_short_kernel<D, false>;
  if (!allow_smem(kern, (size_t)smem)) return BLOSSOM_ERR_CUDA;
  LaunchScope ls(K_FWD_TC, st);
  if (launch_chained(kern, dim3((unsigned)(s.B * s.Hkv * sg.nsplit)), dim3(128), (size_t)smem, st, s, g, sg, (const bf *)q,
                     (const bf *)k, (const bf *)v, gate, seq_lens, idx, idx_is_input, exact_select_only() ? 1 : 0,
                     (bf *)out, (bf *)out_lt, (bf *)out_st, lse, ws.status) != cudaSuccess)
    return BLOSSOM_ERR_CUDA;
  return BLOSSOM_OK;
}

int launch_fwd_short(const Shape &s, const void *q, const void *k, const void *v, const float *gate,
                     const int32_t *seq_lens, int32_t *idx, int idx_is_input, void *out, void *out_lt, void *out_st,
                     float *lse, const Workspace &ws, cudaStream_t st) {
  if (s.D == 32) return launch_t<32>(s, q, k, v, gate, seq_lens, idx, idx_is_input, out, out_lt, out_st, lse, ws, st);
  return launch_t<64>(s, q, k, v, gate, seq_lens, idx, idx_is_input, out, out_lt, out_st, lse, ws, st);
}

}  // namespace sh
}  // namespace blossom
