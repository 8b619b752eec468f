// Certified single-precision scoring, a lane per query row: first stage of the selection (see
// select.cu for the stages, the scored blocks and the promise) for up to 128 scored blocks.
//
// A CTA of four warps takes 128 consecutive positions of a (batch, key/value head); a lane owns a
// row's logits, its norm, its softmax statistics and (in the per-position mode) its whole choice; rows of q
// are in registers (two lanes share the products of two rows) and the candidates' means are broadcast
// from shared memory, so that nothing of a row has to be staged.  The exponentials are taken relative to the bound
// scale |q| max|mean| of the row's logits instead of their maximum, which needs no pass of its own; a row
// for which that bound is so loose that its sum nearly vanishes is left to double precision.
// The register-blocked product of 128 x 64 tiles that this replaces (it remains for more than 128
// scored blocks) read every query row into shared memory as fp32 and computed 64 candidates whether
// there were 64 or 5: 123 us at B 128, H 4, L 1024 (32 blocks), 149 us at B 16, H 8, L 4096 (64
// blocks); 80 us (double precision throughout) without the causal mask at B 16, H 4, L 777, 122 us per
// position at B 8, 8 heads on 2, L 1500.
//
// Error bound, as in select.cu: with u = 2^-24 every logit is within E = (D + 4) u bound of its exact
// value (bound = scale max|q| max|mean|); the exponentials add 2^-21 and 2^-22 per unit of logit range;
// every addition of the normaliser and of the column sums, every head, every term of Eq. 11 one u each,
// with a margin of 40.
#include "select_geom.cuh"
#include "select_rows.cuh"

namespace blossom {
namespace {

constexpr int kRows = 128, kThreads = 128, kWarps = 4;

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  uint64_t d;
  asm("fma.rn.ftz.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<uint64_t *>(&a)), "l"(*reinterpret_cast<uint64_t *>(&b)),
        "l"(*reinterpret_cast<uint64_t *>(&c)));
  return *reinterpret_cast<float2 *>(&d);
}
// N consecutive elements as float pairs (zeros where !ok)
template <int N>
__device__ __forceinline__ void load_part(const __nv_bfloat16 *p, bool ok, float2 (&q)[N / 2]) {
#pragma unroll
  for (int ch = 0; ch < N / 8; ++ch) {
    const uint4 x = ok ? reinterpret_cast<const uint4 *>(p)[ch] : make_uint4(0u, 0u, 0u, 0u);
    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) q[ch * 4 + e] = make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));
  }
}
template <int N>
__device__ __forceinline__ void load_part(const float *p, bool ok, float2 (&q)[N / 2]) {
#pragma unroll
  for (int ch = 0; ch < N / 4; ++ch) {
    const float4 x = ok ? reinterpret_cast<const float4 *>(p)[ch] : make_float4(0.f, 0.f, 0.f, 0.f);
    q[ch * 2] = make_float2(x.x, x.y);
    q[ch * 2 + 1] = make_float2(x.z, x.w);
  }
}
template <int N>
__device__ __forceinline__ float square(const float2 (&q)[N]) {
  float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
  for (int e = 0; e < N; e += 2) {
    a0 = fma2(q[e], q[e], a0);
    a1 = fma2(q[e + 1], q[e + 1], a1);
  }
  return (a0.x + a0.y) + (a1.x + a1.y);
}

// PQ: one selection per query position.
template <typename T, int D, bool PQ>
__global__ void __launch_bounds__(kThreads, 4) score_rows_kernel(
    Shape sh, SelGeom g, RowsGeom rg, const T *__restrict__ q, const float *__restrict__ mean32,
    const float *__restrict__ norm, const int32_t *__restrict__ seq_lens, int32_t *__restrict__ idx,
    int32_t *__restrict__ worklist, int32_t *__restrict__ work_count) {
  grid_chain_enter();
  constexpr int P = D + 4;  // pitch of the means (floats)
  extern __shared__ __align__(16) float fsm[];
  __shared__ float kn_w[kWarps], qn_w[kWarps], inv_s[kWarps][32], bound_s[8][2];
  float *ms = fsm;                                     // [rg.cols][P] candidate means, candidate cmin first
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float *et = ms + rg.cols * P + warp * 32 * rg.pitch;  // [32][pitch] this warp's exponentials / scores
  float *pt = et + kWarps * 32 * rg.pitch;              // (PQ with grouped heads) [32][pitch] probabilities summed over heads
  const int M = sh.M, Bk = sh.Bk;
  const int ntiles = (sh.L + kRows - 1) / kRows, nU = sh.B * sh.Hkv;
  // late tiles have the most candidates: they go first (tile-major)
  const int tile = ntiles - 1 - (int)(blockIdx.x / nU), u = (int)(blockIdx.x % nU), n = u / sh.Hkv, hk = u % sh.Hkv;
  int len = seq_lens ? seq_lens[n] : sh.L;
  len = min(max(len, 0), sh.L);
  const int pad0 = sh.L - len;
  const bool causal = sh.causal;
  const int own = causal ? 0 : 1;
  const int row0 = tile * kRows, t = row0 + tid;  // this lane's query position
  const int qb0 = row0 / Bk, nqb = min(kRows / Bk, M - qb0);
  const int cmin = first_live_scored(g, pad0), jmin = pad0 / Bk;
  const int c_hi = causal ? n_candidates(sh, g, min(M - 1, qb0 + nqb - 1)) : g.n;
  const bool ok = t >= pad0 && t < sh.L;
  const int b = min(t, sh.L - 1) / Bk;
  const int ncol = max(0, c_hi - cmin);

  // Does any query block of the tile have a real choice to make from scores?
  auto choice = [&](int bb, int *want) {
    const int nsel = max(0, (causal ? bb : M) - jmin - own);
    *want = min(sh.topk - 1, nsel);
    return nsel > *want && *want > 0;
  };
  auto live_cands = [&](int bb) { return max(0, (causal ? n_candidates(sh, g, bb) : g.n) - cmin - own); };
  bool need = false;
  for (int i = 0; i < nqb; ++i) {
    int want;
    need |= max((qb0 + i) * Bk, pad0) < min((qb0 + i + 1) * Bk, sh.L) && choice(qb0 + i, &want) && live_cands(qb0 + i) > 0;
  }
  float qn = 0.f, kn = 0.f;  // the lane's largest query norm over the group's heads; the largest mean norm
  bool loose = false;        // a row whose reference was too far from its logits
  float colsum[2][4];        // (per block) summed probabilities of candidates lane, lane + 32, ...: of rows 0..15, 16..31
#pragma unroll
  for (int x = 0; x < 4; ++x) colsum[0][x] = colsum[1][x] = 0.f;

  if (need) {
    const float *kb = mean32 + ((int64_t)u * g.n + cmin) * D;
    for (int i = tid; i < ncol * (D / 4); i += kThreads)
      *reinterpret_cast<float4 *>(ms + (i / (D / 4)) * P + (i % (D / 4)) * 4) = reinterpret_cast<const float4 *>(kb)[i];
    for (int c = tid; c < ncol; c += kThreads) kn = fmaxf(kn, norm[(int64_t)u * g.n + cmin + c]);
    kn = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(kn)));  // (non-negative floats order like integers)
    if (lane == 0) kn_w[warp] = kn;
    __syncthreads();
    kn = fmaxf(fmaxf(kn_w[0], kn_w[1]), fmaxf(kn_w[2], kn_w[3]));
    // this lane's candidates: columns < nc of the table (the own block's column left out without the mask)
    const int nc = ok ? max(0, (causal ? n_candidates(sh, g, b) : g.n) - cmin) : 0;
    const int nc_warp = __reduce_max_sync(0xffffffffu, (unsigned)nc);
    const float sc2 = sh.scale * 1.4426950408889634f;
    float *er = et + lane * rg.pitch;
    const bool up = lane >= 16;
#pragma unroll 1
    for (int hg = 0; hg < sh.G; ++hg) {  // the heads of the group in ascending order (Eq. 12)
      // The products are shared by two lanes: lanes l and l + 16 hold the lower and the upper half of the
      // dimensions of rows l and l + 16, and exchange one partial sum per candidate, so that lane l ends up
      // with row l.  A broadcast load then feeds two rows (alone it took more cycles of the shared-memory
      // pipe than its multiply-adds take of theirs).
      float2 qa[D / 4], qb[D / 4];  // this half of rows (lane & 15) and (lane & 15) + 16
      const int ta = row0 + warp * 32 + (lane & 15), tb = ta + 16;
      const bool oka = ta >= pad0 && ta < sh.L, okb = tb >= pad0 && tb < sh.L;
      const T *base = q + row_offset(sh, n, hk * sh.G + hg, 0) + up * (D / 2);
      load_part<D / 2>(base + (int64_t)(oka ? ta : 0) * sh.sl, oka, qa);
      load_part<D / 2>(base + (int64_t)(okb ? tb : 0) * sh.sl, okb, qb);
      auto own_row = [&](float a, float b) { return (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16); };
      const float qh = sqrtf(own_row(square<D / 4>(qa), square<D / 4>(qb))) * 1.0001f;
      qn = fmaxf(qn, qh);
      const float ref = sc2 * qh * kn;  // >= every logit of the row (log2 units)
      float den = 0.f;
#pragma unroll 1
      for (int c = 0; c < nc_warp; c += 2) {  // (the table has a column more than candidates where their number is odd)
        float2 x0 = make_float2(0.f, 0.f), x1 = x0, y0 = x0, y1 = x0;  // rows a, b of candidate c and of c + 1
        const float4 *m0 = reinterpret_cast<const float4 *>(ms + c * P + up * (D / 2)), *m1 = m0 + P / 4;
#pragma unroll
        for (int e = 0; e < D / 8; ++e) {
          const float4 v = m0[e], w = m1[e];
          x0 = fma2(qa[2 * e], make_float2(v.x, v.y), x0);
          x1 = fma2(qb[2 * e], make_float2(v.x, v.y), x1);
          y0 = fma2(qa[2 * e], make_float2(w.x, w.y), y0);
          y1 = fma2(qb[2 * e], make_float2(w.x, w.y), y1);
          x0 = fma2(qa[2 * e + 1], make_float2(v.z, v.w), x0);
          x1 = fma2(qb[2 * e + 1], make_float2(v.z, v.w), x1);
          y0 = fma2(qa[2 * e + 1], make_float2(w.z, w.w), y0);
          y1 = fma2(qb[2 * e + 1], make_float2(w.z, w.w), y1);
        }
        const float z0 = own_row(x0.x + x0.y, x1.x + x1.y), z1 = own_row(y0.x + y0.y, y1.x + y1.y);
        const float e0 = c < nc && !(own && c + cmin == b) ? exp2f(fmaf(z0, sc2, -ref)) : 0.f;
        const float e1 = c + 1 < nc && !(own && c + 1 + cmin == b) ? exp2f(fmaf(z1, sc2, -ref)) : 0.f;
        er[c] = e0;
        er[c + 1] = e1;
        den += e0 + e1;
      }
      loose |= nc > own && !(den > 1e-30f);
      const float inv = den > 0.f ? 1.f / den : 0.f;
      if (PQ) {
        if (sh.G > 1) {
          float *pr = pt + lane * rg.pitch;
          for (int c = 0; c < nc_warp; ++c) pr[c] = hg == 0 ? er[c] * inv : fmaf(er[c], inv, pr[c]);
        }
      } else {
        inv_s[warp][lane] = inv;
        __syncwarp();
#pragma unroll
        for (int half = 0; half < 2; ++half) {
#pragma unroll 1
          for (int x = 0; x < 4; ++x) {
            const int c = lane + 32 * x;
            if (32 * x >= nc_warp) break;
            float a = 0.f;
            if (c < nc_warp)
#pragma unroll 8
              for (int r = 0; r < 16; ++r) a = fmaf(et[(16 * half + r) * rg.pitch + c], inv_s[warp][16 * half + r], a);
            // (x is a warp-uniform loop index; the registers are selected by constants)
            if (x == 0) colsum[half][0] += a;
            else if (x == 1) colsum[half][1] += a;
            else if (x == 2) colsum[half][2] += a;
            else colsum[half][3] += a;
          }
        }
        __syncwarp();
      }
    }
  }
  const float uu = 5.9604645e-8f, bound0 = sh.scale * kn;
  // relative distance of a score from its exact value, for query norms up to qmax and nsum additions
  auto error = [&](float qmax, float nsum) {
    const float bound = bound0 * qmax, E = (float)(D + 4) * uu * bound * 1.01f;
    return 2.f * E + 4.77e-7f + 2.f * bound * 2.39e-7f + (nsum + 2.f * (float)sh.G + (float)(g.rs * g.rl) + 40.f) * uu;
  };

  if (PQ) {
    // ---- Eq. 11, Eq. 13 and the certificate for this lane's own row ----
    if (t < sh.L) {
      int32_t *row = idx + ((int64_t)u * sh.L + t) * sh.topk;
      if (!ok) {
        for (int i = 0; i < sh.topk; ++i) row[i] = -1;
        return;
      }
      int want;
      const bool ch = choice(b, &want);
      const int nc = max(0, n_candidates(sh, g, b) - cmin);
      uint32_t taken[4] = {0u, 0u, 0u, 0u};  // bit j - jmin (at most 128 blocks)
      bool certain = true;
      if (!ch || nc == 0) {  // everything, or (no candidate yet: every score is zero) the lowest blocks
        for (int i = 0; i < want; ++i) taken[i >> 5] |= 1u << (i & 31);
      } else {
        float *S = sh.G > 1 ? pt + lane * rg.pitch : et + lane * rg.pitch;
        if (!g.plain) {
          float *o = sh.G > 1 ? et + lane * rg.pitch : pt + lane * rg.pitch;  // the table that is free
          for (int j = jmin; j < b; ++j) {
            float a = 0.f;
            for (int m = 0; m < g.rs; ++m)
              for (int e = 0; e < g.rl; ++e) {
                const int i = g.rs * j - m - e - cmin;
                if (i >= 0 && i < nc) a += S[i];
              }
            o[j - jmin] = a;
          }
          S = o;
        }
        const int ns = b - jmin;
        float kept = 0.f, dropped = 0.f;
        for (int k = 0; k <= want; ++k) {  // the want best, then the best that is left out
          float best = -1.f;
          int bi = 0;
          for (int j = 0; j < ns; ++j) {
            const uint32_t tk = j < 64 ? (j < 32 ? taken[0] : taken[1]) : (j < 96 ? taken[2] : taken[3]);
            const float x = S[j];
            if (x > best && !((tk >> (j & 31)) & 1u)) {
              best = x;
              bi = j;
            }
          }
          if (k == want) {
            dropped = best;
          } else {
            kept = best;
            const uint32_t bit = 1u << (bi & 31);
            if (bi < 32) taken[0] |= bit;
            else if (bi < 64) taken[1] |= bit;
            else if (bi < 96) taken[2] |= bit;
            else taken[3] |= bit;
          }
        }
        certain = !rg.exact && !loose && (kept - dropped) > error(qn, (float)nc) * (kept + dropped) * 1.001f;
      }
      if (certain) {
        int pos = 0;
#pragma unroll
        for (int x = 0; x < 4; ++x)
          for (uint32_t m = taken[x]; m; m &= m - 1) row[pos++] = jmin + 32 * x + __ffs(m) - 1;
        row[pos++] = b;
        for (; pos < sh.topk; ++pos) row[pos] = -1;
      } else {
        worklist[atomicAdd(work_count, 1)] = u * sh.L + t;
      }
    }
    return;
  }

  // ---- per query block: column sums of its rows, Eq. 11, Eq. 13 and the certificate ----
  // Sc[i][cols]: the tables are free now; block i's rows are 16-row groups i Bk / 16 ...
  __syncthreads();
  float *part = ms + rg.cols * P;            // [8 groups of 16 rows][128]
  float *Sc = part + 8 * 128;                // [4 warps][128]
  float *Sm = Sc + kWarps * 128;             // [4 warps][128] selection-block scores
  uint8_t *taken = reinterpret_cast<uint8_t *>(Sm + kWarps * 128);  // [4 warps][128]
#pragma unroll
  for (int half = 0; half < 2; ++half)
#pragma unroll
    for (int x = 0; x < 4; ++x) part[(2 * warp + half) * 128 + lane + 32 * x] = colsum[half][x];
  {
    const float w = loose ? INFINITY : qn;  // a loose row makes its block uncertain
    const float lo = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(lane < 16 ? w : 0.f)));
    const float hi = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(lane < 16 ? 0.f : w)));
    if (lane == 0) {
      bound_s[2 * warp][0] = lo;
      bound_s[2 * warp + 1][0] = hi;
    }
  }
  __syncthreads();
  const int gpb = Bk / 16;  // 16-row groups per block
  for (int i = warp; i < nqb; i += kWarps) {
    const int bb = qb0 + i;
    int32_t *row = idx + ((int64_t)u * M + bb) * sh.topk;
    if (max(bb * Bk, pad0) >= min((bb + 1) * Bk, sh.L)) {  // only padding
      for (int x = lane; x < sh.topk; x += 32) row[x] = -1;
      continue;
    }
    const int hi = causal ? bb : M, ncb = causal ? n_candidates(sh, g, bb) : g.n;
    int want;
    const bool ch = choice(bb, &want);
    uint8_t *tk = taken + warp * 128 - jmin;
    bool certain = true;
    __syncwarp();
    if (!ch) {
      for (int j = jmin + lane; j < hi; j += 32) tk[j] = want > 0 ? 1 : 0;
    } else if (live_cands(bb) == 0) {
      for (int j = jmin + lane; j < hi; j += 32) tk[j] = j - jmin < want ? 1 : 0;
    } else {
      float *S = Sc + warp * 128, qmax = 0.f;
      for (int c = lane; c < ncb - cmin; c += 32) {
        float a = 0.f;
        for (int r = 0; r < gpb; ++r) a += part[(i * gpb + r) * 128 + c];
        S[c] = a;
      }
      for (int r = 0; r < gpb; ++r) qmax = fmaxf(qmax, bound_s[i * gpb + r][0]);
      __syncwarp();
      if (!g.plain) {
        float *o = Sm + warp * 128;
        for (int j = jmin + lane; j < hi; j += 32) {
          float a = 0.f;
          for (int m = 0; m < g.rs; ++m)
            for (int e = 0; e < g.rl; ++e) {
              const int x = g.rs * j - m - e;
              if (x >= cmin && x < ncb) a += S[x - cmin];
            }
          o[j - jmin] = a;
        }
        S = o;
        __syncwarp();
      }
      // by rank: block j is kept iff fewer than `want` others beat it (ties to the lower index)
      const int ns = hi - jmin, ob = own ? bb - jmin : -1;
      float kept = -1.f, dropped = -1.f;
      for (int j = lane; j < ns; j += 32) {
        const float sj = S[j];
        int rank = 0;
#pragma unroll 4
        for (int x = 0; x < ns; ++x) {
          const float sx = S[x];
          rank += x != ob && (sx > sj || (sx == sj && x < j)) ? 1 : 0;
        }
        tk[jmin + j] = j != ob && rank < want ? 1 : 0;
        if (j != ob && rank == want - 1) kept = sj;
        if (j != ob && rank == want) dropped = sj;
      }
      // (scores are non-negative: exactly one lane holds each)
      kept = __uint_as_float(__reduce_max_sync(0xffffffffu, kept < 0.f ? 0u : __float_as_uint(kept)));
      dropped = __uint_as_float(__reduce_max_sync(0xffffffffu, dropped < 0.f ? 0u : __float_as_uint(dropped)));
      const float R = error(qmax, (float)(ncb - cmin) + (float)Bk * (float)sh.G);
      certain = !rg.exact && (kept - dropped) > R * (kept + dropped) * 1.001f;  // (false for an infinite qmax)
    }
    if (own && lane == 0) tk[bb] = 1;
    __syncwarp();
    if (certain) {
      int pos = 0;
      for (int base = jmin; base < hi; base += 32) {
        const int j = base + lane;
        const bool f = j < hi && tk[j];
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (f) row[pos + __popc(m & ((1u << lane) - 1u))] = j;
        pos += __popc(m);
      }
      if (!own) {
        if (lane == 0) row[pos] = bb;
        ++pos;
      }
      for (int x = pos + lane; x < sh.topk; x += 32) row[x] = -1;
    } else if (lane == 0) {
      worklist[atomicAdd(work_count, 1)] = u * M + bb;
    }
  }
}

}  // namespace

bool rows_geom(const Shape &sh, const SelGeom &g, RowsGeom *rg, size_t *smem) {
  if (g.n > 128 || sh.M > 128) return false;
  rg->cols = (g.n + 1) / 2 * 2 + 2;
  const int wide = sh.M > rg->cols ? sh.M : rg->cols;  // (per position the table also holds the scores of the selection blocks)
  rg->pitch = (sh.pq ? wide : rg->cols) | 1;
  const bool two = sh.pq && (sh.G > 1 || !g.plain);
  const size_t tables = (size_t)(two ? 2 : 1) * kWarps * 32 * rg->pitch * 4;
  const size_t tail = (size_t)(8 * 128 + 2 * kWarps * 128) * 4 + kWarps * 128;
  *smem = (size_t)rg->cols * (sh.D + 4) * 4 + (tables > tail ? tables : tail) + 16;
  return *smem <= 200 * 1024;
}

template <typename T, int D>
static int launch_t(const Shape &sh, const SelGeom &g, const RowsGeom &rg, size_t smem, const T *q, const float *mean32,
                    const float *norm, const int32_t *seq_lens, int32_t *idx, int32_t *list, int32_t *count,
                    cudaStream_t st) {
  auto kern = sh.pq ? score_rows_kernel<T, D, true> : score_rows_kernel<T, D, false>;
  if (smem > 40 * 1024 &&  // (static shared memory counts too)
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return BLOSSOM_ERR_CUDA;
  const unsigned grid = (unsigned)((sh.L + kRows - 1) / kRows) * (unsigned)(sh.B * sh.Hkv);
  LaunchScope ls(K_SCORE_FAST, st);
  return launch_chained(kern, dim3(grid), dim3(kThreads), smem, st, sh, g, rg, q, mean32, norm, seq_lens, idx, list,
                        count) == cudaSuccess
             ? BLOSSOM_OK
             : BLOSSOM_ERR_CUDA;
}

int launch_score_rows(const Shape &sh, const SelGeom &g, const RowsGeom &rg, size_t smem, int dtype, const void *q,
                      const float *mean32, const float *norm, const int32_t *seq_lens, int32_t *idx, int32_t *list,
                      int32_t *count, cudaStream_t st) {
  typedef __nv_bfloat16 bf;
  if (dtype == BLOSSOM_DTYPE_FP32) {
    if (sh.D == 32) return launch_t<float, 32>(sh, g, rg, smem, (const float *)q, mean32, norm, seq_lens, idx, list, count, st);
    return launch_t<float, 64>(sh, g, rg, smem, (const float *)q, mean32, norm, seq_lens, idx, list, count, st);
  }
  if (sh.D == 32) return launch_t<bf, 32>(sh, g, rg, smem, (const bf *)q, mean32, norm, seq_lens, idx, list, count, st);
  return launch_t<bf, 64>(sh, g, rg, smem, (const bf *)q, mean32, norm, seq_lens, idx, list, count, st);
}

}  // namespace blossom
