// Certified single-precision scoring, a lane per query row: first stage of the selection (see
// select.cu for the stages, the scored blocks and the promise) for up to 128 scored blocks.
//
// A CTA of four warps takes 128 consecutive positions of a (batch, key/value head).  The logits of a warp's
// rows come from warp-level matrix products for bf16 inputs, the means split into three bf16 values whose
// sum they are exactly (a lane holding its row in registers and the means broadcast from shared memory took
// 100 us at B 16, H 8, L 4096, 68 at B 128, H 4, L 1024; the shared-memory pipe bound it), and from
// packed multiply-adds for fp32.  The exponentials, relative to the bound scale |q| max|mean| of the row's
// logits instead of their maximum (which needs no pass of its own; a row for which that bound is so loose
// that its sum nearly vanishes is left to double precision), go through a table in shared memory: a lane
// per column sums them over the rows of a block, or, per position, a lane per row makes its row's choice.
// The register-blocked product of 128 x 64 tiles in select.cu (more than 128 scored blocks) stages every
// query row as fp32 and computes 64 candidates whether there are 64 or 5: 149 and 123 us at these sizes.
//
// Error bound, as in select.cu: with u = 2^-24 every logit is within E of its exact value, bound = scale
// max|q| max|mean|: (D + 4) u bound for multiply-adds.  For the matrix products PTX guarantees exact
// products and accumulation in at least single precision with unspecified rounding, so 2 u per addition; the
// leading parts are accumulated 16 dimensions at a time from zero (16 additions, 32 u) and the D / 16
// results added up, the smaller ones, at 2^-8 of their size, in one go (2 D additions): (32 + D / 16 + 0.1 D
// + 6) u bound.  The exponentials add 2^-21 and 2^-22 per unit of logit range; sums of non-negative
// terms add one u per addition that a term goes through (the normaliser, 16 rows, the 16-row groups of a
// block, the heads, Eq. 11), with a margin of 40.  One loss is not relative to the scores: exponentials (and
// products) below 2^-126 are flushed to zero.  A row is left to double precision unless its sum exceeds
// kMinDen = 2^-63, so each costs a probability less than 2^-62, and the certificate allows the dropped block
// one of them per row, head and term of Eq. 11.  (2^-100 would accept looser references, but then
// scores less than 1e-8 apart were never certain; 2^-63 is a reference 43 above the row's largest logit.)
#include "select_rows.cuh"
#include "short_common.cuh"

namespace blossom {
namespace {

constexpr int kRows = 128, kThreads = 128, kWarps = 4;
constexpr float kMinDen = 1.0842022e-19f, kLost = 2.f * 2.1684043e-19f;  // 2^-63; twice 2^-62

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

// Eight elements as doubles.
__device__ __forceinline__ void to_double(const uint4 &v, double (&x)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    x[2 * e] = (double)__uint_as_float(w[e] << 16);
    x[2 * e + 1] = (double)__uint_as_float(w[e] & 0xffff0000u);
  }
}

struct Columns {
  double s[4];
};
// One warp's part of the column sums of a query block's probabilities in double precision: of the block's
// rows (`nq` positions from `qlo` of G heads, head-major) taken 16 at a time the four rows 4 warp ...; a
// lane forms the logits of one of them against every eighth candidate.  s[x]: candidate lane + 32 x of
// ncol; candidate `skip` takes no part.  Out of line: its registers must not count against the common path.
template <typename T, int D>
__device__ __noinline__ Columns exact_columns(const T *q, int64_t sh, int64_t sl, int G, int nq, int qlo, double scale,
                                              double *zd, int nz, const double *mean, int ncol, int skip, int warp,
                                              int lane) {
  const int r = lane & 3, pt = lane >> 2, nrows = nq * G;
  Columns out = {{0.0, 0.0, 0.0, 0.0}};
#pragma unroll 1
  for (int r0 = 4 * warp; r0 < nrows; r0 += 16) {
    const int x = r0 + r;
    const bool on = x < nrows;
    const T *row = q + (on ? (int64_t)(x / nq) * sh + (int64_t)(qlo + x % nq) * sl : (int64_t)qlo * sl);
    double *z = zd + (4 * warp + r) * nz;
    __syncwarp();
    double mx = -INFINITY, den = 0.0;
#pragma unroll 1
    for (int c = pt; c < ncol; c += 16) {
      const int c1 = c + 8 < ncol ? c + 8 : c;
      const double2 *k0 = reinterpret_cast<const double2 *>(mean + (int64_t)c * D);
      const double2 *k1 = reinterpret_cast<const double2 *>(mean + (int64_t)c1 * D);
      double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 2
      for (int e = 0; e < D / 8; ++e) {
        double v[8];
        if constexpr (sizeof(T) == 2) {
          to_double(reinterpret_cast<const uint4 *>(row)[e], v);
        } else {
          const float4 f = reinterpret_cast<const float4 *>(row)[2 * e], g = reinterpret_cast<const float4 *>(row)[2 * e + 1];
          v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w; v[4] = g.x; v[5] = g.y; v[6] = g.z; v[7] = g.w;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const double2 x0 = k0[4 * e + j], x1 = k1[4 * e + j];
          a[0] = fma(v[2 * j], x0.x, a[0]);
          a[1] = fma(v[2 * j + 1], x0.y, a[1]);
          a[2] = fma(v[2 * j], x1.x, a[2]);
          a[3] = fma(v[2 * j + 1], x1.y, a[3]);
        }
      }
      const double z0 = c == skip ? -INFINITY : scale * (a[0] + a[1]), z1 = c1 == skip ? -INFINITY : scale * (a[2] + a[3]);
      z[c] = z0;
      if (c1 != c) z[c1] = z1;
      mx = fmax(mx, fmax(z0, z1));
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll 1
    for (int c = pt; c < ncol; c += 8) {
      const double e = exp(z[c] - mx);  // exp(-inf) = 0
      z[c] = e;
      den += e;
    }
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
    const double inv = on ? 1.0 / den : 0.0;
    __syncwarp();
#pragma unroll 1
    for (int y = 0; y < 4; ++y) {
      const double iv = __shfl_sync(0xffffffffu, inv, y);
      const double *zy = zd + (4 * warp + y) * nz;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (lane + 32 * i < ncol) out.s[i] = fma(zy[lane + 32 * i], iv, out.s[i]);
    }
  }
  return out;
}

// A head's share of a row's scores: pr (+)= e inv over the candidates, four loads of each ahead of the stores (the compiler
// does not move a load before a store to a table that might be the same).
__device__ __forceinline__ void add_head(int hg, int n, const float *e, float inv, float *pr) {
  for (int c = 0; c < n; c += 4) {
    float x[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[i] = c + i < n ? e[c + i] : 0.f;
      y[i] = hg && c + i < n ? pr[c + i] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (c + i < n) pr[c + i] = hg ? fmaf(x[i], inv, y[i]) : x[i] * inv;
  }
}

// PQ: one selection per query position.  Four CTAs an SM then: in the registers of five (96 a thread) the queries loaded ahead
// do not fit.  The selection alone, us with four | five: 8 heads on 2 L 50, B 256, D 32 20.2 | 20.4; L 200, B 128, D 32
// 32.5 | 34.6, D 64 37.1 | 41.9; L 1500, B 16, D 32 50.4 | 50.3, D 64 62.5 | 64.3; ungrouped L 200, B 256, D 32 26.9 | 27.3.  Five are
// better by 1 - 2 % with many candidates at D 32: L 300, B 128 48.4 | 47.7, four heads L 1500, B 16 34.6 | 33.8.
template <typename T, int D, bool PQ>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 2 ? (PQ ? 4 : 5) : 4) score_rows_kernel(
    Shape sh, SelGeom g, RowsGeom rg, const T *__restrict__ q, const float *__restrict__ mean32,
    const float *__restrict__ norm, const double *__restrict__ mean, const int32_t *__restrict__ seq_lens,
    int32_t *__restrict__ idx, int32_t *__restrict__ worklist, int32_t *__restrict__ work_count) {
  grid_chain_enter();
  constexpr bool kMma = sizeof(T) == 2;  // bf16: products on the warp-level matrix pipe
  constexpr int P = D + 4;               // pitch of the means (floats; the fp32 form)
  // rows of a warp that its table holds at a time
  constexpr int kTab = kMma && !PQ ? 16 : 32;
  extern __shared__ __align__(128) float fsm[];
  __shared__ float kn_w[kWarps], inv_s[kWarps][32], rowq_s[kWarps][32], bound_s[8][2];
  __shared__ int n_uncertain, uncertain[8];
  // candidate means, candidate cmin first: [rg.cols][P] floats, or bf16 tiles [hi, mid, lo][rg.cols][D]
  float *ms = fsm, *tab = fsm + rg.means;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float *et = tab + warp * kTab * rg.pitch;  // [kTab][pitch] this warp's exponentials / scores
  const int M = sh.M, Bk = sh.Bk;
  // (PQ) hs warps share 32 rows: a head each, then a share of the rows' choices.  A tile is 128 / hs rows.
  const int lg = PQ && kMma ? rg.lg_heads : 0, hs = 1 << lg, rw = warp >> lg, hw = warp & (hs - 1), rows = kRows >> lg;
  const int ntiles = (sh.L + rows - 1) / rows, nU = sh.B * sh.Hkv;
  // late tiles have the most candidates: they go first (tile-major)
  const int tile = ntiles - 1 - (int)(blockIdx.x / nU), u = (int)(blockIdx.x % nU), n = u / sh.Hkv, hk = u % sh.Hkv;
  int len = seq_lens ? seq_lens[n] : sh.L;
  len = min(max(len, 0), sh.L);
  const int pad0 = sh.L - len;
  const bool causal = sh.causal;
  const int own = causal ? 0 : 1;
  const int row0 = tile * rows, wrow0 = row0 + 32 * rw;  // first row of the CTA, of the warp
  // this lane's query position: of its warp's rows; where warps share rows, hs lanes make the choice of one
  const int lrow = hw * (32 >> lg) + (lane >> lg), sub = lane & (hs - 1), t = wrow0 + lrow;
  float *pt = tab + (kWarps * kTab + rw * 32) * rg.pitch;  // (PQ with grouped heads or Eq. 11) [32][pitch] probabilities summed over heads
  const int qb0 = row0 / Bk, nqb = min((row0 + rows - 1) / Bk + 1, M) - qb0;
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
  if (tid == 0) n_uncertain = 0;
  float qn = 0.f, kn = 0.f;  // the lane's largest query norm over the group's heads; the largest mean norm
  bool loose = false;        // a row whose reference was too far from its logits
  float colsum[2][4];        // (per block) summed probabilities of candidates lane, lane + 32, ...: of rows 0..15, 16..31
#pragma unroll
  for (int x = 0; x < 4; ++x) colsum[0][x] = colsum[1][x] = 0.f;

  if (need) {
    const float *kb = mean32 + ((int64_t)u * g.n + cmin) * D;
    if constexpr (kMma) {
      // a mean of 24 significant bits as the exact sum of three bf16 values
      uint8_t *tiles = reinterpret_cast<uint8_t *>(ms);
      for (int i = tid; i < rg.cols * (D / 8); i += kThreads) {
        const int c = i / (D / 8), ch = i % (D / 8);
        float x[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (c < ncol) {
          const float4 a = reinterpret_cast<const float4 *>(kb)[2 * i], e = reinterpret_cast<const float4 *>(kb)[2 * i + 1];
          x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = e.x; x[5] = e.y; x[6] = e.z; x[7] = e.w;
        }
#pragma unroll
        for (int part = 0; part < 3; ++part) {
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            w[e] = sh::pack2(x[2 * e], x[2 * e + 1]);
            x[2 * e] -= sh::lo_bf(w[e]);
            x[2 * e + 1] -= sh::hi_bf(w[e]);
          }
          *reinterpret_cast<uint4 *>(tiles + part * rg.cols * D * 2 + sh::tile_off<D>(c, ch)) =
              make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
      rowq_s[warp][lane] = 0.f;
    } else {
      for (int i = tid; i < ncol * (D / 4); i += kThreads)
        *reinterpret_cast<float4 *>(ms + (i / (D / 4)) * P + (i % (D / 4)) * 4) = reinterpret_cast<const float4 *>(kb)[i];
    }
    for (int c = tid; c < ncol; c += kThreads) kn = fmaxf(kn, norm[(int64_t)u * g.n + cmin + c]);
    kn = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(kn)));  // (non-negative floats order like integers)
    if (lane == 0) kn_w[warp] = kn;
    __syncthreads();
    kn = fmaxf(fmaxf(kn_w[0], kn_w[1]), fmaxf(kn_w[2], kn_w[3]));
    // this lane's candidates: columns < nc of the table (the own block's column left out without the mask)
    const int nc = ok ? max(0, (causal ? n_candidates(sh, g, b) : g.n) - cmin) : 0;
    int nc_warp = __reduce_max_sync(0xffffffffu, (unsigned)nc);
    if (hs > 1) {  // of all 32 rows: under the causal mask (a selection per position has it) the last one's
      const int tl = min(wrow0 + 31, sh.L - 1);
      nc_warp = tl >= pad0 && wrow0 < sh.L ? max(0, n_candidates(sh, g, tl / Bk) - cmin) : 0;
    }
    const float sc2 = sh.scale * 1.4426950408889634f;
    float *er = et + lane * rg.pitch;
    const bool up = lane >= 16;
    // column sums of 16 rows' probabilities (tables: exponentials and the rows' reciprocal normalisers)
    auto sums = [&](int half, const float *e16, const float *inv16) {
#pragma unroll 1
      for (int x = 0; x < 4; ++x) {
        const int c = lane + 32 * x;
        if (32 * x >= nc_warp) break;
        float a = 0.f;
        if (c < nc_warp)
#pragma unroll 8
          for (int r = 0; r < 16; ++r) a = fmaf(e16[r * rg.pitch + c], inv16[r], a);
        // (half and x are warp-uniform; the registers are selected by constants)
        float(&cs)[4] = half ? colsum[1] : colsum[0];
        if (x == 0) cs[0] += a;
        else if (x == 1) cs[1] += a;
        else if (x == 2) cs[2] += a;
        else cs[3] += a;
      }
    };
    uint32_t qnext[kMma && PQ ? D / 16 : 1][4];  // (PQ) the next 16 rows' queries, a product loop ahead: few warps a scheduler
    if constexpr (kMma && PQ)
      sh::load_a_rows<D>(q + row_offset(sh, n, hk * sh.G + hw, 0), sh.sl, wrow0, pad0, sh.L, lane, qnext);
#pragma unroll 1
    for (int hg = hw; hg < sh.G; hg += hs) {  // the heads of the group in ascending order (Eq. 12)
      if constexpr (kMma) {
        const int gid = lane >> 2, tig = lane & 3;
        const uint32_t tiles = sh::smem_addr(ms) + sh::lane_off_nt<D>(lane), part_bytes = (uint32_t)rg.cols * D * 2;
#pragma unroll
        for (int mt = 0; mt < 2; ++mt) {  // 16 rows at a time
          const int tm = wrow0 + 16 * mt;
          uint32_t qa[D / 16][4];
          if constexpr (PQ) {
#pragma unroll
            for (int k = 0; k < D / 16; ++k)
#pragma unroll
              for (int e = 0; e < 4; ++e) qa[k][e] = qnext[k][e];
            if (mt == 0 || hg + hs < sh.G)
              sh::load_a_rows<D>(q + row_offset(sh, n, hk * sh.G + hg + mt * hs, 0), sh.sl, wrow0 + 16 * (1 - mt), pad0,
                                 sh.L, lane, qnext);
          } else {
            sh::load_a_rows<D>(q + row_offset(sh, n, hk * sh.G + hg, 0), sh.sl, tm, pad0, sh.L, lane, qa);
          }
          float ref[2] = {0.f, 0.f}, den[2] = {0.f, 0.f}, qh[2];
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              ref[e & 1] = fmaf(sh::lo_bf(qa[k][e]), sh::lo_bf(qa[k][e]), ref[e & 1]);
              ref[e & 1] = fmaf(sh::hi_bf(qa[k][e]), sh::hi_bf(qa[k][e]), ref[e & 1]);
            }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            qh[i] = sqrtf(sh::quad_sum(ref[i])) * 1.0001f;
            ref[i] = sc2 * qh[i] * kn;  // >= every logit of the row (log2 units)
          }
          const int t0 = tm + gid;
          const bool ok0 = t0 >= pad0 && t0 < sh.L, ok1 = t0 + 8 >= pad0 && t0 + 8 < sh.L;
          int ncm[2], skip[2];  // (blocks of 8: rows gid and gid + 8 lie in different ones)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int bm = min(t0 + 8 * i, sh.L - 1) / Bk;
            ncm[i] = max(0, (causal ? n_candidates(sh, g, bm) : g.n) - cmin);
            skip[i] = own ? bm - cmin : -1;
          }
          float *e0 = et + ((PQ ? 16 * mt : 0) + gid) * rg.pitch + 2 * tig, *e1 = e0 + 8 * rg.pitch;
#pragma unroll 1
          for (int c = 0; c < nc_warp; c += 16) {
            const uint32_t chunk = tiles + c * D * 2;
            float z[2][4];
            sh::product_nt<D>(qa, chunk + 2 * part_bytes, z);       // the small parts first
            sh::product_nt_add<D>(qa, chunk + part_bytes, z);
            sh::product_nt_steps<D>(qa, chunk, z);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                const int cc = c + 8 * nt + 2 * tig + j;
                z[nt][j] = ok0 && cc < ncm[0] && cc != skip[0] ? exp2f(fmaf(z[nt][j], sc2, -ref[0])) : 0.f;
                z[nt][2 + j] = ok1 && cc < ncm[1] && cc != skip[1] ? exp2f(fmaf(z[nt][2 + j], sc2, -ref[1])) : 0.f;
                e0[c + 8 * nt + j] = z[nt][j];
                e1[c + 8 * nt + j] = z[nt][2 + j];
              }
            den[0] += (z[0][0] + z[0][1]) + (z[1][0] + z[1][1]);
            den[1] += (z[0][2] + z[0][3]) + (z[1][2] + z[1][3]);
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            den[i] = sh::quad_sum(den[i]);
            if (tig == 0) {
              const int r = 16 * mt + gid + 8 * i;
              const bool bad = (i ? ok1 : ok0) && ncm[i] > own && !(den[i] > kMinDen);  // the reference is too far away
              inv_s[warp][r] = den[i] > 0.f ? 1.f / den[i] : 0.f;
              rowq_s[warp][r] = fmaxf(rowq_s[warp][r], bad ? INFINITY : qh[i]);
            }
          }
          __syncwarp();
          if (!PQ) {
            sums(mt, et, inv_s[warp] + 16 * mt);
            __syncwarp();
          }
        }
        if (PQ && sh.G > 1) {
          if (hs == 1) {
            add_head(hg, nc_warp, er, inv_s[warp][lane], pt + lane * rg.pitch);
            __syncwarp();
          } else {  // the hs heads in ascending order too: a lane takes every hs-th candidate of its row
            __syncthreads();
            const float *eh = tab + (rw * hs * 32 + lrow) * rg.pitch;
            float *pr = pt + lrow * rg.pitch;
#pragma unroll 4
            for (int c = sub; c < nc_warp; c += hs) {
              float a = hg >= hs ? pr[c] : 0.f;
              for (int h = 0; h < hs; ++h) a = fmaf(eh[h * 32 * rg.pitch + c], inv_s[rw * hs + h][lrow], a);
              pr[c] = a;
            }
            __syncthreads();
          }
        }
      } else {
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
      loose |= nc > own && !(den > kMinDen);
      const float inv = den > 0.f ? 1.f / den : 0.f;
      if (PQ) {
        if (sh.G > 1) {
          float *pr = pt + lane * rg.pitch;
          add_head(hg, nc_warp, er, inv, pr);
        }
      } else {
        inv_s[warp][lane] = inv;
        __syncwarp();
        sums(0, et, inv_s[warp]);
        sums(1, et + 16 * rg.pitch, inv_s[warp] + 16);
        __syncwarp();
      }
      }
    }
    if constexpr (kMma) {
      for (int h = 0; h < hs; ++h) qn = fmaxf(qn, rowq_s[rw * hs + h][lrow]);
      loose = qn == INFINITY;
    }
  }
  const float uu = 5.9604645e-8f, bound0 = sh.scale * kn;
  // relative distance of a score from its exact value, for query norms up to qmax and nsum additions in a row
  const auto den_adds = [](int cols) { return kMma ? cols / 16 + 6 : cols / 2 + 2; };
  auto error = [&](float qmax, float nsum) {
    const float bound = bound0 * qmax, E = (kMma ? 32.f + 0.1f * D + (float)(D / 16) + 6.f : (float)(D + 4)) * uu * bound * 1.01f;
    return 2.f * E + 4.77e-7f + 2.f * bound * 2.39e-7f + (nsum + 2.f * (float)sh.G + (float)(g.rs * g.rl) + 40.f) * uu;
  };

  // what flushed exponentials of so many rows can take from a score
  auto lost = [&](int rows) { return (float)(rows * sh.G * g.rs * g.rl) * kLost; };

  if (PQ) {
    // ---- Eq. 11, Eq. 13 and the certificate for this lane's row, or its share of it ----
    int want = 0;
    const bool scored = ok && choice(b, &want) && n_candidates(sh, g, b) > cmin;
    const int nc = max(0, n_candidates(sh, g, b) - cmin), ns = scored ? b - jmin : 0;
    float *S = (sh.G > 1 ? pt : et) + lrow * rg.pitch;
    if (!g.plain) {
      // the other table (with hs warps on a row its first one's: nobody reads the exponentials any more)
      float *o = sh.G > 1 ? tab + (rw * hs * 32 + lrow) * rg.pitch : pt + lrow * rg.pitch;
      for (int j = jmin + 4 * sub; j < jmin + ns; j += 4 * hs) {  // (four at a time, as in add_head)
        float a[4] = {0.f, 0.f, 0.f, 0.f};
        for (int m = 0; m < g.rs; ++m)
          for (int e = 0; e < g.rl; ++e)
#pragma unroll
            for (int y = 0; y < 4; ++y) {
              const int i = g.rs * (j + y) - m - e - cmin;
              if (i >= 0 && i < nc) a[y] += S[i];
            }
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (j + y < b) o[j + y - jmin] = a[y];
      }
      S = o;
      __syncwarp();
    }
    uint32_t taken[4] = {0u, 0u, 0u, 0u};  // bit j - jmin (at most 128 blocks)
    float kept = 0.f, dropped = 0.f;
    // The want best, then the best that is left out.  A chain of loads per lane and few warps a scheduler: what is
    // taken is overwritten.  (A test of its bit per score and one load after the other: with add_head's and Eq. 11's
    // loads one by one too 36.6 us at B 8, 8 heads on 2, L 1500, D 64, 72.7 at B 64; now 30.9 and 64.6, and 28.1 and
    // 58.0 with the queries loaded ahead.)
    const int most = __reduce_max_sync(0xffffffffu, (unsigned)(scored ? want + 1 : 0));
    for (int k = 0; k < most; ++k) {
      float best = -1.f;
      int bi = 0;
      if (k <= want) {
#pragma unroll 8
        for (int j = sub; j < ns; j += hs) {
          const float x = S[j];
          if (x > best) {
            best = x;
            bi = j;
          }
        }
      }
      for (int o = 1; o < hs; o <<= 1) {  // the best of the row's lanes, ties to the lower index
        const float x = __shfl_xor_sync(0xffffffffu, best, o);
        const int xi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (x > best || (x == best && xi < bi)) {
          best = x;
          bi = xi;
        }
      }
      if (scored && k == want) dropped = best;
      if (scored && k < want) {
        kept = best;
        if ((bi & (hs - 1)) == sub) S[bi] = -1.f;
        const uint32_t bit = 1u << (bi & 31);
        if (bi < 32) taken[0] |= bit;
        else if (bi < 64) taken[1] |= bit;
        else if (bi < 96) taken[2] |= bit;
        else taken[3] |= bit;
      }
    }
    if (t < sh.L && sub == 0) {
      int32_t *row = idx + ((int64_t)u * sh.L + t) * sh.topk;
      if (!ok) {
        for (int i = 0; i < sh.topk; ++i) row[i] = -1;
        return;
      }
      if (!scored)  // everything, or (no candidate yet: every score is zero) the lowest blocks
        for (int i = 0; i < want; ++i) taken[i >> 5] |= 1u << (i & 31);
      if (!scored || (!loose && (kept - dropped) > error(qn, (float)den_adds(nc)) * (kept + dropped) * 1.001f + lost(1))) {
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
  float *part = tab;                         // [8 groups of 16 rows][128]
  float *Sc = part + 8 * 128;                // [4 warps][132]
  float *Sm = Sc + kWarps * 132;             // [4 warps][132] selection-block scores
  uint8_t *taken = reinterpret_cast<uint8_t *>(Sm + kWarps * 132);  // [4 warps][128]
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
      float *S = Sc + warp * 132, qmax = 0.f;
      for (int c = lane; c < ncb - cmin; c += 32) {
        float a = 0.f;
        for (int r = 0; r < gpb; ++r) a += part[(i * gpb + r) * 128 + c];
        S[c] = a;
      }
      for (int r = 0; r < gpb; ++r) qmax = fmaxf(qmax, bound_s[i * gpb + r][0]);
      __syncwarp();
      if (!g.plain) {
        float *o = Sm + warp * 132;
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
      if (lane < 4) S[ns + lane] = -1.f;
      if (lane == 0 && ob >= 0) S[ob] = -1.f;
      __syncwarp();
      for (int j = lane; j < ns; j += 32) {
        const float sj = S[j];
        int rank = 0;
        // (non-negative floats order like integers; the own block, -1, beats nobody; four at a time, the
        // scores padded with -1)
        const int kj = __float_as_int(sj);
        for (int x = 0; x < ns; x += 4) {
          const int4 k4 = *reinterpret_cast<const int4 *>(S + x);
          rank += k4.x > kj || (k4.x == kj && x < j) ? 1 : 0;
          rank += k4.y > kj || (k4.y == kj && x + 1 < j) ? 1 : 0;
          rank += k4.z > kj || (k4.z == kj && x + 2 < j) ? 1 : 0;
          rank += k4.w > kj || (k4.w == kj && x + 3 < j) ? 1 : 0;
        }
        tk[jmin + j] = j != ob && rank < want ? 1 : 0;
        if (j != ob && rank == want - 1) kept = sj;
        if (j != ob && rank == want) dropped = sj;
      }
      // (scores are non-negative: exactly one lane holds each)
      kept = __uint_as_float(__reduce_max_sync(0xffffffffu, kept < 0.f ? 0u : __float_as_uint(kept)));
      dropped = __uint_as_float(__reduce_max_sync(0xffffffffu, dropped < 0.f ? 0u : __float_as_uint(dropped)));
      const float R = error(qmax, (float)(den_adds(ncb - cmin) + 16 + gpb));
      certain = (kept - dropped) > R * (kept + dropped) * 1.001f + lost(Bk);  // (false for an infinite qmax)
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
      if (rg.list) worklist[atomicAdd(work_count, 1)] = u * M + bb;
      else uncertain[atomicAdd(&n_uncertain, 1)] = bb;
    }
  }
  if (rg.list) return;
  // ---- the blocks that could not be certified, in double precision by all warps ----
  __syncthreads();
  const int nun = n_uncertain;  // (in any order: every one is decided by itself)
  const int nz = (g.n + 1) | 1;
  double *zd = reinterpret_cast<double *>(fsm), *partd = zd + 16 * nz, *Sc2 = partd + kWarps * 128, *S2 = Sc2 + 128;
  uint8_t *tk = reinterpret_cast<uint8_t *>(S2 + 128);
  for (int i = 0; i < nun; ++i) {
    const int bb = uncertain[i], hi = causal ? bb : M, ncb = causal ? n_candidates(sh, g, bb) : g.n;
    const int qlo = max(bb * Bk, pad0), nq = min((bb + 1) * Bk, sh.L) - qlo;
    int want;
    choice(bb, &want);
    const Columns c = exact_columns<T, D>(q + row_offset(sh, n, hk * sh.G, 0), sh.sh, sh.sl, sh.G, nq, qlo, sh.scale_d, zd, nz,
                                          mean + ((int64_t)u * g.n + cmin) * D, ncb - cmin, own ? bb - cmin : -1, warp, lane);
#pragma unroll
    for (int x = 0; x < 4; ++x) partd[warp * 128 + lane + 32 * x] = c.s[x];
    __syncthreads();
    Sc2[tid] = (partd[tid] + partd[128 + tid]) + (partd[256 + tid] + partd[384 + tid]);
    __syncthreads();
    const int j = jmin + tid;
    const bool in = j < hi && !(own && j == bb);
    if (j < hi) {
      double a = 0.0;
      for (int m = 0; m < g.rs; ++m)
        for (int e = 0; e < g.rl; ++e) {
          const int y = g.rs * j - m - e;
          if (y >= cmin && y < ncb) a += Sc2[y - cmin];
        }
      S2[tid] = in ? rankable(a) : -INFINITY;  // (the own block is not ranked: it is kept anyway)
    }
    __syncthreads();
    if (j < hi) {
      const double sj = S2[tid];
      int rk = 0;
#pragma unroll 4
      for (int y = 0; y < hi - jmin; ++y) {
        const double sy = S2[y];
        rk += (sy > sj || (sy == sj && y < tid)) ? 1 : 0;
      }
      tk[tid] = !in || rk < want ? 1 : 0;
    }
    __syncthreads();
    if (warp == 0) {
      int32_t *row = idx + ((int64_t)u * M + bb) * sh.topk;
      int pos = 0;
      for (int base = 0; base < hi - jmin; base += 32) {
        const bool f = base + lane < hi - jmin && tk[base + lane];
        const unsigned m = __ballot_sync(0xffffffffu, f);
        if (f) row[pos + __popc(m & ((1u << lane) - 1u))] = jmin + base + lane;
        pos += __popc(m);
      }
      if (!own) {
        if (lane == 0) row[pos] = bb;
        ++pos;
      }
      for (int x = pos + lane; x < sh.topk; x += 32) row[x] = -1;
    }
    __syncthreads();
  }
}

}  // namespace

bool rows_geom(const Shape &sh, const SelGeom &g, int dtype, RowsGeom *rg, size_t *smem) {
  if (g.n > 128 || sh.M > 128) return false;
  const bool mma = dtype == BLOSSOM_DTYPE_BF16;
  rg->cols = mma ? (g.n + 15) / 16 * 16 : (g.n + 1) / 2 * 2 + 2;
  rg->means = mma ? 3 * rg->cols * sh.D / 2 : rg->cols * (sh.D + 4);  // (a multiple of four)
  const int wide = sh.M > rg->cols ? sh.M : rg->cols;  // (per position the table also holds the scores of the selection blocks)
  rg->pitch = (sh.pq ? wide : rg->cols) | 1;
  // (Per position) warps that share rows, a head each, while tiles of 128 rows are fewer than the CTAs that fit: a warp with all
  // heads of its rows is a chain of some 3000 instructions, and its scheduler had one or two such.  With more tiles the
  // copies of the means in each CTA cost more.  us of a forward, 8 heads, with 1 | 2 | 4 heads at once:
  //   2 key/value heads, L 1500, D 64: 48 tiles 84 | 81 | 76, 192 115 | 109 | 98, 384 150 | 152 | 145, 768 209 | 211 | 213;
  //     L 600, D 32: 160 71 | 66 | 62, 640 118 | 114 | 116; L 200, D 32: 64 47 | 45 | 42, 512 88 | 87 | 87
  //   4 key/value heads, 1 | 2: L 1500, D 64: 384 79 | 75, 768 132 | 136; L 600, D 32: 320 66 | 62; L 200: 512 60 | 60
  const int64_t tiles = (int64_t)((sh.L + kRows - 1) / kRows) * sh.B * sh.Hkv;
  rg->lg_heads = 0;
  if (sh.pq && mma && tiles <= 448)
    while (rg->lg_heads < 2 && sh.G % (2 << rg->lg_heads) == 0) ++rg->lg_heads;
  const bool two = sh.pq && (sh.G > 1 || !g.plain);
  const size_t tables = (size_t)(kWarps + (two ? kWarps >> rg->lg_heads : 0)) * (mma && !sh.pq ? 16 : 32) * rg->pitch * 4;
  const size_t tail = (size_t)(8 * 128 + 2 * kWarps * 132) * 4 + kWarps * 128;
  *smem = (size_t)rg->means * 4 + (tables > tail ? tables : tail) + 16;
  // What single precision cannot certify (some percent of the blocks) the kernel decides itself while that
  // takes a CTA a few microseconds: no second launch.  With more rows, candidates or dimensions the CTA that
  // has such a block ends long after the others, unless there are waves of others behind it: a list, shared by
  // clusters of CTAs.  Time with a list / without one over 176 shapes (D 32 and 64, blocks of 16 - 64, L 256 -
  // 2048, 8 - 512 units), by the block's products x and the CTAs (740 fit on the GPU):
  //     x up to              16384   24576   32768   45056   65536  131072
  //     fewer than 1480 CTAs  1.07    1.05    0.95    0.99    0.85    0.73
  //     1480 CTAs and more    1.13    1.08    1.04    1.01    1.01    0.94
  const int64_t x = (int64_t)sh.G * sh.Bk * g.n * sh.D;
  rg->list = sh.pq || sh.G * sh.Bk > 128 || x > (tiles >= 1480 ? 65536 : 24576);
  const size_t own = ((size_t)16 * ((g.n + 1) | 1) + kWarps * 128 + 128 + 128) * 8 + 128;
  if (!rg->list && *smem < own) *smem = own;
  return *smem <= 200 * 1024;
}

template <typename T, int D>
static int launch_t(const Shape &sh, const SelGeom &g, const RowsGeom &rg, size_t smem, const T *q, const float *mean32,
                    const float *norm, const double *mean, const int32_t *seq_lens, int32_t *idx,
                    int32_t *list, int32_t *count, cudaStream_t st) {
  auto kern = sh.pq ? score_rows_kernel<T, D, true> : score_rows_kernel<T, D, false>;
  if (!allow_smem(kern, smem)) return BLOSSOM_ERR_CUDA;
  const int rows = kRows >> rg.lg_heads;
  const unsigned grid = (unsigned)((sh.L + rows - 1) / rows) * (unsigned)(sh.B * sh.Hkv);
  LaunchScope ls(K_SCORE_FAST, st);
  return launch_chained(kern, dim3(grid), dim3(kThreads), smem, st, sh, g, rg, q, mean32, norm, mean, seq_lens, idx,
                        list, count) == cudaSuccess
             ? BLOSSOM_OK
             : BLOSSOM_ERR_CUDA;
}

int launch_score_rows(const Shape &sh, const SelGeom &g, const RowsGeom &rg, size_t smem, int dtype, const void *q,
                      const float *mean32, const float *norm, const double *mean, const int32_t *seq_lens, int32_t *idx,
                      int32_t *list, int32_t *count, cudaStream_t st) {
  typedef __nv_bfloat16 bf;
  if (dtype == BLOSSOM_DTYPE_FP32) {
    if (sh.D == 32) return launch_t<float, 32>(sh, g, rg, smem, (const float *)q, mean32, norm, mean, seq_lens, idx, list, count, st);
    return launch_t<float, 64>(sh, g, rg, smem, (const float *)q, mean32, norm, mean, seq_lens, idx, list, count, st);
  }
  if (sh.D == 32) return launch_t<bf, 32>(sh, g, rg, smem, (const bf *)q, mean32, norm, mean, seq_lens, idx, list, count, st);
  return launch_t<bf, 64>(sh, g, rg, smem, (const bf *)q, mean32, norm, mean, seq_lens, idx, list, count, st);
}

}  // namespace blossom
