// Single-precision forward and backward of the fused two-branch attention (blocks of 16 and more, one
// selection per query block, per-head gate).
//
// The tolerance of fp32 inputs rules out a tensor-core product of rounded operands (one of bf16 or TF32; three
// bf16 parts per operand, six products, would do, and have not been tried), so the products are register tiles
// of packed fp32 multiply-adds.  A warp owns 16 query rows (forward, dQ) or 16 keys (dK/dV) of a head and
// walks the 16-position chunks that its block selected (or was selected by) or its window reaches, with the
// next chunk's rows on their way by cp.async: no barrier between warps, any number of warps per CTA.  A
// chunk in both branches costs one S product and, in the forward, one exponential per pair (as in
// attn_short_fwd.cu: a common reference, checked at the end).  The layout of a 16 x 16 tile over a warp is
// that of a warp-level matrix product (rows lane / 4 and lane / 4 + 8, columns 2 (lane % 4) + {0, 1, 8, 9}),
// so the mask helpers of the short-history kernels serve here too; probabilities pass through shared
// memory into the second products, where a lane owns float4 columns 16 n + 4 (lane % 4).
// The kernels that these replace (four lanes a row, a chain of maximum, two exponentials and two
// shuffles per key) took 48 + 60 + 108 us at B 128, H 2, L 200, D 32, padded; bound by that chain and by CTAs
// of 64 threads, not by their 13 us of multiply-adds.
#include "short_common.cuh"

namespace blossom {
namespace f32 {
namespace {

using namespace sh;

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }

constexpr int kPP = 20;  // pitch of a 16 x 16 tile in shared memory (floats)
template <int D>
struct Geo {
  static constexpr int P = D + 4;       // pitch of a row (floats): the reads below are free of conflicts
  static constexpr int kTile = 16 * P;  // floats of a 16-row tile
};

// rows r0 .. r0 + 15 of a [.][D] tensor into a tile, rows outside [lo, hi) as zeros
template <int D>
__device__ __forceinline__ void fetch(float *tile, const float *base, int64_t sl, int r0, int lo, int hi, int lane) {
#pragma unroll
  for (int i = 0; i < D / 8; ++i) {
    const int e = i * 32 + lane, r = e / (D / 4), ch = e % (D / 4), p = r0 + r;
    float *dst = tile + r * Geo<D>::P + ch * 4;
    if (p >= lo && p < hi) cp_async16(smem_addr(dst), base + (int64_t)p * sl + ch * 4);
    else *reinterpret_cast<float4 *>(dst) = make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

// s = A (16 x D) B^T (16 x D), both tiles in shared memory
template <int D>
__device__ __forceinline__ void product_s(const float *a, const float *b, int gid, int tig, float (&s)[2][4]) {
  constexpr int P = Geo<D>::P;
  float2 acc[2][4];
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[nt][e] = make_float2(0.f, 0.f);
  const float *a0 = a + gid * P, *a1 = a0 + 8 * P, *bt = b + 2 * tig * P;
#pragma unroll 4
  for (int d = 0; d < D; d += 4) {
    const float4 x0 = *reinterpret_cast<const float4 *>(a0 + d), x1 = *reinterpret_cast<const float4 *>(a1 + d);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const float4 y = *reinterpret_cast<const float4 *>(bt + (8 * nt + j) * P + d);
        acc[nt][j] = fma2(make_float2(x0.x, x0.y), make_float2(y.x, y.y), acc[nt][j]);
        acc[nt][2 + j] = fma2(make_float2(x1.x, x1.y), make_float2(y.x, y.y), acc[nt][2 + j]);
        acc[nt][j] = fma2(make_float2(x0.z, x0.w), make_float2(y.z, y.w), acc[nt][j]);
        acc[nt][2 + j] = fma2(make_float2(x1.z, x1.w), make_float2(y.z, y.w), acc[nt][2 + j]);
      }
  }
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[nt][e] = acc[nt][e].x + acc[nt][e].y;
}

// a warp's 16 x 16 tile -> shared memory
__device__ __forceinline__ void put_tile(float *t, const float (&p)[2][4], int gid, int tig) {
#pragma unroll
  for (int nt = 0; nt < 2; ++nt)
#pragma unroll
    for (int i = 0; i < 2; ++i)
      *reinterpret_cast<float2 *>(t + (gid + 8 * i) * kPP + 8 * nt + 2 * tig) = make_float2(p[nt][2 * i], p[nt][2 * i + 1]);
}

// 16 rows x D of one output: rows gid, gid + 8; columns 16 n + 4 tig .. + 3
template <int D>
struct Acc {
  float2 v[2][D / 16][2];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int n = 0; n < D / 16; ++n) v[i][n][0] = v[i][n][1] = make_float2(0.f, 0.f);
  }
  __device__ __forceinline__ void scale(float f0, float f1) {
#pragma unroll
    for (int n = 0; n < D / 16; ++n)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        v[0][n][j].x *= f0; v[0][n][j].y *= f0;
        v[1][n][j].x *= f1; v[1][n][j].y *= f1;
      }
  }
  // += T (16 x 16 tile in shared memory) times the 16 rows of tile b
  __device__ __forceinline__ void add(const float *t, const float *b, int gid, int tig) {
#pragma unroll 1
    for (int k = 0; k < 16; k += 4) {
      const float4 t0 = *reinterpret_cast<const float4 *>(t + gid * kPP + k);
      const float4 t1 = *reinterpret_cast<const float4 *>(t + (gid + 8) * kPP + k);
      const float w0[4] = {t0.x, t0.y, t0.z, t0.w}, w1[4] = {t1.x, t1.y, t1.z, t1.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
#pragma unroll
        for (int n = 0; n < D / 16; ++n) {
          const float4 y = *reinterpret_cast<const float4 *>(b + (k + e) * Geo<D>::P + 16 * n + 4 * tig);
          v[0][n][0] = fma2(dup(w0[e]), make_float2(y.x, y.y), v[0][n][0]);
          v[0][n][1] = fma2(dup(w0[e]), make_float2(y.z, y.w), v[0][n][1]);
          v[1][n][0] = fma2(dup(w1[e]), make_float2(y.x, y.y), v[1][n][0]);
          v[1][n][1] = fma2(dup(w1[e]), make_float2(y.z, y.w), v[1][n][1]);
        }
    }
  }
  // += the accumulators the other warps of the tile left in shared memory, and leaving one there
  __device__ __forceinline__ void put(float *b, int lane) const {
    float2 *o = reinterpret_cast<float2 *>(b) + lane;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int n = 0; n < D / 16; ++n)
#pragma unroll
        for (int j = 0; j < 2; ++j) o[32 * ((i * (D / 16) + n) * 2 + j)] = v[i][n][j];
  }
  __device__ __forceinline__ void take(const float *b, int lane) {
    const float2 *o = reinterpret_cast<const float2 *>(b) + lane;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int n = 0; n < D / 16; ++n)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float2 x = o[32 * ((i * (D / 16) + n) * 2 + j)];
          v[i][n][j].x += x.x;
          v[i][n][j].y += x.y;
        }
  }
  static constexpr int kFloats = 16 * D;  // of one accumulator in shared memory
  // rows r0 + gid, r0 + gid + 8 (those < hi) of a tensor
  __device__ __forceinline__ void store(float *base, int64_t sl, int r0, int hi, float f0, float f1, int gid, int tig) const {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int r = r0 + gid + 8 * i;
      const float f = i ? f1 : f0;
      if (r < hi)
#pragma unroll
        for (int n = 0; n < D / 16; ++n)
          *reinterpret_cast<float4 *>(base + (int64_t)r * sl + 16 * n + 4 * tig) =
              make_float4(v[i][n][0].x * f, v[i][n][0].y * f, v[i][n][1].x * f, v[i][n][1].y * f);
    }
  }
};

// The chunks of 16 positions a warp visits, 64 at a time (bit = chunk): sets(w) fills L and S for chunks
// 64 w ...; next() hands out every split-th of them (the sub-th, ...) in ascending order, -1 at the end.
template <typename F>
struct Walk {
  F sets;
  int w, nw, skip, sub, split, count;
  uint64_t L, S, todo;
  __device__ __forceinline__ Walk(F f, int nw_, int skip_, int sub_, int split_)
      : sets(f), w(-1), nw(nw_), skip(skip_), sub(sub_), split(split_), count(0), L(0), S(0), todo(0) {}
  __device__ __forceinline__ int next(bool *inL, bool *inS) {
    while (true) {
      while (!todo) {
        if (++w >= nw) return -1;
        sets(w, L, S);
        todo = L | S;
        if (skip >= 0 && (skip >> 6) == w) todo &= ~(1ull << (skip & 63));
      }
      const int b = __ffsll((long long)todo) - 1;
      todo &= todo - 1;
      const bool mine = count == sub;
      if (++count == split) count = 0;
      if (!mine) continue;
      *inL = (L >> b) & 1;
      *inS = (S >> b) & 1;
      return 64 * w + b;
    }
  }
};
template <typename F>
__device__ __forceinline__ Walk<F> make_walk(F f, int nw, int skip, int sub, int split) {
  return Walk<F>(f, nw, skip, sub, split);
}

// chunk sets of a query tile: the blocks its block selected, the chunks its rows' window touches
__device__ __forceinline__ void query_sets(const Shape &s, const int32_t *idxrow, int b, int t0, int t_last, int pad0, int w,
                                           int lane, uint64_t &L, uint64_t &S) {
  const int cpb = s.Bk >> 4;  // chunks per block
  uint64_t l = 0ull;
  for (int i = lane; i < s.topk; i += 32) {
    const int j = idxrow[i];
    if (j >= 0 && j < s.M && (j <= b || !s.causal)) {
      const int c = j * cpb - 64 * w;
      if (c >= 0 && c < 64) l |= (cpb == 4 ? 0xfull : cpb == 2 ? 3ull : 1ull) << c;
    }
  }
  l = (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)l) | ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(l >> 32)) << 32);
  bool in[2], fs[2];
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int p = (64 * w + lane + 32 * x) * 16;
    in[x] = p + 15 >= pad0 && p < s.L && (!s.causal || p <= t_last);
    fs[x] = in[x] && st_ranges_touch(s, max(t0, pad0), t_last, p, min(p + 15, s.L - 1));
  }
  L = l & ballot64(in[0], in[1]);
  S = ballot64(fs[0], fs[1]);
}
// The pairs of query tile t0 and key chunk p0 that take part in a branch: 16 key columns per row, shifted so
// that this thread's are bits 0, 1, 8, 9 (rows t0 + gid, t0 + gid + 8).
template <bool PLAIN>
__device__ __forceinline__ void query_masks(const Shape &s, int t0, int p0, int pad0, bool inL, bool inS, int gid, int tig,
                                            uint32_t (&bL)[2], uint32_t (&bS)[2]) {
  const bool causal = PLAIN || s.causal;
  const bool past = t0 >= pad0 && t0 + 15 < s.L && p0 >= pad0 && (causal ? p0 + 15 <= t0 : p0 + 15 < s.L);
  const bool win = t0 + 15 - p0 < s.window && (causal || p0 + 15 - t0 < s.window);
  bL[0] = bL[1] = bS[0] = bS[1] = 0xffffu;
  if (!past || (inS && !win)) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = t0 + gid + 8 * i;
      bL[i] = (past ? 0xffffu : t >= pad0 && t < s.L ? cols16(pad0 - p0, (causal ? t : s.L - 1) - p0) : 0u) >> (2 * tig);
      bS[i] = win ? bL[i] : bL[i] & (st_keys16<PLAIN>(s, t, p0, causal) >> (2 * tig));
    }
  }
  if (!inL) bL[0] = bL[1] = 0u;
  if (!inS) bS[0] = bS[1] = 0u;
}
__device__ __forceinline__ bool pair_on(const uint32_t (&b)[2], int e) {  // e = 4 nt + 2 i + j
  return (b[(e >> 1) & 1] >> ((e >> 2) * 8 + (e & 1))) & 1u;
}

// ------------------------------------------------------------------------------------ forward
template <int D, bool PLAIN>
__global__ void __launch_bounds__(128) fwd_f32_kernel(Shape s, const float *__restrict__ q, const float *__restrict__ k,
                                                      const float *__restrict__ v, const float *__restrict__ gate,
                                                      const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ idx,
                                                      float *__restrict__ out, float *__restrict__ out_lt,
                                                      float *__restrict__ out_st, float *__restrict__ lse, int split) {
  grid_chain_enter();
  extern __shared__ __align__(16) float fsm[];
  constexpr int T = Geo<D>::kTile, kWarp = 5 * T + 2 * 16 * kPP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  float *qt = fsm + warp * kWarp, *kv = qt + T, *pl = kv + 4 * T, *ps = pl + 16 * kPP;  // kv: [2 stages][K, V]
  const int units = s.B * s.H, ntile = (s.L + 15) >> 4;
  const int sub = split > 1 ? warp : 0;  // with split > 1 the CTA's warps share one tile's chunks
  const int64_t task = split > 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  if (task >= (int64_t)units * ntile) return;
  const int u = (int)(task % units), t0 = (ntile - 1 - (int)(task / units)) * 16;  // late tiles first
  const int n = u / s.H, h = u % s.H, hk = h / s.G;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len, t_last = min(t0 + 15, s.L - 1), b = t0 / s.Bk;
  const int64_t off = row_offset(s, n, h, 0), koff = row_offset_kv(s, n, hk, 0);
  const float alpha = head_alpha(gate, h), beta = 1.f - alpha, sc2 = s.scale * kLog2e;
  Acc<D> aL, aS;
  aL.zero();
  aS.zero();
  float l[4] = {0.f, 0.f, 0.f, 0.f};  // sums {long-term rows gid, gid + 8, short-term rows ...}
  float mL[2] = {0.f, 0.f}, mS[2] = {0.f, 0.f};
  if (t_last >= pad0) {
    const int32_t *idxrow = idx + (((int64_t)n * s.Hkv + hk) * s.M + b) * s.topk;
    const int nw = (ntile + 63) >> 6, own = t0 >> 4;
    auto sets = [&](int w, uint64_t &L, uint64_t &S) { query_sets(s, idxrow, b, t0, t_last, pad0, w, lane, L, S); };
    auto load = [&](int c, int st) {
      fetch<D>(kv + 2 * st * T, k + koff, s.ksl, c * 16, pad0, s.L, lane);
      fetch<D>(kv + (2 * st + 1) * T, v + koff, s.ksl, c * 16, pad0, s.L, lane);
      cp_async_commit();
    };
    fetch<D>(qt, q + off, s.sl, t0, pad0, s.L, lane);
    load(own, 0);
    // The tile's own chunk first (it holds every row's own key): its maximum is the reference of both
    // branches for all chunks; the sums show at the end whether that was near enough.
    float m[2];
    bool inL, inS;
    {
      uint64_t L, S;
      sets(own >> 6, L, S);
      inL = (L >> (own & 63)) & 1;
      inS = (S >> (own & 63)) & 1;
    }
    auto walk = make_walk(sets, nw, own, sub, split);
    int c = own, st = 0;
    bool first = true;
#pragma unroll 1
    while (c >= 0) {
      bool nL = false, nS = false;
      const int cn = walk.next(&nL, &nS);
      if (cn >= 0) {
        load(cn, st ^ 1);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();
      const float *kt = kv + 2 * st * T, *vt = kt + T;
      uint32_t bL[2], bS[2];
      query_masks<PLAIN>(s, t0, c * 16, pad0, inL, inS, gid, tig, bL, bS);
      float z[2][4];
      product_s<D>(qt, kt, gid, tig, z);
      if (first) {
        float cm[2] = {-INFINITY, -INFINITY};
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (pair_on(bL, e) || pair_on(bS, e)) cm[(e >> 1) & 1] = fmaxf(cm[(e >> 1) & 1], z[e >> 2][e & 3]);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float x = quad_max(cm[i]) * sc2;
          m[i] = x > -INFINITY ? x : 0.f;
        }
        first = false;
        if (sub) {  // (every warp of the tile needs the reference; the first one adds the chunk)
          inL = inS = false;
          bL[0] = bL[1] = bS[0] = bS[1] = 0u;
        }
      }
      float pL[2][4], pS[2][4];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int i = (e >> 1) & 1;
        const float x = exp2f(fmaf(z[e >> 2][e & 3], sc2, -m[i]));
        pL[e >> 2][e & 3] = pair_on(bL, e) ? x : 0.f;
        pS[e >> 2][e & 3] = pair_on(bS, e) ? x : 0.f;
        l[i] += pL[e >> 2][e & 3];
        l[2 + i] += pS[e >> 2][e & 3];
      }
      if (inL) put_tile(pl, pL, gid, tig);
      if (inS) put_tile(ps, pS, gid, tig);
      __syncwarp();
      if (inL) aL.add(pl, vt, gid, tig);
      if (inS) aS.add(ps, vt, gid, tig);
      __syncwarp();  // the stage and the tiles are free again
      c = cn;
      inL = nL;
      inS = nS;
      st ^= 1;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) l[i] = quad_sum(l[i]);
    if (split > 1) {
      constexpr int F = Acc<D>::kFloats;
      if (sub) {
        aL.put(kv, lane);
        aS.put(kv + F, lane);
        *reinterpret_cast<float4 *>(kv + 2 * F + 4 * lane) = make_float4(l[0], l[1], l[2], l[3]);
      }
      __syncthreads();
      if (sub) return;
      for (int w = 1; w < split; ++w) {  // in warp order
        const float *o = kv + w * kWarp;
        aL.take(o, lane);
        aS.take(o + F, lane);
        const float4 x = *reinterpret_cast<const float4 *>(o + 2 * F + 4 * lane);
        l[0] += x.x; l[1] += x.y; l[2] += x.z; l[3] += x.w;
      }
    }
    mL[0] = mS[0] = m[0];
    mL[1] = mS[1] = m[1];
    bool bad = false;
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (t0 + gid + 8 * i >= pad0 && t0 + gid + 8 * i < s.L)
        bad |= !(fminf(l[i], l[2 + i]) > 1e-24f && fmaxf(l[i], l[2 + i]) < 1e24f);
    if (__any_sync(0xffffffffu, bad)) {
      // Logits spread too far for one reference (or a branch without a key): the rows once more with a
      // running maximum, one branch after the other (branch 0 through aS, then moved to aL).
#pragma unroll 1
      for (int br = 0; br < 2; ++br) {
        if (br) aL = aS;
        aS.zero();
        float mm[2] = {-INFINITY, -INFINITY}, ll[2] = {0.f, 0.f};
#pragma unroll 1
        for (int w = 0; w < nw; ++w) {
          uint64_t L, S;
          sets(w, L, S);
#pragma unroll 1
          for (uint64_t todo = br ? S : L; todo; todo &= todo - 1) {
            const int p0 = (64 * w + __ffsll((long long)todo) - 1) * 16;
            load(p0 >> 4, 0);
            cp_async_wait<0>();
            __syncwarp();
            uint32_t b0[2], b1[2];
            query_masks<PLAIN>(s, t0, p0, pad0, br == 0, br == 1, gid, tig, b0, b1);
            float z[2][4], fac[2];
            product_s<D>(qt, kv, gid, tig, z);
            float cm[2] = {-INFINITY, -INFINITY};
#pragma unroll
            for (int e = 0; e < 8; ++e)
              if (pair_on(b0, e) || pair_on(b1, e)) cm[(e >> 1) & 1] = fmaxf(cm[(e >> 1) & 1], z[e >> 2][e & 3]);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float x = fmaxf(mm[i], quad_max(cm[i]) * sc2);
              fac[i] = x > -INFINITY ? exp2f(mm[i] - x) : 1.f;
              mm[i] = x;
              ll[i] *= fac[i];
            }
            aS.scale(fac[0], fac[1]);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int i = (e >> 1) & 1;
              const float x = pair_on(b0, e) || pair_on(b1, e) ? exp2f(fmaf(z[e >> 2][e & 3], sc2, -mm[i])) : 0.f;
              z[e >> 2][e & 3] = x;
              ll[i] += x;
            }
            put_tile(pl, z, gid, tig);
            __syncwarp();
            aS.add(pl, kv + T, gid, tig);
            __syncwarp();
          }
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          ll[i] = quad_sum(ll[i]);
          if (br) {
            l[2 + i] = ll[i];
            mS[i] = mm[i];
          } else {
            l[i] = ll[i];
            mL[i] = mm[i];
          }
        }
      }
    }
  }
  if (sub) return;  // (a tile of padding)
  // normalise, mix (Eq. 19), store; padded rows are zeros
  float f[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) f[i] = l[i] > 0.f ? 1.f / l[i] : 0.f;
  aL.scale(f[0], f[1]);
  aS.scale(f[2], f[3]);
  if (out_lt) {
    aL.store(out_lt + off, s.sl, t0, s.L, 1.f, 1.f, gid, tig);
    aS.store(out_st + off, s.sl, t0, s.L, 1.f, 1.f, gid, tig);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int x = 0; x < D / 16; ++x)
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        aL.v[i][x][j].x = alpha * aL.v[i][x][j].x + beta * aS.v[i][x][j].x;
        aL.v[i][x][j].y = alpha * aL.v[i][x][j].y + beta * aS.v[i][x][j].y;
      }
  aL.store(out + off, s.sl, t0, s.L, 1.f, 1.f, gid, tig);
  if (lse && tig == 0) {
    const int64_t BHL = (int64_t)s.B * s.H * s.L;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int t = t0 + gid + 8 * i;
      if (t < s.L) {
        const int64_t row = (int64_t)u * s.L + t;
        lse[row] = l[i] > 0.f ? (mL[i] + log2f(l[i])) * kLn2 : 0.f;
        lse[BHL + row] = l[2 + i] > 0.f ? (mS[i] + log2f(l[2 + i])) * kLn2 : 0.f;
      }
    }
  }
}

// ------------------------------------------------------------------------------------ dQ
// Also the records {lse_lt, lse_st (log2 units), Delta_lt, Delta_st (weighted)} of every row for the dK/dV
// kernel, and a partial of d alpha per tile.
template <int D, bool PLAIN>
__global__ void __launch_bounds__(128) dq_f32_kernel(Shape s, const float *__restrict__ q, const float *__restrict__ k,
                                                     const float *__restrict__ v, const float *__restrict__ gate,
                                                     const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ idx,
                                                     const float *__restrict__ out_lt, const float *__restrict__ out_st,
                                                     const float *__restrict__ lse, const float *__restrict__ dout,
                                                     float *__restrict__ dq, float4 *__restrict__ records,
                                                     double *__restrict__ dalpha_part, int split) {
  grid_chain_enter();
  extern __shared__ __align__(16) float fsm[];
  constexpr int T = Geo<D>::kTile, kWarp = 6 * T + 16 * kPP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3;
  float *qt = fsm + warp * kWarp, *gt = qt + T, *kv = gt + T, *pt = kv + 4 * T;
  const int units = s.B * s.H, ntile = (s.L + 15) >> 4;
  const int sub = split > 1 ? warp : 0;  // with split > 1 the CTA's warps share one tile's chunks
  const int64_t task = split > 1 ? (int64_t)blockIdx.x : (int64_t)blockIdx.x * (blockDim.x >> 5) + warp;
  if (task >= (int64_t)units * ntile) return;
  const int u = (int)(task % units), tile = ntile - 1 - (int)(task / units), t0 = tile * 16;
  const int n = u / s.H, h = u % s.H, hk = h / s.G, Lpad = (s.L + 63) / 64 * 64;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len, t_last = min(t0 + 15, s.L - 1), b = t0 / s.Bk;
  const int64_t off = row_offset(s, n, h, 0), koff = row_offset_kv(s, n, hk, 0);
  const float alpha = head_alpha(gate, h), beta = 1.f - alpha, sc2 = s.scale * kLog2e;
  Acc<D> acc;
  acc.zero();
  float dal = 0.f;
  if (t_last >= pad0) {
    const int32_t *idxrow = idx + (((int64_t)n * s.Hkv + hk) * s.M + b) * s.topk;
    auto sets = [&](int w, uint64_t &L, uint64_t &S) { query_sets(s, idxrow, b, t0, t_last, pad0, w, lane, L, S); };
    auto load = [&](int c, int st) {
      fetch<D>(kv + 2 * st * T, k + koff, s.ksl, c * 16, pad0, s.L, lane);
      fetch<D>(kv + (2 * st + 1) * T, v + koff, s.ksl, c * 16, pad0, s.L, lane);
      cp_async_commit();
    };
    fetch<D>(qt, q + off, s.sl, t0, pad0, s.L, lane);
    fetch<D>(gt, dout + off, s.sl, t0, pad0, s.L, lane);
    cp_async_commit();
    auto walk = make_walk(sets, (ntile + 63) >> 6, -1, sub, split);
    bool inL = false, inS = false;
    int c = walk.next(&inL, &inS), st = 0;
    if (c >= 0) load(c, 0);
    // Delta of the tile's rows: lanes 2 r, 2 r + 1 take the halves of row r
    float l2[4], dl[4];  // {long-term rows gid, gid + 8, short-term rows ...}
    {
      const int r = lane >> 1, t = t0 + r;
      const bool ok = t >= pad0 && t < s.L;
      const int64_t o = off + (int64_t)(ok ? t : t_last) * s.sl + (lane & 1) * (D / 2);
      float a = 0.f, c2 = 0.f;
#pragma unroll 4
      for (int e = 0; e < D / 2; e += 4) {
        const float4 g = *reinterpret_cast<const float4 *>(dout + o + e);
        const float4 x = *reinterpret_cast<const float4 *>(out_lt + o + e), y = *reinterpret_cast<const float4 *>(out_st + o + e);
        a = fmaf(g.x, x.x, a); a = fmaf(g.y, x.y, a); a = fmaf(g.z, x.z, a); a = fmaf(g.w, x.w, a);
        c2 = fmaf(g.x, y.x, c2); c2 = fmaf(g.y, y.y, c2); c2 = fmaf(g.z, y.z, c2); c2 = fmaf(g.w, y.w, c2);
      }
      a += __shfl_xor_sync(0xffffffffu, a, 1);
      c2 += __shfl_xor_sync(0xffffffffu, c2, 1);
      const int64_t row = (int64_t)u * s.L + (ok ? t : t_last), BHL = (int64_t)s.B * s.H * s.L;
      float4 rec = make_float4(lse[row] * kLog2e, lse[BHL + row] * kLog2e, alpha * a, beta * c2);
      if (!ok) rec = make_float4(0.f, 0.f, 0.f, 0.f);
      if ((lane & 1) == 0 && t < Lpad && !sub) records[(int64_t)u * Lpad + t] = rec;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int src = 2 * (gid + 8 * i);
        l2[i] = __shfl_sync(0xffffffffu, rec.x, src);
        l2[2 + i] = __shfl_sync(0xffffffffu, rec.y, src);
        dl[i] = __shfl_sync(0xffffffffu, rec.z, src);
        dl[2 + i] = __shfl_sync(0xffffffffu, rec.w, src);
      }
    }
#pragma unroll 1
    while (c >= 0) {
      bool nL = false, nS = false;
      const int cn = walk.next(&nL, &nS);
      if (cn >= 0) {
        load(cn, st ^ 1);
        cp_async_wait<1>();
      } else {
        cp_async_wait<0>();
      }
      __syncwarp();
      const float *kt = kv + 2 * st * T, *vt = kt + T;
      uint32_t bL[2], bS[2];
      query_masks<PLAIN>(s, t0, c * 16, pad0, inL, inS, gid, tig, bL, bS);
      float z[2][4], dp[2][4];
      product_s<D>(qt, kt, gid, tig, z);
      product_s<D>(gt, vt, gid, tig, dp);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int i = (e >> 1) & 1;
        const float zz = z[e >> 2][e & 3], dd = dp[e >> 2][e & 3];
        const float x = pair_on(bL, e) ? exp2f(fmaf(zz, sc2, -l2[i])) : 0.f;
        const float y = pair_on(bS, e) ? exp2f(fmaf(zz, sc2, -l2[2 + i])) : 0.f;
        dal = fmaf(x - y, dd, dal);
        z[e >> 2][e & 3] = fmaf(x, fmaf(alpha, dd, -dl[i]), y * fmaf(beta, dd, -dl[2 + i]));
      }
      put_tile(pt, z, gid, tig);
      __syncwarp();
      acc.add(pt, kt, gid, tig);
      __syncwarp();
      c = cn;
      inL = nL;
      inS = nS;
      st ^= 1;
    }
    if (split > 1) {
      if (sub) {
        acc.put(kv, lane);
        kv[Acc<D>::kFloats + lane] = dal;
      }
      __syncthreads();
      if (!sub)
        for (int w = 1; w < split; ++w) {
          const float *o = kv + w * kWarp;
          acc.take(o, lane);
          dal += o[Acc<D>::kFloats + lane];
        }
    }
  } else if (lane < 16 && t0 + lane < Lpad) {
    records[(int64_t)u * Lpad + t0 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  if (sub) return;
  acc.store(dq + off, s.sl, t0, s.L, s.scale, s.scale, gid, tig);
  double a = (double)dal;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) dalpha_part[(int64_t)u * ntile + tile] = a;
}

// ------------------------------------------------------------------------------------ dK, dV
// The first CTA reduces the gate gradient instead (one warp per head, fixed order).
template <int D, bool PLAIN>
__global__ void __launch_bounds__(128) dkdv_f32_kernel(Shape s, const float *__restrict__ q, const float *__restrict__ k,
                                                       const float *__restrict__ v, const float *__restrict__ gate,
                                                       const int32_t *__restrict__ seq_lens, const int32_t *__restrict__ idx,
                                                       const float4 *__restrict__ records, const float *__restrict__ dout,
                                                       float *__restrict__ dk, float *__restrict__ dv,
                                                       const double *__restrict__ dalpha_part, float *__restrict__ dgate,
                                                       int split) {
  grid_chain_enter();
  extern __shared__ __align__(16) float fsm[];
  constexpr int T = Geo<D>::kTile, kStage = 2 * T + 64, kWarp = 2 * T + 2 * kStage + 2 * 16 * kPP;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, gid = lane >> 2, tig = lane & 3, nwarp = blockDim.x >> 5;
  const int ntile = (s.L + 15) >> 4;
  if (blockIdx.x == 0) {
    for (int h = warp; h < s.H; h += nwarp) {
      double a = 0.0;
#pragma unroll 8
      for (int i = lane; i < s.B * ntile; i += 32) a += dalpha_part[((int64_t)(i / ntile) * s.H + h) * ntile + i % ntile];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) {
        const double al = 1.0 / (1.0 + exp(-((double)gate[h * 2 + 0] - (double)gate[h * 2 + 1])));
        const double g0 = al * (1.0 - al) * a;
        dgate[h * 2 + 0] = (float)g0;
        dgate[h * 2 + 1] = (float)(-g0);
      }
    }
    return;
  }
  float *kt = fsm + warp * kWarp, *vt = kt + T, *stages = vt + T, *wt = stages + 2 * kStage, *dt = wt + 16 * kPP;
  const bool causal = PLAIN || s.causal;
  const int units = s.B * s.Hkv;
  const int sub = split > 1 ? warp : 0;  // with split > 1 the CTA's warps share one tile's chunks
  const int64_t task = split > 1 ? (int64_t)blockIdx.x - 1 : (int64_t)(blockIdx.x - 1) * nwarp + warp;
  if (task >= (int64_t)units * ntile) return;
  const int uk = (int)(task % units), p0 = (int)(task / units) * 16;  // early keys (the most visitors) first
  const int n = uk / s.Hkv, hk = uk % s.Hkv, Lpad = (s.L + 63) / 64 * 64;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len, p_last = min(p0 + 15, s.L - 1), j = p0 / s.Bk;
  const int64_t koff = row_offset_kv(s, n, hk, 0);
  const float sc2 = s.scale * kLog2e;
  Acc<D> ak, av;
  ak.zero();
  av.zero();
  if (p_last >= pad0) {
    // the query chunks whose block selected this key block, or whose window touches these keys
    auto sets = [&](int w, uint64_t &L, uint64_t &S) {
      const int cpb = s.Bk >> 4;
      uint64_t l = 0ull;
      for (int qb = 64 * w / cpb + lane; qb < min(s.M, 64 * (w + 1) / cpb); qb += 32) {
        if (causal && qb < j) continue;
        const int32_t *row = idx + ((int64_t)uk * s.M + qb) * s.topk;
        bool sel = false;
        for (int i = 0; i < s.topk; ++i) sel |= row[i] == j;
        if (sel) l |= (cpb == 4 ? 0xfull : cpb == 2 ? 3ull : 1ull) << (qb * cpb - 64 * w);
      }
      l = (uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)l) |
          ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(l >> 32)) << 32);
      bool in[2], fs[2];
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int t = (64 * w + lane + 32 * x) * 16, tl = min(t + 15, s.L - 1);
        in[x] = t < s.L && tl >= pad0 && (!causal || tl >= p0);
        fs[x] = in[x] && st_ranges_touch(s, t, tl, max(p0, pad0), p_last);
      }
      L = l & ballot64(in[0], in[1]);
      S = ballot64(fs[0], fs[1]);
    };
    fetch<D>(kt, k + koff, s.ksl, p0, pad0, s.L, lane);
    fetch<D>(vt, v + koff, s.ksl, p0, pad0, s.L, lane);
    cp_async_commit();
#pragma unroll 1
    for (int hg = 0; hg < s.G; ++hg) {
      const int h = hk * s.G + hg;
      const int64_t off = row_offset(s, n, h, 0), u = (int64_t)n * s.H + h;
      const float alpha = head_alpha(gate, h), beta = 1.f - alpha;
      auto load = [&](int c, int st) {
        float *x = stages + st * kStage;
        fetch<D>(x, q + off, s.sl, c * 16, pad0, s.L, lane);
        fetch<D>(x + T, dout + off, s.sl, c * 16, pad0, s.L, lane);
        if (lane < 16) cp_async16(smem_addr(x + 2 * T + 4 * lane), records + u * Lpad + c * 16 + lane);
        cp_async_commit();
      };
      auto walk = make_walk(sets, (ntile + 63) >> 6, -1, sub, split);
      bool inL = false, inS = false;
      int c = walk.next(&inL, &inS), st = 0;
      if (c >= 0) load(c, 0);
#pragma unroll 1
      while (c >= 0) {
        bool nL = false, nS = false;
        const int cn = walk.next(&nL, &nS);
        if (cn >= 0) {
          load(cn, st ^ 1);
          cp_async_wait<1>();
        } else {
          cp_async_wait<0>();
        }
        __syncwarp();
        const float *qt = stages + st * kStage, *gt = qt + T;
        const float4 *rec = reinterpret_cast<const float4 *>(gt + T) + 2 * tig;
        const int t0 = c * 16;
        const bool past = p0 >= pad0 && p0 + 15 < s.L && t0 >= pad0 && t0 + 15 < s.L && (!causal || t0 >= p0 + 15);
        uint32_t bL[2] = {0xffffu, 0xffffu}, bS[2] = {0xffffu, 0xffffu};
        if (!past)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int p = p0 + gid + 8 * i;
            bL[i] = bS[i] = p >= pad0 && p < s.L ? cols16((causal ? p : pad0) - t0, s.L - 1 - t0) >> (2 * tig) : 0u;
          }
        if (inS && !(past && t0 + 15 - p0 < s.window && (causal || p0 + 15 - t0 < s.window)))
#pragma unroll
          for (int i = 0; i < 2; ++i) bS[i] &= st_queries16<PLAIN>(s, p0 + gid + 8 * i, t0, causal) >> (2 * tig);
        if (!inL) bL[0] = bL[1] = 0u;
        if (!inS) bS[0] = bS[1] = 0u;
        float z[2][4], dp[2][4];
        product_s<D>(kt, qt, gid, tig, z);
        product_s<D>(vt, gt, gid, tig, dp);
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int nt = x >> 1, jj = x & 1;
          const float4 r = rec[nt * 8 + jj];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int e = 4 * nt + 2 * i + jj;
            const float zz = z[nt][2 * i + jj], dd = dp[nt][2 * i + jj];
            const float a = pair_on(bL, e) ? exp2f(fmaf(zz, sc2, -r.x)) : 0.f;
            const float bb = pair_on(bS, e) ? exp2f(fmaf(zz, sc2, -r.y)) : 0.f;
            dp[nt][2 * i + jj] = fmaf(a, fmaf(alpha, dd, -r.z), bb * fmaf(beta, dd, -r.w));
            z[nt][2 * i + jj] = alpha * a + beta * bb;
          }
        }
        put_tile(wt, z, gid, tig);
        put_tile(dt, dp, gid, tig);
        __syncwarp();
        av.add(wt, gt, gid, tig);
        ak.add(dt, qt, gid, tig);
        __syncwarp();
        c = cn;
        inL = nL;
        inS = nS;
        st ^= 1;
      }
    }
    cp_async_wait<0>();
    if (split > 1) {
      if (sub) {
        ak.put(stages, lane);
        av.put(stages + Acc<D>::kFloats, lane);
      }
      __syncthreads();
      if (!sub)
        for (int w = 1; w < split; ++w) {
          const float *o = stages + w * kWarp;
          ak.take(o, lane);
          av.take(o + Acc<D>::kFloats, lane);
        }
    }
  }
  if (sub) return;
  av.store(dv + koff, s.ksl, p0, s.L, 1.f, 1.f, gid, tig);
  ak.store(dk + koff, s.ksl, p0, s.L, s.scale, s.scale, gid, tig);
}

// CTAs are four warps.  While the tiles leave SMs without work a CTA's warps share one tile's chunks
// instead of taking a tile each: the tile with the most chunks is then the kernel's time.
constexpr int kCtaWarps = 4;
int chunk_split(int64_t tasks) { return tasks <= 148 * 6 ? kCtaWarps : 1; }
unsigned ctas(int64_t tasks, int split) { return (unsigned)(split > 1 ? tasks : (tasks + kCtaWarps - 1) / kCtaWarps); }

template <int D>
int launch_fwd_t(const Shape &s, const float *q, const float *k, const float *v, const float *gate, const int32_t *seq_lens,
                 const int32_t *idx, float *out, float *out_lt, float *out_st, float *lse, cudaStream_t st) {
  const bool plain = s.causal && s.stis_mode == 0;
  auto kern = plain ? fwd_f32_kernel<D, true> : fwd_f32_kernel<D, false>;
  const int64_t tasks = (int64_t)s.B * s.H * ((s.L + 15) / 16);
  const int split = chunk_split(tasks);
  const size_t smem = (size_t)kCtaWarps * (5 * Geo<D>::kTile + 2 * 16 * kPP) * sizeof(float);
  if (!allow_smem(kern, smem)) return BLOSSOM_ERR_CUDA;
  LaunchScope ls(K_FWD_SIMT, st);
  return launch_chained(kern, dim3(ctas(tasks, split)), dim3(32 * kCtaWarps), smem, st, s, q, k, v, gate, seq_lens, idx, out,
                        out_lt, out_st, lse, split) == cudaSuccess
             ? BLOSSOM_OK
             : BLOSSOM_ERR_CUDA;
}

template <int D>
int launch_bwd_t(const Shape &s, const float *q, const float *k, const float *v, const float *gate, const int32_t *seq_lens,
                 const int32_t *idx, const float *out_lt, const float *out_st, const float *lse, const float *dout, float *dq,
                 float *dk, float *dv, float *dgate, const Workspace &ws, cudaStream_t st) {
  const bool plain = s.causal && s.stis_mode == 0;
  auto kq = plain ? dq_f32_kernel<D, true> : dq_f32_kernel<D, false>;
  auto kk = plain ? dkdv_f32_kernel<D, true> : dkdv_f32_kernel<D, false>;
  const int ntile = (s.L + 15) / 16;
  const int64_t tq = (int64_t)s.B * s.H * ntile, tk = (int64_t)s.B * s.Hkv * ntile;
  const int wq = chunk_split(tq), wk = chunk_split(tk);
  constexpr int T = Geo<D>::kTile;
  const size_t sq = (size_t)kCtaWarps * (6 * T + 16 * kPP) * sizeof(float);
  const size_t sk = (size_t)kCtaWarps * (2 * T + 2 * (2 * T + 64) + 2 * 16 * kPP) * sizeof(float);
  if (!allow_smem(kq, sq) || !allow_smem(kk, sk)) return BLOSSOM_ERR_CUDA;
  {
    LaunchScope ls(K_BWD_DQ_SIMT, st);
    if (launch_chained(kq, dim3(ctas(tq, wq)), dim3(32 * kCtaWarps), sq, st, s, q, k, v, gate, seq_lens, idx, out_lt, out_st, lse,
                       dout, dq, ws.qstats, ws.dalpha, wq) != cudaSuccess)
      return BLOSSOM_ERR_CUDA;
  }
  LaunchScope ls(K_BWD_DKDV_SIMT, st);
  return launch_chained(kk, dim3(ctas(tk, wk) + 1), dim3(32 * kCtaWarps), sk, st, s, q, k, v, gate, seq_lens, idx,
                        (const float4 *)ws.qstats, dout, dk, dv, (const double *)ws.dalpha, dgate, wk) == cudaSuccess
             ? BLOSSOM_OK
             : BLOSSOM_ERR_CUDA;
}

}  // namespace

bool supported(const Shape &s, int dtype) {
  return dtype == BLOSSOM_DTYPE_FP32 && s.Bk >= 16 && !s.pq && !s.gate_mode;
}

int launch_fwd(const Shape &s, const void *q, const void *k, const void *v, const float *gate, const int32_t *seq_lens,
               const int32_t *idx, void *out, void *out_lt, void *out_st, float *lse, cudaStream_t st) {
  typedef const float *F;
  auto f = s.D == 32 ? launch_fwd_t<32> : launch_fwd_t<64>;
  return f(s, (F)q, (F)k, (F)v, gate, seq_lens, idx, (float *)out, (float *)out_lt, (float *)out_st, lse, st);
}
int launch_bwd(const Shape &s, const void *q, const void *k, const void *v, const float *gate, const int32_t *seq_lens,
               const int32_t *idx, const void *out_lt, const void *out_st, const float *lse, const void *dout, void *dq,
               void *dk, void *dv, float *dgate, const Workspace &ws, cudaStream_t st) {
  typedef const float *F;
  auto f = s.D == 32 ? launch_bwd_t<32> : launch_bwd_t<64>;
  return f(s, (F)q, (F)k, (F)v, gate, seq_lens, idx, (F)out_lt, (F)out_st, lse, (F)dout, (float *)dq, (float *)dk, (float *)dv,
           dgate, ws, st);
}

}  // namespace f32
}  // namespace blossom
