// Backward for short histories (bf16): Delta, dQ, dK, dV, d alpha and the gate gradient in ONE kernel.
//
// As in the forward (attn_short_fwd.cu) the fixed costs of a launch and of a CTA bound these batches,
// not their arithmetic: pre-pass, dQ, dK/dV and gate-gradient kernels took 8-35 us each at a memory
// floor of 1-3 us.  Two kinds of CTA of 128 threads share the grid, so that one kind fills the gaps
// of the other:
//   key CTAs    64 keys of a (batch, key/value head), one warp per 16 keys with dK, dV in registers:
//               for every head of the group the queries' Q, dO rows and their records come into shared
//               memory, then a warp walks the 16-query chunks that selected its block or whose window
//               reaches it: S^T = K Q^T, dP^T = V dO^T, dV += W^T dO, dK += dS^T Q;
//   query CTAs  some 16-row tiles of a (batch, head): K, V rows in shared memory, a warp per tile,
//               dQ += dS K; they also produce d alpha from the fp32 probabilities, and the last of
//               them to finish adds the partial sums in a fixed order into dgate.
// With grouped heads and few (batch, key/value head) pairs a cluster of CTAs shares a key tile, each with its part of
// the heads, and adds dK and dV over the cluster (head_split).
// Key CTAs come first in the grid, those of the early keys (the most visitors) before the others.
// Both kinds recompute Delta = rowsum(dO o O_x) of the rows they need: 3 more row reads out of L2
// instead of a launch.  No gradient is written by more than one warp: no atomics on results.
#include <cooperative_groups.h>

#include "short_common.cuh"

namespace blossom {
namespace sh {
namespace {

struct BwdGeom {
  int nkey_ctas, nkt;  // key CTAs of the grid; tiles of 64 keys per (batch, key/value head)
  int split, heads;    // CTAs of a cluster that share a key tile's heads (1: no clusters); heads of each
  int per, nq;         // tiles per query CTA; query CTAs per (batch, head)
  int o_b, o_rec, o_stage, o_sel;  // byte offsets in shared memory
};


// (The branches are told apart by warp-uniform tests, not by instantiations: a warp runs through this
// code a few times, and the instructions it has to fetch first are a good part of a CTA's time.)
// A thread's 8 (key row, query column) pairs: W^T and dS^T.  rc: the records of its columns.
__device__ __forceinline__ void key_pairs(bool inL, bool inS, const float (&z)[2][4], const float (&dp)[2][4],
                                          const uint32_t (&bL)[2], const uint32_t (&bS)[2], float sc2, const float4 *rc,
                                          float (&w)[2][4], float (&d)[2][4]) {
#pragma unroll
  for (int e = 0; e < 8; ++e) w[e >> 2][e & 3] = d[e >> 2][e & 3] = 0.f;
#pragma unroll
  for (int br = 0; br < 2; ++br)
    if (br ? inS : inL) {
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int nt = x >> 1, j = x & 1, c = nt * 8 + j;
        const float2 r = *reinterpret_cast<const float2 *>(reinterpret_cast<const float *>(rc + c) + 2 * br);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint32_t b = br ? bS[i] : bL[i];
          const float y = ((b >> c) & 1u) ? exp2f(fmaf(z[nt][2 * i + j], sc2, r.x)) : 0.f;
          w[nt][2 * i + j] += y;
          d[nt][2 * i + j] = fmaf(y, dp[nt][2 * i + j] + r.y, d[nt][2 * i + j]);
        }
      }
    }
}
// A thread's 8 (query row, key column) pairs: dS and d alpha = sum (P_lt - P_st) dP.  nl = -lse (log2 units)
// and nD = -weight Delta: {long-term rows gid, gid + 8, short-term rows gid, gid + 8}.  The probabilities are
// unweighted and subtracted pair by pair, so that pairs which both branches see alike (the same keys, hence the
// same bits of lse) add exactly nothing: as two sums, subtracted at the end, histories shorter than the window
// left their rounding in the place of a zero.  (The weights ride in an addition; a chunk of the short-term branch
// alone takes eight subtractions more: forward + backward at B 256, L 200 71.2 -> 70.8 us, with eight heads on
// two, overlapping blocks and the power-law mask at B 128 140.9 -> 142.8.)
__device__ __forceinline__ void query_pairs(bool inL, bool inS, const float (&z)[2][4], const float (&dp)[2][4],
                                            const uint32_t (&bL)[2], const uint32_t (&bS)[2], float sc2, float alpha,
                                            float beta, const float (&nl)[4], const float (&nD)[4], float &dal,
                                            float (&d)[2][4]) {
  float diff[2][4];
#pragma unroll
  for (int e = 0; e < 8; ++e) d[e >> 2][e & 3] = diff[e >> 2][e & 3] = 0.f;
#pragma unroll
  for (int br = 0; br < 2; ++br)
    if (br ? inS : inL) {
      const float weight = br ? beta : alpha;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int i = (e >> 1) & 1, c = (e >> 2) * 8 + (e & 1);
        const uint32_t b = br ? bS[i] : bL[i];
        const float y = ((b >> c) & 1u) ? exp2f(fmaf(z[e >> 2][e & 3], sc2, nl[2 * br + i])) : 0.f;
        diff[e >> 2][e & 3] = br ? diff[e >> 2][e & 3] - y : y;
        d[e >> 2][e & 3] = fmaf(y, fmaf(weight, dp[e >> 2][e & 3], nD[2 * br + i]), d[e >> 2][e & 3]);
      }
    }
#pragma unroll
  for (int e = 0; e < 8; ++e) dal = fmaf(diff[e >> 2][e & 3], dp[e >> 2][e & 3], dal);
}

template <int D, bool PLAIN, bool SPLIT>
__global__ void __launch_bounds__(128, D == 32 ? 5 : 3) bwd_short_kernel(
    Shape s, BwdGeom bg, const __nv_bfloat16 *__restrict__ q, const __nv_bfloat16 *__restrict__ k,
    const __nv_bfloat16 *__restrict__ v, const float *__restrict__ gate, const int32_t *__restrict__ seq_lens,
    const int32_t *__restrict__ idx, const __nv_bfloat16 *__restrict__ out_lt, const __nv_bfloat16 *__restrict__ out_st,
    const float *__restrict__ lse, const __nv_bfloat16 *__restrict__ dout, __nv_bfloat16 *__restrict__ dq,
    __nv_bfloat16 *__restrict__ dk, __nv_bfloat16 *__restrict__ dv, float *__restrict__ dgate,
    double *__restrict__ part, int32_t *__restrict__ counter) {
  grid_chain_enter();
  constexpr int kThreads = 128, kWarps = 4;
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ double red[kThreads];
  __shared__ int last;
  uint8_t *ta = smem, *tb = smem + bg.o_b;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, gid = lane >> 2, tig = lane & 3;
  uint8_t *stage = smem + bg.o_stage + warp * 16 * D * 2;
  uint32_t *sel = reinterpret_cast<uint32_t *>(smem + bg.o_sel);
  const bool causal = PLAIN || s.causal;
  const float sc2 = s.scale * kLog2e;
  const int64_t BHL = (int64_t)s.B * s.H * s.L;
  const int bsh = __ffs(s.Bk) - 1;
  const uint32_t ta_a = smem_addr(ta), tb_a = smem_addr(tb), ont = lane_off_nt<D>(lane), onn = lane_off_nn<D>(lane);
  const int nU = s.B * s.Hkv;

  // which blocks every query block selected
  auto load_sel = [&](int uk, int b_lo, int b_hi) {
    for (int b = b_lo + warp; b < b_hi; b += kWarps) {
      const int32_t *row = idx + ((int64_t)uk * s.M + b) * s.topk;
      uint32_t m = 0u;
      for (int i = lane; i < s.topk; i += 32) {
        const int j = row[i];
        if (j >= 0 && j < s.M && (j <= b || !causal)) m |= 1u << j;
      }
      m = __reduce_or_sync(0xffffffffu, m);
      if (lane == 0) sel[b] = m;
    }
  };

  if ((int)blockIdx.x < bg.nkey_ctas) {
    // ============================================================ key CTA: dK, dV of 64 keys
    float4 *rec = reinterpret_cast<float4 *>(smem + bg.o_rec);  // {nl_lt, -Delta_lt, nl_st, -Delta_st} per query
    const int rank = SPLIT ? (int)blockIdx.x % bg.split : 0, kc = SPLIT ? (int)blockIdx.x / bg.split : (int)blockIdx.x;
    const int kt = kc / nU, uk = kc % nU, n = uk / s.Hkv, hk = uk % s.Hkv;
    int len = seq_lens ? seq_lens[n] : s.L;
    len = min(max(len, 0), s.L);
    const int pad0 = s.L - len;
    const int p0 = kt * 64 + warp * 16, p_last = min(p0 + 15, s.L - 1);
    const bool warp_live = p0 < s.L && p_last >= pad0, cta_live = min(kt * 64 + 63, s.L - 1) >= pad0;
    const int q_lo = causal ? max(kt * 64, pad0 & ~15) : pad0 & ~15, q_hi = (s.L + 15) & ~15;
    const int64_t koff = row_offset_kv(s, n, hk, 0);
    float ak[D / 8][4], av[D / 8][4];
#pragma unroll
    for (int e = 0; e < D / 8; ++e)
#pragma unroll
      for (int i = 0; i < 4; ++i) ak[e][i] = av[e][i] = 0.f;
    if (cta_live) {
      load_sel(uk, q_lo >> bsh, s.M);
      uint32_t ka[D / 16][4], va[D / 16][4];
      load_a_rows<D>(k + koff, s.ksl, p0, pad0, s.L, lane, ka);
      load_a_rows<D>(v + koff, s.ksl, p0, pad0, s.L, lane, va);
      uint64_t setL = 0ull, setS = 0ull;
      for (int hg = 0; hg < (SPLIT ? bg.heads : s.G); ++hg) {
        const int h = hk * s.G + (SPLIT ? rank * bg.heads : 0) + hg;
        const int64_t off = row_offset(s, n, h, 0);
        if (hg) __syncthreads();  // the previous head's rows are no longer read
        stage_rows<D>(ta, q + off, s.sl, q_lo, q_hi, pad0, s.L, tid, kThreads);
        cp_async_commit();
        const float alpha = head_alpha(gate, h), la = log2f(alpha), lb = log2f(1.f - alpha);
        constexpr int LPR = D / 8;
        for (int base = 0; base < (q_hi - q_lo) * LPR; base += kThreads) {
          const int i = base + tid, r = i / LPR, ch = i % LPR, t = q_lo + r;
          const bool in = t < q_hi, ok = t >= pad0 && t < s.L;
          uint4 gv = make_uint4(0u, 0u, 0u, 0u), lv = gv, sv = gv;
          if (ok) {
            const int64_t o = off + (int64_t)t * s.sl + ch * 8;
            gv = *reinterpret_cast<const uint4 *>(dout + o);
            lv = *reinterpret_cast<const uint4 *>(out_lt + o);
            sv = *reinterpret_cast<const uint4 *>(out_st + o);
          }
          const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w}, lw[4] = {lv.x, lv.y, lv.z, lv.w}, sw[4] = {sv.x, sv.y, sv.z, sv.w};
          float dL = 0.f, dS = 0.f;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            dL = fmaf(lo_bf(gw[e]), lo_bf(lw[e]), dL);
            dL = fmaf(hi_bf(gw[e]), hi_bf(lw[e]), dL);
            dS = fmaf(lo_bf(gw[e]), lo_bf(sw[e]), dS);
            dS = fmaf(hi_bf(gw[e]), hi_bf(sw[e]), dS);
          }
#pragma unroll
          for (int o = LPR / 2; o > 0; o >>= 1) {
            dL += __shfl_xor_sync(0xffffffffu, dL, o);
            dS += __shfl_xor_sync(0xffffffffu, dS, o);
          }
          if (in) {
            *reinterpret_cast<uint4 *>(tb + tile_off<D>(r, ch)) = gv;
            if (ch == 0) {
              const int64_t row = ((int64_t)n * s.H + h) * s.L + t;
              rec[r] = ok ? make_float4(la - lse[row] * kLog2e, -dL, lb - lse[BHL + row] * kLog2e, -dS)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
            }
          }
        }
        cp_async_wait<0>();
        __syncthreads();
        if (!warp_live) continue;
        if (hg == 0) {  // the query chunks that visit this warp's keys: lane = chunk
          bool fl[2], fs[2];
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const int t = (lane + 32 * x) * 16, t_last = min(t + 15, s.L - 1);
            const bool in = t >= q_lo && t < s.L && (!causal || t_last >= p0);
            fl[x] = in && ((sel[min(t >> bsh, s.M - 1)] >> (p0 >> bsh)) & 1u);
            fs[x] = in && st_ranges_touch(s, t, t_last, max(p0, pad0), p_last);
          }
          setL = ballot64(fl[0], fl[1]);
          setS = ballot64(fs[0], fs[1]);
        }
#pragma unroll 1
        for (uint64_t todo = setL | setS; todo; todo &= todo - 1) {
          const int c = __ffsll((long long)todo) - 1, t0 = c * 16;
          const bool inL = (setL >> c) & 1, inS = (setS >> c) & 1;
          float z[2][4], dp[2][4];
          const uint32_t co = (uint32_t)(t0 - q_lo) * (2 * D);
          product_nt<D>(ka, ta_a + co + ont, z);
          product_nt<D>(va, tb_a + co + ont, dp);
          const bool past = p0 >= pad0 && p0 + 15 < s.L && t0 >= pad0 && t0 + 15 < s.L && (!causal || t0 >= p0 + 15);
          uint32_t bL[2] = {0xffffu, 0xffffu}, bS[2] = {0xffffu, 0xffffu};  // pairs that take part: bits 0, 1, 8, 9
          if (!past)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const int p = p0 + gid + 8 * i;
              bL[i] = bS[i] = p >= pad0 && p < s.L ? cols16((causal ? p : pad0) - t0, s.L - 1 - t0) >> (2 * tig) : 0u;
            }
          if (inS && !(past && t0 + 15 - p0 < s.window && (causal || p0 + 15 - t0 < s.window)))
#pragma unroll
            for (int i = 0; i < 2; ++i) bS[i] &= st_queries16<PLAIN>(s, p0 + gid + 8 * i, t0, causal) >> (2 * tig);
          float w[2][4], d[2][4];
          const float4 *rc = rec + (t0 - q_lo) + 2 * tig;
          key_pairs(inL, inS, z, dp, bL, bS, sc2, rc, w, d);
          uint32_t pa[4];
          to_a(w, pa);
          product_nn<D>(pa, tb_a + co + onn, av);
          to_a(d, pa);
          product_nn<D>(pa, ta_a + co + onn, ak);
        }
      }
    }
    if (SPLIT) {  // rank 0 adds dV over the cluster and writes it, rank 1 dK; in rank order
      if (cta_live) {    // (the same for all of a cluster)
        namespace cg = cooperative_groups;
        cg::cluster_group cluster = cg::this_cluster();
        float4 *own = reinterpret_cast<float4 *>(smem) + tid;
        __syncthreads();  // the last head's rows are no longer read
#pragma unroll
        for (int e = 0; e < D / 8; ++e) {
          own[e * kThreads] = make_float4(av[e][0], av[e][1], av[e][2], av[e][3]);
          own[(D / 8 + e) * kThreads] = make_float4(ak[e][0], ak[e][1], ak[e][2], ak[e][3]);
        }
        cluster.sync();
        if (rank < 2) {
#pragma unroll
          for (int e = 0; e < D / 8; ++e)
#pragma unroll
            for (int i = 0; i < 4; ++i) av[e][i] = 0.f;
#pragma unroll 1
          for (int r = 0; r < bg.split; ++r) {
            const float4 *o = cluster.map_shared_rank(own, r) + rank * (D / 8) * kThreads;
#pragma unroll
            for (int e = 0; e < D / 8; ++e) {
              const float4 x = o[e * kThreads];
              av[e][0] += x.x;
              av[e][1] += x.y;
              av[e][2] += x.z;
              av[e][3] += x.w;
            }
          }
        }
        cluster.sync();  // nobody leaves while its sums are being read
      }
      if (rank < 2 && p0 < s.L) {
        const float f = rank ? s.scale : 1.f;
        store_rows<D>((rank ? dk : dv) + koff, s.ksl, p0, s.L, av, f, f, stage, lane);
      }
      return;
    }
    if (p0 < s.L) {
      store_rows<D>(dv + koff, s.ksl, p0, s.L, av, 1.f, 1.f, stage, lane);
      store_rows<D>(dk + koff, s.ksl, p0, s.L, ak, s.scale, s.scale, stage, lane);
    }
    return;
  }

  // ============================================================ query CTA: dQ, d alpha of some tiles
  // the last positions' CTAs first: they have the most keys, and the early ones may be all padding
  const int nQ = s.B * s.H, x = (int)blockIdx.x - bg.nkey_ctas, u = x % nQ, sp = bg.nq - 1 - x / nQ, n = u / s.H, h = u % s.H, hk = h / s.G;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len;
  const int ntiles = (s.L + 15) >> 4, tile0 = sp * bg.per, tile1 = min(ntiles, tile0 + bg.per);
  const int q1 = min(s.L, tile1 * 16), p_lo = pad0 & ~15, p_hi = causal ? q1 : s.L;
  const int64_t off = row_offset(s, n, h, 0), koff = row_offset_kv(s, n, hk, 0);
  const float alpha = head_alpha(gate, h), beta = 1.f - alpha;
  if (q1 > pad0) {
    const int hi16 = (p_hi + 15) & ~15;
    stage_rows<D>(ta, k + koff, s.ksl, p_lo, hi16, pad0, p_hi, tid, kThreads);
    stage_rows<D>(tb, v + koff, s.ksl, p_lo, hi16, pad0, p_hi, tid, kThreads);
    cp_async_commit();
    load_sel(n * s.Hkv + hk, (tile0 * 16) >> bsh, ((tile1 * 16 - 1) >> bsh) + 1 < s.M ? ((tile1 * 16 - 1) >> bsh) + 1 : s.M);
    cp_async_wait<0>();
  }
  __syncthreads();
  double dal = 0.0;
  for (int tile = tile0 + warp; tile < tile1; tile += kWarps) {
    const int t0 = tile * 16, t_last = min(t0 + 15, s.L - 1);
    float acc[D / 8][4];
#pragma unroll
    for (int e = 0; e < D / 8; ++e)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[e][i] = 0.f;
    if (t_last >= pad0) {
      uint32_t qa[D / 16][4], ga[D / 16][4];
      load_a_rows<D>(q + off, s.sl, t0, pad0, s.L, lane, qa);
      load_a_rows<D>(dout + off, s.sl, t0, pad0, s.L, lane, ga);
      float nD[4] = {0.f, 0.f, 0.f, 0.f}, nl[4];  // {long-term rows gid, gid + 8, short-term rows ...}
#pragma unroll
      for (int br = 0; br < 2; ++br) {
        uint32_t oa[D / 16][4];
        load_a_rows<D>((br ? out_st : out_lt) + off, s.sl, t0, pad0, s.L, lane, oa);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            nD[2 * br + (e & 1)] = fmaf(lo_bf(ga[kk][e]), lo_bf(oa[kk][e]), nD[2 * br + (e & 1)]);
            nD[2 * br + (e & 1)] = fmaf(hi_bf(ga[kk][e]), hi_bf(oa[kk][e]), nD[2 * br + (e & 1)]);
          }
      }
      const int r0 = t0 + gid;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        nD[i] = -(i < 2 ? alpha : beta) * quad_sum(nD[i]);
        const int t = r0 + 8 * (i & 1);
        nl[i] = t >= pad0 && t < s.L ? -(lse[(i < 2 ? 0 : BHL) + (int64_t)u * s.L + t] * kLog2e) : 0.f;
      }
      const uint32_t sb = sel[t0 >> bsh];
      uint64_t setL, setS;
      {  // the key chunks this tile visits: lane = chunk
        bool fl[2], fs[2];
#pragma unroll
        for (int y = 0; y < 2; ++y) {
          const int p = (lane + 32 * y) * 16;
          const bool in = p + 15 >= pad0 && p < s.L && (!causal || p <= t_last);
          fl[y] = in && ((sb >> min(p >> bsh, 31)) & 1u);
          fs[y] = in && st_ranges_touch(s, max(t0, pad0), t_last, p, min(p + 15, s.L - 1));
        }
        setL = ballot64(fl[0], fl[1]);
        setS = ballot64(fs[0], fs[1]);
      }
      const bool rows_in = t0 >= pad0 && t0 + 15 < s.L;
      float dal_t = 0.f;
#pragma unroll 1
      for (uint64_t todo = setL | setS; todo; todo &= todo - 1) {
        const int c = __ffsll((long long)todo) - 1, p0 = c * 16;
        const bool inL = (setL >> c) & 1, inS = (setS >> c) & 1;
        float z[2][4], dp[2][4], d[2][4];
        const uint32_t co = (uint32_t)(p0 - p_lo) * (2 * D);
        product_nt<D>(qa, ta_a + co + ont, z);
        product_nt<D>(ga, tb_a + co + ont, dp);
        const bool past = rows_in && p0 >= pad0 && (causal ? p0 + 15 <= t0 : p0 + 15 < s.L);
        uint32_t bL[2] = {0xffffu, 0xffffu}, bS[2] = {0xffffu, 0xffffu};  // pairs that take part: bits 0, 1, 8, 9
        if (!past)
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int t = r0 + 8 * i;
            bL[i] = bS[i] = t >= pad0 && t < s.L ? cols16(pad0 - p0, (causal ? t : s.L - 1) - p0) >> (2 * tig) : 0u;
          }
        if (inS && !(past && t0 + 15 - p0 < s.window && (causal || p0 + 15 - t0 < s.window)))
#pragma unroll
          for (int i = 0; i < 2; ++i) bS[i] &= st_keys16<PLAIN>(s, r0 + 8 * i, p0, causal) >> (2 * tig);
        query_pairs(inL, inS, z, dp, bL, bS, sc2, alpha, beta, nl, nD, dal_t, d);
        uint32_t pa[4];
        to_a(d, pa);
        product_nn<D>(pa, ta_a + co + onn, acc);
      }
      dal += (double)dal_t;
    }
    store_rows<D>(dq + off, s.sl, t0, s.L, acc, s.scale, s.scale, stage, lane);
  }
  // partial of d alpha of this CTA, then the gate gradient by the last query CTA to arrive
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dal += __shfl_xor_sync(0xffffffffu, dal, o);
  if (lane == 0) red[warp] = dal;
  __syncthreads();
  if (tid == 0) {
    part[u * bg.nq + sp] = (red[0] + red[1]) + (red[2] + red[3]);
    __threadfence();
    const int total = s.B * s.H * bg.nq;
    last = atomicAdd(counter, 1) == total - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (tid == 0) *counter = 0;  // (a repeated backward on this workspace starts from zero again)
  // A warp per head, its lanes in ascending order and a fixed tree: this tail is a chain of latencies.
  const int per_head = s.B * bg.nq;
  for (int hh = warp; hh < s.H; hh += kWarps) {
    double a = 0.0;
#pragma unroll 8
    for (int i = lane; i < per_head; i += 32) a += __ldcg(part + ((int64_t)(i / bg.nq) * s.H + hh) * bg.nq + i % bg.nq);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) {
      const double al = 1.0 / (1.0 + exp(-((double)gate[hh * 2 + 0] - (double)gate[hh * 2 + 1])));
      const double g0 = al * (1.0 - al) * a;
      dgate[hh * 2 + 0] = (float)g0;
      dgate[hh * 2 + 1] = (float)(-g0);
    }
  }
}

}  // namespace

// Which calls take this kernel.  Measured against pre-pass + dQ + dK/dV + gate gradient (us, without the
// 10 - 15 us of tile lists that those need after a short forward; 4 heads):
//              B 4              B 32             B 256
//   D 32  L 100    12 / 23        14 / 22          54 / 75
//         L 300    18 / 27        33 / 40         207 / 196
//         L 400    23 / 28        63 / 49         479 / 275
//   D 64  L 100    10 / 19        21 / 23          95 / 79
//         L 180    18 / 24        30 / 29         195 / 138
//         L 300    24 / 29        60 / 43         497 / 232
bool bwd_short_supported(const Shape &s, int dtype) {
  if (!fwd_short_supported(s, dtype, true)) return false;
  const int64_t rows = (int64_t)s.B * s.H * s.L;  // (beyond L D = 25000 one CTA fills an SM)
  return s.L <= (s.D == 32 ? 300 : 128) || rows <= (s.L * s.D <= 25000 ? 32768 : 8192);
}

// CTAs of a cluster that share the heads of a key tile.  A key CTA with all heads of a group is a chain (stage, wait,
// walk, a head after the other) that sets the time of a small batch: with four heads on one at L 200, D 32 the backward
// took 46 us at B 4 and 54 at B 16, against 83 at B 128; split, forward + backward 68 -> 41, 84 -> 49 (B 32: 88 -> 64).
// The chip full, the copies of the fixed part (selection, K and V rows, the sums over the cluster) cost 3 - 17 %: B 128
// 141 -> 146 with two CTAs and 163 with four.  The lines, from 178 shapes (two to eight heads a group, L 50 - 300,
// B 2 - 256): as many CTAs as divide the heads while (batch, key/value head) pairs x CTAs stay below them.
int head_split(const Shape &s) {
  const int64_t units = (int64_t)s.B * s.Hkv;
  for (int split = 8; split > 1; split /= 2) {
    const int line = split == s.G ? (s.D == 32 ? 256 : 192) : (s.D == 32 ? 384 : 256);
    if (s.G % split == 0 && units * split <= line) return split;
  }
  return 1;
}

template <int D>
static int launch_t(const Shape &s, const void *q, const void *k, const void *v, const float *gate, const int32_t *seq_lens,
                    const int32_t *idx, const void *out_lt, const void *out_st, const float *lse, const void *dout, void *dq,
                    void *dk, void *dv, float *dgate, const Workspace &ws, cudaStream_t st) {
  typedef __nv_bfloat16 bf;
  BwdGeom bg;
  const int ntiles = (s.L + 15) / 16, rows = ntiles * 16;
  bg.nkt = (s.L + 63) / 64;
  bg.split = head_split(s);
  bg.heads = s.G / bg.split;
  bg.nkey_ctas = s.B * s.Hkv * bg.nkt * bg.split;
  bg.per = s.B * s.H >= 296 ? 8 : 4;
  bg.nq = (ntiles + bg.per - 1) / bg.per;
  bg.per = (ntiles + bg.nq - 1) / bg.nq;  // of equal size
  bg.o_b = rows * D * 2;
  bg.o_rec = 2 * rows * D * 2;
  bg.o_stage = bg.o_rec + rows * 16;
  const int sums = 2 * (D / 8) * 128 * 16;  // a CTA's dV and dK, over the tiles
  if (bg.split > 1 && bg.o_stage < sums) bg.o_stage = sums;
  bg.o_sel = bg.o_stage + 4 * 16 * D * 2;
  const int smem = bg.o_sel + 128;
  const bool plain = s.causal && s.stis_mode == 0;
  auto kern = bg.split > 1 ? (plain ? bwd_short_kernel<D, true, true> : bwd_short_kernel<D, false, true>)
                           : (plain ? bwd_short_kernel<D, true, false> : bwd_short_kernel<D, false, false>);
  if (!allow_smem(kern, (size_t)smem)) return BLOSSOM_ERR_CUDA;
  LaunchScope ls(K_BWD_SHORT, st);
  const dim3 grid((unsigned)(bg.nkey_ctas + s.B * s.H * bg.nq));
  auto launch = [&](auto... args) {
    return bg.split > 1 ? launch_chained_cluster(kern, grid, dim3(128), (size_t)smem, (unsigned)bg.split, st, args...)
                        : launch_chained(kern, grid, dim3(128), (size_t)smem, st, args...);
  };
  if (launch(s, bg, (const bf *)q, (const bf *)k, (const bf *)v, gate, seq_lens, idx, (const bf *)out_lt, (const bf *)out_st,
             lse, (const bf *)dout, (bf *)dq, (bf *)dk, (bf *)dv, dgate, ws.dalpha, ws.status + kCounterWord) != cudaSuccess)
    return BLOSSOM_ERR_CUDA;
  return BLOSSOM_OK;
}

int launch_bwd_short(const Shape &s, const void *q, const void *k, const void *v, const float *gate,
                     const int32_t *seq_lens, const int32_t *idx, const void *out_lt, const void *out_st, const float *lse,
                     const void *dout, void *dq, void *dk, void *dv, float *dgate, const Workspace &ws, cudaStream_t st) {
  if (s.D == 32)
    return launch_t<32>(s, q, k, v, gate, seq_lens, idx, out_lt, out_st, lse, dout, dq, dk, dv, dgate, ws, st);
  return launch_t<64>(s, q, k, v, gate, seq_lens, idx, out_lt, out_st, lse, dout, dq, dk, dv, dgate, ws, st);
}

}  // namespace sh
}  // namespace blossom
