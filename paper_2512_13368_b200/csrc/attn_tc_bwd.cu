// Tensor-core backward of the fused two-branch attention (bf16 storage, fp32 accumulate): a small
// pre-pass and two main kernels, all deterministic (no atomics on any gradient); the main kernels
// recompute the probabilities from the saved log-sum-exps.
//
//  pre-pass  Delta_x = rowsum(dO o O_x) of both branches from coalesced reads, and the per-row
//            records the main kernels read: per pair of rows {nl_lt(2), -Delta_lt(2)}
//            {nl_st(2), -Delta_st(2)}, nl = -(lse*log2e - log2 weight): in the dK/dV kernel the branch
//            weights alpha, beta ride in the exponent, alpha P_lt = exp2(s*log2e + nl_lt); the dQ kernel
//            needs unweighted probabilities and takes the log-sum-exps themselves.
//
// Main kernels: CTA = 384 threads.  Warps 0..7 compute; warps 8, 9 stay converged and one elected lane
// of each issues the TMA loads and the MMAs (10 and 11 are spare); registers move from those warps to the
// compute warps (setmaxnreg).  A CTA owns a resident 128-row tile (rows = TMEM lanes) and streams pairs of
// half tiles of 32 rows past it (any two: tc_meta_kernel lists only those that are needed), each half with a buffer in
// tensor memory and four compute warps of its own: warps w and w + 4 both address TMEM lane quarter w % 4; the first
// takes the first half of every pair, the second the other, so the two halves never wait for each other.  The tile arithmetic runs in
// 16-column passes, two columns per FMA / ADD / MUL (packed f32x2); outputs are staged in shared
// memory and written with whole-line TMA stores.
//
// What the products of a half tile wait for is one thing, its second operand in tensor memory: the warp that
// issues them puts the first stage of the next half tile behind the second stage of this one, into the same
// buffer, without waiting in between (the order assumed in tc_common.cuh).  With eight
// warps on every half tile (16 columns each, twice the hand-offs and their instructions), a warp for each
// stage and without the uniform registers of tc_common.cuh the kernels took 197 and 232 us at B 128, H 4,
// L 1024, D 64 (without: 181 and 223), 384 and 479 at B 16, H 8, L 4096 (353 and 453), 64 and 80 with a selection
// per position at B 8, L 1500 (50 and 73).  After that the code: half tiles of one branch without masks are one code for
// either branch, everything else goes through one masked code; with a code for each branch, both, and masked tiles the
// instructions did not come fast enough (173 and 221 -> 166 and 212 us; 341 and 450 -> 331 and 435; D 32 82 and 98 -> 78
// and 93).  What is left is the chain of a half tile: arithmetic 1300 cycles, from there to the next logits 700, while
// the issue slots are 49 % (dQ) and 41 % (dK/dV) and the tensor pipe 39 % busy (B 4, H 8, L 4096); and the 8000 cycles that a
// CTA spends outside its loop.
//
//  dQ     resident Q, dO (128 queries: 128 positions of a head, or with grouped heads 64 positions
//         of two heads of a group, as in the forward); streams pairs of half tiles of K, V (same walk as the
//         forward), 32 keys each.  Tensor memory: a buffer of 64 columns for each half (S in its first 32 columns, dP in the other 32),
//         Q and dO as first operands of the first-stage products [128,128+D/2), [160,160+D/2)
//         (read from shared memory they cost 4 KB per product, more than the data pipe delivers
//         in the product's run time), and dQ [192,192+D).  S = Q K^T, dP = dO V^T; P_x = exp(S - lse_x);
//         dS = P_lt (alpha dP - alpha Delta_lt) + P_st (beta dP - beta Delta_st) (one tile for both
//         branches, they share K).  A thread writes the dS (bf16 pairs) of a pass's 16 columns over the first 8
//         of them in S, from where dQ += dS K reads it: the compute warps wait for one
//         thing per half tile (its S and dP).  d alpha = sum (P_lt - P_st) dP from the fp32 probabilities, subtracted pair by pair.
//  dK/dV  transposed: resident K, V of 128 keys, streams pairs of half tiles of Q, dO, 32 queries each (and
//         their row records, by bulk copy), that selected one of its key blocks or whose window reaches them.
//         Tensor memory: a buffer of 64 columns for each half (S^T in its first 32 columns, dP^T in the other
//         32), dV [128,128+D), dK [192,192+D).  S^T = K Q^T, dP^T = V dO^T; thread = key row and
//         32 query columns; it writes W^T = P'_lt + P'_st and dS^T (bf16 pairs) of a pass's 16 columns over
//         the first 8 of them in S^T / dP^T, from where dV += W^T dO and dK += dS^T Q read
//         their first operand: nothing of a tile's arithmetic goes through shared memory, whose
//         data pipe (operand reads of the products, row records) is the busiest unit of this
//         kernel.
// Every wait is bounded (tc_common.cuh).
#include "tc_common.cuh"

#include <cooperative_groups.h>
#include <type_traits>

namespace blossom {
namespace tc {
namespace cg = cooperative_groups;
namespace {

// warps 0..7 compute; 8 loader, 9 issuer of the products; 10, 11 spare
constexpr int kKvThreads = 384;
constexpr int kProducerRegs = 64, kKvComputeRegs = 88;  // 256 * 88 + 128 * 64 = 384 * 80 (measured: the issuing warps spill below 48)
constexpr int kComputeWarps = 8;
constexpr int kDqStages = 4;
constexpr int kKvStages = 4;
constexpr uint32_t kBwdTmemCols = 256;
constexpr int kStatBytes = 64 * 16;  // row records of a pair of half tiles of queries

__device__ __forceinline__ bool bit(uint32_t w, int c) { return (w >> c) & 1u; }

// ------------------------------------------------------------------ backward pre-pass
// Delta_x = rowsum(dO o O_x) of both branches and the per-row records of the backward kernels (of which the
// dQ kernel reads Delta, and nl where a pass has a weight of its own per row):
// per pair of rows {nl_lt(2), -Delta_lt(2)} {nl_st(2), -Delta_st(2)} with
// nl = -(lse * log2e - log2 weight), the branch weight (alpha, beta) riding in the exponent;
// zeros for padded rows and for the rows that pad L to a multiple of 64.
// D / 16 lanes share a row (two 16-byte loads per tensor each, half a row apart): fully coalesced reads.  Grid: units x
// runs of rows.  Bound by memory, and nearly by issue slots (with D / 8 lanes a row, a row's fixed instructions and
// shuffles on twice as many threads: 71 % of the slots; B 128, H 4, L 1024, D 64 45.5 -> 43.6 us, B 16, H 4, L 777 10.5 -> 8.7).
template <int D>
__host__ __device__ constexpr int prep_rows() { return 256 / (D / 16); }  // rows per block
template <int D>
__global__ void __launch_bounds__(256) bwd_prep_kernel(Shape s, const float *__restrict__ gate,
                                                       const int32_t *__restrict__ seq_lens,
                                                       const __nv_bfloat16 *__restrict__ out_lt,
                                                       const __nv_bfloat16 *__restrict__ out_st,
                                                       const float *__restrict__ lse,
                                                       const __nv_bfloat16 *__restrict__ dout,
                                                       float4 *__restrict__ qstats, int Lpad,
                                                       int32_t *__restrict__ status) {
  grid_chain_enter();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 4) status[threadIdx.x] = 0;  // the backward's status words
  constexpr int LPR = D / 16;  // lanes per row
  const int u = blockIdx.x, n = u / s.H, h = u - n * s.H;
  const int t = blockIdx.y * prep_rows<D>() + threadIdx.x / LPR, ch = threadIdx.x % LPR;
  const int len = min(max(seq_lens ? seq_lens[n] : s.L, 0), s.L);
  const bool row_valid = t < s.L && t >= s.L - len;
  float aL = 0.f, aS = 0.f, l0 = 0.f, l1 = 0.f;
  if (row_valid) {
    const int64_t off = row_offset(s, n, h, t) + ch * 8;
    uint4 gv[2], lv[2], sv[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      gv[i] = *reinterpret_cast<const uint4 *>(dout + off + i * (D / 2));
      lv[i] = *reinterpret_cast<const uint4 *>(out_lt + off + i * (D / 2));
      sv[i] = *reinterpret_cast<const uint4 *>(out_st + off + i * (D / 2));
    }
    if (ch == 0) {
      l0 = lse[(int64_t)u * s.L + t];
      l1 = lse[((int64_t)s.B * s.H + u) * s.L + t];
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t gw[4] = {gv[i].x, gv[i].y, gv[i].z, gv[i].w}, lw[4] = {lv[i].x, lv[i].y, lv[i].z, lv[i].w},
                     sw[4] = {sv[i].x, sv[i].y, sv[i].z, sv[i].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float g0 = __uint_as_float(gw[e] << 16), g1 = __uint_as_float(gw[e] & 0xffff0000u);
        aL = fmaf(g0, __uint_as_float(lw[e] << 16), aL);
        aL = fmaf(g1, __uint_as_float(lw[e] & 0xffff0000u), aL);
        aS = fmaf(g0, __uint_as_float(sw[e] << 16), aS);
        aS = fmaf(g1, __uint_as_float(sw[e] & 0xffff0000u), aS);
      }
    }
  }
#pragma unroll
  for (int o = LPR / 2; o > 0; o >>= 1) {  // fixed-shape tree over the row's lanes
    aL += __shfl_xor_sync(0xffffffffu, aL, o);
    aS += __shfl_xor_sync(0xffffffffu, aS, o);
  }
  if (ch == 0 && t < Lpad) {
    float r0 = 0.f, r2 = 0.f, r4 = 0.f, r6 = 0.f;
    if (row_valid) {
      const float alpha = gate_alpha(gate, h), beta = 1.f - alpha;
      r0 = -(l0 * kLog2e - log2f(alpha));
      r4 = -(l1 * kLog2e - log2f(beta));
      r2 = -aL;
      r6 = -aS;
    }
    float *rec = reinterpret_cast<float *>(qstats) + ((int64_t)u * Lpad + (t & ~1)) * 4 + (t & 1);
    rec[0] = r0;
    rec[2] = r2;
    rec[4] = r4;
    rec[6] = r6;
  }
}

// eight bf16 of a row += the eight at p (of the pass before), one rounding
__device__ __forceinline__ void add_row_chunk(uint32_t (&w)[4], const __nv_bfloat16 *p) {
  const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(p));
  const uint32_t x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    w[e] = pack_bf16(__uint_as_float(w[e] << 16) + __uint_as_float(x[e] << 16),
                     __uint_as_float(w[e] & 0xffff0000u) + __uint_as_float(x[e] & 0xffff0000u));
}

// ---------------------------------------------------------------------------- backward dQ
// 16 columns of one tile for one row: dS packed to bf16 pairs, and this row's part of d alpha = sum (P_lt -
// P_st) dP.  nlL / nlS = -lse (log2 units), wL / wS: the branches' weights, nDL / nDS = -weight Delta.  The
// unweighted probabilities are subtracted pair by pair, so that pairs which both branches see alike (the same
// keys, hence the same bits of lse) add exactly nothing; with the weights in the exponent and a sum per
// branch, subtracted at the end, rows whose window holds the whole history left their rounding instead of a
// zero.  (As many instructions: the weight rides in what was the addition of -Delta; the kernel went from
// 0.381 to 0.388 ms at B 16, H 8, L 4096.)  dalS collects what only the short-term branch sees.  Two columns
// per FMA / ADD / MUL instruction.
// BOTH: both branches see columns of the tile; else the one whose record, weight and mask come as the first ones
// (one code for either branch: the instructions of the variants have to be fetched, and that is felt).
template <bool BOTH, bool FULL>
__device__ __forceinline__ void dq_tile(const float (&sv)[16], const float (&dp)[16], uint32_t hL, uint32_t hS, float sc2,
                                        float nlL, float nlS, float wL, float wS, float nDL, float nDS, float2 &dal,
                                        uint32_t (&dw)[8]) {
  const float2 sc = make_float2(sc2, sc2);
#pragma unroll
  for (int c = 0; c < 16; c += 2) {
    const float2 s2 = make_float2(sv[c], sv[c + 1]), dp2 = make_float2(dp[c], dp[c + 1]);
    const float2 x = ffma2(s2, sc, make_float2(nlL, nlL));
    float2 pL = make_float2(exp2f(x.x), exp2f(x.y));
    if (!FULL) {
      pL.x = bit(hL, c) ? pL.x : 0.f;
      pL.y = bit(hL, c + 1) ? pL.y : 0.f;
    }
    float2 acc = fmul2(pL, ffma2(dp2, make_float2(wL, wL), make_float2(nDL, nDL)));
    if (BOTH) {
      const float2 y = ffma2(s2, sc, make_float2(nlS, nlS));
      float2 p = make_float2(exp2f(y.x), exp2f(y.y));
      if (!FULL) {
        p.x = bit(hS, c) ? p.x : 0.f;
        p.y = bit(hS, c + 1) ? p.y : 0.f;
      }
      dal = ffma2(ffma2(p, make_float2(-1.f, -1.f), pL), dp2, dal);
      acc = ffma2(p, ffma2(dp2, make_float2(wS, wS), make_float2(nDS, nDS)), acc);
    } else {
      dal = ffma2(pL, dp2, dal);
    }
    dw[c >> 1] = pack_bf16(acc.x, acc.y);
  }
}

// MODE of both kernels below.  kPlain: the causal mask, one selection per query block and both branches: the
// other modes' tests fold away at compile time, and a masked tile is taken for both branches at once (tiles
// with the masks of one branch only are rare there, and the code for them cost 2 %; in the other modes
// it saves 5 - 12 %: selection per position, L 1500: dQ 63 -> 55 us, dK/dV 76 -> 72 us; a pass for one
// branch of a gate that depends on the input: 27 -> 25 us).  kPass: a pass for one branch, the second of
// which adds to what the first has written.
constexpr int kGeneral = 0, kPlain = 1, kPass = 2;
// PACK (dQ kernel): rows 0..63 and 64..127 of the CTA are the same 64 positions of two query heads
// with a common key/value head, as in the forward kernel.
template <int D, int MODE, bool PACK>
__global__ void __launch_bounds__(kKvThreads, 2) bwd_dq_tc_kernel(
    const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
    const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmg, Shape s,
    const float *__restrict__ gate, const int32_t *__restrict__ seq_lens, const float *__restrict__ lse,
    const uint8_t *__restrict__ qmeta, const __grid_constant__ CUtensorMap tmdq,
    const __grid_constant__ CUtensorMap tmk32, const __grid_constant__ CUtensorMap tmv32,
    const float4 *__restrict__ qstats, double *__restrict__ dalpha_part, int32_t *__restrict__ status,
    int nT, const __nv_bfloat16 *add_dq) {
  constexpr bool PLAIN = MODE == kPlain, ADDS = MODE == kPass;
  grid_wait();
  grid_release();  // (the dK/dV kernel depends on nothing of this one)
  using C = Cfg<D>;
  constexpr int STAGES = kDqStages;
  constexpr int OC = D / 2;  // accumulator columns per thread
  extern __shared__ uint8_t smem_raw[];
  // barriers: full[STAGES], empty[STAGES], res, meta, a_ready, then one per buffer: s_full[2],
  // t_full[2]; all_done
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 8];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ double red[kComputeWarps];

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const int nST = (s.L + 127) >> 7;
  // long rows first, tile-major: every unit's last tile, then every unit's last but one, ...
  // (PACK: a unit is a pair of heads, a tile 64 positions; h = the pair's first head)
  const int nU = PACK ? s.B * (s.H / 2) : s.B * s.H, nQT = PACK ? nT : nST;
  const int st = nQT - 1 - (int)(blockIdx.x / nU);
  const int u = (int)(blockIdx.x % nU);
  const int n = PACK ? u / (s.H / 2) : u / s.H, h = PACK ? 2 * (u % (s.H / 2)) : u % s.H;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len;
  const int row0 = PACK ? st * 64 : st * 128;
  const int Lpad = nT * 64;

  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t *tiles = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint8_t *q_tile = tiles;
  uint8_t *g_tile = q_tile + C::kBigBytes;
  uint8_t *kv_tiles = g_tile + C::kBigBytes;
  uint8_t *meta = kv_tiles + STAGES * 2 * C::kSmallBytes;  // image built by tc_meta_kernel
  const bool causal = PLAIN || s.causal;
  const int pq = PLAIN ? 0 : s.pq;
  const MetaLayout ml = meta_layout(nT, pq);
  const uint8_t *selb = meta + ml.sel;
  const uint8_t *rowb = meta + ml.rows;  // (selection per query position) [128 rows][nT]
  const uint16_t *list = reinterpret_cast<const uint16_t *>(meta + ml.list);
  const uint8_t *lflags = meta + ml.flags;
  const uint8_t *jcls = meta + ml.jcls;  // [pair][half][compute warp]

  const uint32_t b_full = smem_u32(&bars[0]), b_empty = smem_u32(&bars[STAGES]);
  const uint32_t b_res = smem_u32(&bars[2 * STAGES]), b_meta = smem_u32(&bars[2 * STAGES + 1]);
  const uint32_t b_aready = smem_u32(&bars[2 * STAGES + 2]);
  const uint32_t b_sfull = smem_u32(&bars[2 * STAGES + 3]), b_tfull = smem_u32(&bars[2 * STAGES + 5]);
  const uint32_t b_all = smem_u32(&bars[2 * STAGES + 7]);

  // this thread's row (compute warps) and its record from the pre-pass: asked for here, used after the set-up
  const int quarter = warp & 3, half = warp >> 2;
  const int r = quarter * 32 + lane, t = PACK ? row0 + (r & 63) : row0 + r;
  const int hr = PACK ? h + (r >> 6) : h;  // this row's head
  const bool row_ok = t < s.L;
  float rec0 = 0.f, rec2 = 0.f, rec4 = 0.f, rec6 = 0.f;
  if (row_ok && warp < kComputeWarps) {
    const int64_t hrow = (int64_t)n * s.H + hr;
    const float *rec = reinterpret_cast<const float *>(qstats) + (hrow * Lpad + (t & ~1)) * 4 + (t & 1);
    rec0 = ADDS ? rec[0] : lse[hrow * s.L + t];
    rec2 = rec[2];
    rec4 = ADDS ? rec[4] : lse[((int64_t)s.B * s.H + hrow) * s.L + t];
    rec6 = rec[6];
  }
  // The set-up is shared out so that the first loads leave at once: nothing before them waits for memory.
  if (warp == kComputeWarps && lane == 0) {
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(b_full + 8 * i, 1);
      mbar_init(b_empty + 8 * i, 1);
    }
    mbar_init(b_res, 1);
    mbar_init(b_aready, kComputeWarps);
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_sfull + 8 * i, 1);
      mbar_init(b_tfull + 8 * i, kComputeWarps / 2);
    }
    mbar_init(b_meta, 1);
    mbar_init(b_all, 1);
    mbar_fence_init();
    // the CTA's tile lists (the streamed tiles wait for them) and its resident tiles
    mbar_expect_tx(b_meta, (uint32_t)ml.bwd);
    bulk_load(smem_u32(meta), qmeta + ((size_t)u * nQT + (nQT - 1 - st)) * ml.bytes, (uint32_t)ml.bwd, b_meta);
    mbar_expect_tx(b_res, 2 * C::kBigBytes);
    tma_load_4d(smem_u32(q_tile), &tmq, b_res, 0, row0, h, n);
    tma_load_4d(smem_u32(g_tile), &tmg, b_res, 0, row0, h, n);
    tma_prefetch_desc(&tmk);
    tma_prefetch_desc(&tmv);
  }
  if (warp == kComputeWarps + 1) {
    tmem_alloc(smem_u32(&tmem_slot), kBwdTmemCols);
    tmem_relinquish();
  }
  if (warp == kComputeWarps + 2 && lane == 0) abort_flag = (*status != 0) ? 1 : 0;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  mbar_wait(b_meta, 0, &abort_flag, 223);
  const int listed = *reinterpret_cast<const int *>(meta + ml.counts);
  const int nvis = uniform(*(volatile int *)&abort_flag ? 0 : listed);  // (the lists may not be there)
  const uint32_t tmem_base = (uint32_t)uniform((int)tmem_slot);
  // buffers at tmem_base + 64 * (half tile % 2); Q and dO as first operands (bf16 pairs, D / 2
  // columns each) at 128 and 160; the dQ accumulator at 192
  const uint32_t tmem_qa = tmem_base + 128, tmem_ga = tmem_base + 160, tmem_dq = tmem_base + 192;

  if (warp >= kComputeWarps) {
    // ============ two single-thread roles, one converged warp each ============
    setmaxnreg_dec<kProducerRegs>();
    if (warp == kComputeWarps && nvis > 0) {
      // ---- loader: Q, dO once; K/V tiles up to STAGES ahead of their consumers ----
      bool go = true;
      for (int j = 0; j < nvis; ++j) {
        const int sj = j % STAGES;
        if (j >= STAGES) go = mbar_wait(b_empty + 8 * sj, ((j - STAGES) / STAGES) & 1, &abort_flag, 205) && go;
        const uint32_t bar = b_full + 8 * sj;
        const uint32_t kt = smem_u32(kv_tiles + sj * 2 * C::kSmallBytes);
        const uint32_t pair = reinterpret_cast<const uint32_t *>(list)[j];
        const int row0 = (int)(pair & 0xffffu) * 32, row1 = (int)(pair >> 16) * 32, hk = h / s.G;  // the key/value head of this query head
        if (elect_one() && go) {
          mbar_expect_tx(bar, 2 * C::kSmallBytes);
          tma_load_halves(kt, C::kSmallBytes / 2, &tmk, &tmk32, bar, row0, row1, hk, n);
          tma_load_halves(kt + C::kSmallBytes, C::kSmallBytes / 2, &tmv, &tmv32, bar, row0, row1, hk, n);
        }
        __syncwarp();
      }
    } else if (warp == kComputeWarps + 1 && nvis > 0) {
      // ---- S = Q K^T and dP = dO V^T of a half tile (32 keys) into buffer x % 2, then, once its dS is in
      // tensor memory, dQ += dS K (K MN-major) and behind it the first stage of half tile x + 2 into the same
      // buffer, without a wait for the second stage to have read it (the order assumed in tc_common.cuh).  Q and dO are read from tensor memory (the compute warps
      // copied the resident tiles there), so a product fetches only its 32 keys from shared memory instead
      // of 128 rows of Q or dO as well ----
      constexpr uint32_t idesc_s = instr_desc(128, 32, 0, 0), idesc_dq = instr_desc(128, D, 0, 1);
      auto first_stage = [&](int sj, int hh) {
        const uint32_t kt = smem_u32(kv_tiles + sj * 2 * C::kSmallBytes) + hh * 32 * C::kRowBytes;
        const uint64_t dkd = smem_desc(kt, 16, C::kAtomBytes, C::kSwizzle);
        const uint64_t dvd = smem_desc(kt + C::kSmallBytes, 16, C::kAtomBytes, C::kSwizzle);
        const uint32_t ts = tmem_base + 64 * hh;
#pragma unroll
        for (int k = 0; k < D / 16; ++k) umma_bf16_ts(ts, tmem_qa + 8 * k, dkd + 2 * k, idesc_s, k > 0);
#pragma unroll
        for (int k = 0; k < D / 16; ++k) umma_bf16_ts(ts + 32, tmem_ga + 8 * k, dvd + 2 * k, idesc_s, k > 0);
        umma_commit(b_sfull + 8 * hh);
      };
      mbar_wait(b_aready, 0, &abort_flag, 201);
      mbar_wait(b_full, 0, &abort_flag, 202);
      tc_fence_after();
      if (elect_one()) {
        first_stage(0, 0);
        first_stage(0, 1);
      }
      __syncwarp();
      for (int i = 0, sj = 0; i < nvis; ++i) {
        const int sn = sj + 1 == STAGES ? 0 : sj + 1;
        const bool more = i + 1 < nvis;
        const uint64_t dkm = smem_desc(smem_u32(kv_tiles + sj * 2 * C::kSmallBytes), C::kSmallBytes, C::kAtomBytes, C::kSwizzle);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          if (hh == 0 && more) mbar_wait(b_full + 8 * sn, ((i + 1) / STAGES) & 1, &abort_flag, 206);
          mbar_wait(b_tfull + 8 * hh, i & 1, &abort_flag, 204);
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              umma_bf16_ts(tmem_dq, tmem_base + 64 * hh + 16 * kk, dkm + (2 * hh + kk) * C::kKStep, idesc_dq,
                           (i | hh | kk) != 0);
            if (hh == 1) umma_commit(more ? b_empty + 8 * sj : b_all);  // every product on this stage has completed
            if (more) first_stage(sn, hh);
          }
          __syncwarp();
        }
        sj = sn;
      }
    }
  } else {
    setmaxnreg_inc<kKvComputeRegs>();
    const int g = r / s.Bk;
    const bool row_valid = row_ok && t >= pad0;
    const int t_last = row_valid ? (causal ? t : s.L - 1) : -1;  // the last key this row may see
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    // kPass: the row's weight rides in its record's exponents (the gate's gradient is not formed here)
    const float alpha = ADDS ? 1.f : gate_alpha(gate, hr), beta = ADDS ? 1.f : 1.f - alpha;
    // this row's record from the pre-pass: nl = -(lse * log2e - log2 weight), nD = -Delta
    float nlL = 0.f, nlS = 0.f, nDL = 0.f, nDS = 0.f;
    if (row_valid) {
      nlL = ADDS ? rec0 : -(rec0 * kLog2e);
      nDL = alpha * rec2;
      nlS = ADDS ? rec4 : -(rec4 * kLog2e);
      nDS = beta * rec6;
    }
    float2 dalL = make_float2(0.f, 0.f), dalS = make_float2(0.f, 0.f);  // see dq_tile
    const float sc2 = s.scale * kLog2e;
    if (nvis > 0) {
      // The resident tiles become first operands in tensor memory: row r of Q (warps 0..3) or of dO
      // (warps 4..7) goes to lane r as it is stored, two bf16 per 32-bit column.
      mbar_wait(b_res, 0, &abort_flag, 208);
      const uint8_t *src = (half ? g_tile : q_tile) + r * C::kRowBytes;
      uint32_t wr[D / 2];
#pragma unroll
      for (int ch = 0; ch < D / 8; ++ch) {
        const int pos = D == 64 ? (ch ^ (r & 7)) : (ch ^ ((r >> 1) & 3));  // the TMA swizzle of the tile
        const uint4 v4 = *reinterpret_cast<const uint4 *>(src + (pos << 4));
        wr[4 * ch] = v4.x; wr[4 * ch + 1] = v4.y; wr[4 * ch + 2] = v4.z; wr[4 * ch + 3] = v4.w;
      }
      const uint32_t ta = (half ? tmem_ga : tmem_qa) + lane_off;
      if constexpr (D == 64) tmem_st32u(ta, wr); else tmem_st16u(ta, wr);
      tmem_wait_st();
      tc_fence_before();
      warp_arrive(b_aready, lane);
    }

    // Half `half` of every pair belongs to the four warps of group `half`, which have a buffer of their own:
    // a thread takes all 32 columns, in two passes of 16.
    const uint32_t tb = tmem_base + 64 * half + lane_off;  // S; dP 32 columns further
    const uint8_t *jc = jcls + 8 * half + quarter;  // classes of the half tile's two column halves: [0], [4]
    int c0_n = nvis > 0 ? jc[0] : 0, c1_n = nvis > 0 ? jc[4] : 0;
    for (int i = 0; i < nvis; ++i) {
      const int cls0 = c0_n, cls1 = c1_n;
      if (i + 1 < nvis) {  // ahead of their use
        c0_n = jc[(i + 1) * 16];
        c1_n = jc[(i + 1) * 16 + 4];
      }
      uint32_t hL = 0u, hS = 0u;  // this thread's 32 keys
      const bool masked = ((cls0 | cls1) & 8) || (cls0 & 3) == 3 || (cls1 & 3) == 3;
      if ((cls0 | cls1) & 8) {  // mixed: per-lane column masks
        const int hx = list[2 * i + half], f = lflags[2 * i + half], jt = hx >> 1, col = 32 * (hx & 1), c0 = 32 * hx;
        const uint32_t mc = cols32_le(t_last - c0) & cols32_ge(pad0 - c0);
        if (f & 1) hL = mc & expand_block_bits32(pq ? rowb[r * nT + jt] : selb[g * nT + jt], s.Bk, col);
        if (f & 2) hS = mc & (s.stis_mode ? (uint32_t)(st_key_cols(s, t, jt * 64, causal) >> col) : st_window32(s, t, c0, causal));
      } else if (masked) {
        hL = (cls0 & 1 ? 0xffffu : 0u) | (cls1 & 1 ? 0xffff0000u : 0u);
        hS = (cls0 & 2 ? 0xffffu : 0u) | (cls1 & 2 ? 0xffff0000u : 0u);
      }
      mbar_wait(b_sfull + 8 * half, i & 1, &abort_flag, 207);
      __syncwarp();
      tc_fence_after();
      // dS (bf16 pairs) goes over the first 8 of a pass's 16 S columns
      auto pass = [&](auto full_tag, int ps, bool anyL, bool anyS, uint32_t xL, uint32_t xS) {
        constexpr bool FULL = decltype(full_tag)::value;
        uint32_t dw[8];
        if (anyL || anyS) {
          float sv[16], dp[16];
          tmem_ld16(tb + 16 * ps, sv);
          tmem_ld16(tb + 32 + 16 * ps, dp);
          tmem_wait_ld();
          if (!FULL && (PLAIN || (anyL && anyS))) {
            dq_tile<true, FULL>(sv, dp, xL, xS, sc2, nlL, nlS, alpha, beta, nDL, nDS, dalL, dw);
          } else {
            float2 dal = make_float2(0.f, 0.f);
            dq_tile<false, FULL>(sv, dp, anyL ? xL : xS, 0u, sc2, anyL ? nlL : nlS, 0.f, anyL ? alpha : beta, 0.f, anyL ? nDL : nDS, 0.f, dal, dw);
            if (anyL) dalL = fadd2(dalL, dal);
            else dalS = fadd2(dalS, dal);
          }
        } else {
#pragma unroll
          for (int c = 0; c < 8; ++c) dw[c] = 0u;
        }
        tmem_st8u(tb + 16 * ps, dw);
      };
      if (masked) {
#pragma unroll 2
        for (int ps = 0; ps < 2; ++ps) {
          const uint32_t xL = (hL >> (16 * ps)) & 0xffffu, xS = (hS >> (16 * ps)) & 0xffffu;
          pass(std::false_type(), ps, __any_sync(0xffffffffu, xL != 0u), __any_sync(0xffffffffu, xS != 0u), xL, xS);
        }
      } else {
        pass(std::true_type(), 0, cls0 & 1, cls0 & 2, 0u, 0u);
        pass(std::true_type(), 1, cls1 & 1, cls1 & 2, 0u, 0u);
      }
      tmem_wait_st();
      tc_fence_before();
      warp_arrive(b_tfull + 8 * half, lane);
    }

    {
      const float dal = (dalL.x + dalL.y) - (dalS.x + dalS.y);
      double a = row_valid ? (double)dal : 0.0;  // fixed-shape tree over the warp, then over the warps
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      if (lane == 0) red[warp] = a;
    }
    if (nvis > 0) {
      mbar_wait(b_all, 0, &abort_flag, 209);
      __syncwarp();
      tc_fence_after();
    }
    float o[OC];
    if (nvis > 0) {
      tmem_ld<OC>(tmem_dq + lane_off + half * OC, o);
      tmem_wait_ld();
    }
    {
      // The rows go to shared memory in the layout a TMA store expects (the K/V stages are free:
      // every load has landed and every MMA has completed); one bulk store then writes whole lines,
      // clipped at L by the hardware.  Padded rows are written as zeros.
      const bool live = nvis > 0 && row_valid;
#pragma unroll
      for (int ch = 0; ch < OC / 8; ++ch) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int c = ch * 8 + e * 2;
          w[e] = live ? pack_bf16(o[c] * s.scale, o[c + 1] * s.scale) : 0u;
        }
        if (ADDS && add_dq && live) add_row_chunk(w, add_dq + row_offset(s, n, hr, t) + half * OC + ch * 8);
        store_row_chunk<D>(kv_tiles, r, half * (OC / 8) + ch, make_uint4(w[0], w[1], w[2], w[3]));
      }
      fence_async_smem();
      named_bar_sync(5, kComputeWarps * 32);
      if (tid == 0) {
        tma_store_4d(&tmdq, smem_u32(kv_tiles), 0, row0, h, n);
        tma_store_commit();
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  // d alpha partial of this CTA -> first query-block slot of its rows, zeros in the rest
  // (PACK: one partial per head, from the warps of that head's 64 rows)
  if (tid == 0) {
    if (PACK) {
      const int nb = 64 / s.Bk;
      for (int hh = 0; hh < 2; ++hh) {
        double a = 0.0;
        for (int i = 0; i < kComputeWarps; ++i)
          if (((i & 3) >> 1) == hh) a += red[i];  // fixed order
        for (int gq = 0; gq < nb; ++gq)
          if (st * nb + gq < s.M) dalpha_part[((int64_t)n * s.H + h + hh) * s.M + st * nb + gq] = gq == 0 ? a : 0.0;
      }
    } else {
      const int G = 128 / s.Bk;
      double a = 0.0;
      for (int i = 0; i < kComputeWarps; ++i) a += red[i];  // fixed order
      for (int gq = 0; gq < G; ++gq)
        if (st * G + gq < s.M) dalpha_part[(int64_t)u * s.M + st * G + gq] = gq == 0 ? a : 0.0;
    }
  }
  if (nvis == 0 && tid == 0) mbar_wait(b_res, 0, &abort_flag, 221);  // no load may outlive the CTA
  if (tid == 0) tma_store_wait_read();
  finish(warp, tmem_base, kBwdTmemCols, &abort_flag, status);
}

// ------------------------------------------------------------------------- backward dK, dV
// 16 query columns of one tile for one key row: W^T and dS^T packed to bf16 pairs.  st points at
// the records of these 8 query pairs: {nl_lt(2), -Delta_lt(2)} {nl_st(2), -Delta_st(2)} per pair
// (nl = -(lse * log2e - log2 weight): the branch weight rides in the exponent).  Two columns per
// FMA / ADD / MUL instruction.
// BOTH as in dq_tile: with one branch st points at that branch's half of the records.
template <bool BOTH, bool FULL>
__device__ __forceinline__ void dkdv_tile(const float (&sv)[16], const float (&dp)[16], uint32_t hL,
                                          uint32_t hS, float sc2, const float4 *st, uint32_t (&ww)[8],
                                          uint32_t (&dw)[8]) {
  const float2 sc = make_float2(sc2, sc2);
#pragma unroll
  for (int c = 0; c < 16; c += 2) {
    const float2 s2 = make_float2(sv[c], sv[c + 1]), dp2 = make_float2(dp[c], dp[c + 1]);
    const float4 r = st[c];  // pair c / 2
    const float2 x = ffma2(s2, sc, make_float2(r.x, r.y));
    float2 w = make_float2(exp2f(x.x), exp2f(x.y));
    if (!FULL) {
      w.x = bit(hL, c) ? w.x : 0.f;
      w.y = bit(hL, c + 1) ? w.y : 0.f;
    }
    float2 d = fmul2(w, fadd2(dp2, make_float2(r.z, r.w)));
    if (BOTH) {
      const float4 q = st[c + 1];  // short-term half
      const float2 y = ffma2(s2, sc, make_float2(q.x, q.y));
      float2 p = make_float2(exp2f(y.x), exp2f(y.y));
      if (!FULL) {
        p.x = bit(hS, c) ? p.x : 0.f;
        p.y = bit(hS, c + 1) ? p.y : 0.f;
      }
      w = fadd2(w, p);
      d = ffma2(p, fadd2(dp2, make_float2(q.z, q.w)), d);
    }
    ww[c >> 1] = pack_bf16(w.x, w.y);
    dw[c >> 1] = pack_bf16(d.x, d.y);
  }
}

// d alpha partials -> dgate[H][2], by one CTA, head after head: thread i adds the entries i, i + 384, ... in
// ascending order, then a fixed shuffle tree and the warps in order.  (As a kernel of its own it was
// another 8 us of launch and latency.)
__device__ __forceinline__ void reduce_gate(const Shape &s, const float *gate, const double *part, float *dgate) {
  __shared__ double red[2][kKvThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, total = s.B * s.M;
  for (int h = 0; h < s.H; ++h) {
    double a = 0.0;
#pragma unroll 8
    for (int i = threadIdx.x; i < total; i += kKvThreads) a += __ldcg(part + ((int64_t)(i / s.M) * s.H + h) * s.M + i % s.M);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) red[h & 1][warp] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
      double x = 0.0;
      for (int w = 0; w < kKvThreads / 32; ++w) x += red[h & 1][w];
      const double al = 1.0 / (1.0 + exp(-((double)gate[h * 2 + 0] - (double)gate[h * 2 + 1])));
      const double g0 = al * (1.0 - al) * x;
      dgate[h * 2 + 0] = (float)g0;
      dgate[h * 2 + 1] = (float)(-g0);
    }
  }
}

template <int D, int MODE>
__global__ void __launch_bounds__(kKvThreads, 2) bwd_dkdv_tc_kernel(
    const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
    const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmg, Shape s,
    const int32_t *__restrict__ seq_lens, const uint8_t *__restrict__ kmeta,
    const float4 *__restrict__ qstats, const __grid_constant__ CUtensorMap tmdk,
    const __grid_constant__ CUtensorMap tmdv, const __grid_constant__ CUtensorMap tmq32,
    const __grid_constant__ CUtensorMap tmg32, int32_t *__restrict__ status, int nT, int hs,
    __nv_bfloat16 *dk, __nv_bfloat16 *dv, const float *__restrict__ gate,
    const double *__restrict__ dalpha_part, float *__restrict__ dgate, int accumulate) {
  constexpr bool PLAIN = MODE == kPlain, ADDS = MODE == kPass;
  using C = Cfg<D>;
  constexpr int STAGES = kKvStages;
  constexpr int OC = D / 2;
  constexpr int kStageBytes = 2 * C::kSmallBytes + kStatBytes;  // Q, dO, row records
  extern __shared__ uint8_t smem_raw[];
  // barriers: full[STAGES], empty[STAGES], res, meta, per buffer s_full[2], t_full[2]; all_done
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 7];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  grid_release();
  const int nKT = (s.L + 127) >> 7;
  // A CTA owns 128 keys of one (batch, key/value head) and collects from every query head of the
  // group.  Early keys have the most visitors, so the grid runs tile-major: every unit's first
  // tile, then every unit's second, ... and the light tiles fill the tail.
  // With clusters (hs CTAs) the heads of the group are split over a cluster's CTAs, rank r taking the
  // r-th G / hs of them, and the CTAs add their sums at the end.
  const int nU = s.B * s.Hkv;
  const int rank = (int)blockIdx.x % hs;
  int blk = (int)blockIdx.x / hs;
  if (dgate && --blk < 0) {  // one more CTA (or cluster), the first (as the last it would be the tail): the gate gradient
    grid_wait();             // the dQ kernel's partial sums
    if (rank == 0) reduce_gate(s, gate, dalpha_part, dgate);
    return;
  }
  const int kt = blk / nU, uk = blk % nU, n = uk / s.Hkv, hk = uk % s.Hkv, Gs = s.G / hs, h_first = hk * s.G + rank * Gs;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len;
  const int key0 = kt * 128, key_last = min(s.L - 1, key0 + 127);
  const int Lpad = nT * 64;

  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t *tiles = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint8_t *k_tile = tiles;
  uint8_t *v_tile = k_tile + C::kBigBytes;
  uint8_t *qg_tiles = v_tile + C::kBigBytes;  // [stage][Q, dO, row records]
  uint8_t *meta = qg_tiles + STAGES * kStageBytes;  // image built by tc_meta_kernel
  const bool causal = PLAIN || s.causal;
  const int pq = PLAIN ? 0 : s.pq;
  const MetaLayout ml = meta_layout(nT, pq);
  const uint64_t *inv64 = reinterpret_cast<const uint64_t *>(meta + ml.rows);  // (selection per query position) [8][nT]
  const uint8_t *invb = meta + ml.sel;                  // [8][nT] bytes: per key block, per query tile
  const uint16_t *list = reinterpret_cast<const uint16_t *>(meta + ml.list);
  const uint8_t *lflags = meta + ml.flags;
  const uint8_t *kcls = meta + ml.jcls;                 // [listed pair][half][compute warp]

  const uint32_t b_full = smem_u32(&bars[0]), b_empty = smem_u32(&bars[STAGES]);
  const uint32_t b_res = smem_u32(&bars[2 * STAGES]), b_meta = smem_u32(&bars[2 * STAGES + 1]);
  const uint32_t b_sfull = smem_u32(&bars[2 * STAGES + 2]), b_tfull = smem_u32(&bars[2 * STAGES + 4]);
  const uint32_t b_all = smem_u32(&bars[2 * STAGES + 6]);

  if (tid == 0) {
    abort_flag = (*status != 0) ? 1 : 0;
    tma_prefetch_desc(&tmq);
    tma_prefetch_desc(&tmk);
    tma_prefetch_desc(&tmv);
    tma_prefetch_desc(&tmg);
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(b_full + 8 * i, 1);
      mbar_init(b_empty + 8 * i, 1);
    }
    mbar_init(b_res, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_sfull + 8 * i, 1);
      mbar_init(b_tfull + 8 * i, kComputeWarps / 2);
    }
    mbar_init(b_meta, 1);
    mbar_init(b_all, 1);
    mbar_fence_init();
    // the CTA's tile lists and its resident tiles
    mbar_expect_tx(b_meta, (uint32_t)ml.bwd);
    bulk_load(smem_u32(meta), kmeta + ((size_t)uk * nKT + kt) * ml.bwd, (uint32_t)ml.bwd, b_meta);
    mbar_expect_tx(b_res, 2 * C::kBigBytes);
    tma_load_4d(smem_u32(k_tile), &tmk, b_res, 0, key0, hk, n);
    tma_load_4d(smem_u32(v_tile), &tmv, b_res, 0, key0, hk, n);
  }
  if (warp == 0) {
    __syncwarp();
    tmem_alloc(smem_u32(&tmem_slot), kBwdTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  mbar_wait(b_meta, 0, &abort_flag, 224);
  // The tile list is the same for every query head of the group (one selection per group): the
  // kernel walks it once per head, item x = (head x / nlist, pair x % nlist).
  const int listed = *reinterpret_cast<const int *>(meta + ml.counts);
  const int nlist = uniform(*(volatile int *)&abort_flag ? 0 : listed);  // (the lists may not be there)
  const int nvis = nlist * Gs;
  const uint32_t tmem_base = (uint32_t)uniform((int)tmem_slot);
  // the half tile of group hh uses the buffer at column 64 hh: S^T in its first 32 columns, dP^T behind
  const uint32_t tmem_dv = tmem_base + 128, tmem_dk = tmem_base + 192;

  if (warp >= kComputeWarps) {
    // ===================== two single-thread roles, one warp each =====================
    setmaxnreg_dec<kProducerRegs>();
    if (warp == kComputeWarps && nvis > 0) {
      // ---- loader: K, V once; Q, dO tiles and their row records up to STAGES ahead ----
      int lj = 0, h = h_first;
      bool go = true;
      for (int j = 0; j < nvis; ++j) {
        const int sj = j % STAGES;
        if (j >= STAGES) go = mbar_wait(b_empty + 8 * sj, ((j - STAGES) / STAGES) & 1, &abort_flag, 214) && go;
        const uint32_t bar = b_full + 8 * sj;
        const uint32_t qt_ = smem_u32(qg_tiles + sj * kStageBytes);
        if (lj == nlist) { lj = 0; ++h; }  // the next query head of the group walks the same list
        const uint32_t pair = reinterpret_cast<const uint32_t *>(list)[lj++];
        const int row0 = (int)(pair & 0xffffu) * 32, row1 = (int)(pair >> 16) * 32;
        const float4 *rec = qstats + ((int64_t)n * s.H + h) * Lpad;
        if (elect_one() && go) {
          mbar_expect_tx(bar, kStageBytes);
          tma_load_halves(qt_, C::kSmallBytes / 2, &tmq, &tmq32, bar, row0, row1, h, n);
          tma_load_halves(qt_ + C::kSmallBytes, C::kSmallBytes / 2, &tmg, &tmg32, bar, row0, row1, h, n);
          const int rec1 = row1 < Lpad ? row1 : row0;  // (the half behind the last has no records)
          if (rec1 == row0 + 32) {
            bulk_load(qt_ + 2 * C::kSmallBytes, rec + row0, kStatBytes, bar);
          } else {
            bulk_load(qt_ + 2 * C::kSmallBytes, rec + row0, kStatBytes / 2, bar);
            bulk_load(qt_ + 2 * C::kSmallBytes + kStatBytes / 2, rec + rec1, kStatBytes / 2, bar);
          }
        }
        __syncwarp();
      }
    } else if (warp == kComputeWarps + 1 && nvis > 0) {
      // ---- S^T = K Q^T, dP^T = V dO^T of half tile x into buffer x % 2, then, once its W^T and dS^T are in
      // tensor memory, dV += W^T dO, dK += dS^T Q and behind them the first stage of half tile x + 2 (see the
      // dQ kernel) ----
      constexpr uint32_t idesc_s = instr_desc(128, 32, 0, 0), idesc_o = instr_desc(128, D, 0, 1);
      const uint64_t dkd = smem_desc(smem_u32(k_tile), 16, C::kAtomBytes, C::kSwizzle);
      const uint64_t dvd = smem_desc(smem_u32(v_tile), 16, C::kAtomBytes, C::kSwizzle);
      auto first_stage = [&](int sj, int hh) {
        const uint32_t qt_ = smem_u32(qg_tiles + sj * kStageBytes) + hh * 32 * C::kRowBytes;
        const uint64_t dqd = smem_desc(qt_, 16, C::kAtomBytes, C::kSwizzle);
        const uint64_t dgd = smem_desc(qt_ + C::kSmallBytes, 16, C::kAtomBytes, C::kSwizzle);
        const uint32_t ts = tmem_base + 64 * hh;
#pragma unroll
        for (int k = 0; k < D / 16; ++k) umma_bf16(ts, dkd + 2 * k, dqd + 2 * k, idesc_s, k > 0);
#pragma unroll
        for (int k = 0; k < D / 16; ++k) umma_bf16(ts + 32, dvd + 2 * k, dgd + 2 * k, idesc_s, k > 0);
        umma_commit(b_sfull + 8 * hh);
      };
      mbar_wait(b_res, 0, &abort_flag, 210);
      mbar_wait(b_full, 0, &abort_flag, 213);
      tc_fence_after();
      if (elect_one()) {
        first_stage(0, 0);
        first_stage(0, 1);
      }
      __syncwarp();
      for (int i = 0, sj = 0; i < nvis; ++i) {
        const int sn = sj + 1 == STAGES ? 0 : sj + 1;
        const bool more = i + 1 < nvis;
        const uint32_t q_tile = smem_u32(qg_tiles + sj * kStageBytes);
        const uint64_t dgm = smem_desc(q_tile + C::kSmallBytes, C::kSmallBytes, C::kAtomBytes, C::kSwizzle);
        const uint64_t dqm = smem_desc(q_tile, C::kSmallBytes, C::kAtomBytes, C::kSwizzle);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          const uint32_t tb = tmem_base + 64 * hh;
          if (hh == 0 && more) mbar_wait(b_full + 8 * sn, ((i + 1) / STAGES) & 1, &abort_flag, 215);
          mbar_wait(b_tfull + 8 * hh, i & 1, &abort_flag, 211);
          tc_fence_after();
          if (elect_one()) {
            // 16 queries per step: the bf16 pairs of column half kk, 8 columns
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              umma_bf16_ts(tmem_dv, tb + 16 * kk, dgm + (2 * hh + kk) * C::kKStep, idesc_o, (i | hh | kk) != 0);
#pragma unroll
            for (int kk = 0; kk < 2; ++kk)
              umma_bf16_ts(tmem_dk, tb + 32 + 16 * kk, dqm + (2 * hh + kk) * C::kKStep, idesc_o, (i | hh | kk) != 0);
            if (hh == 1) umma_commit(more ? b_empty + 8 * sj : b_all);  // every product on this stage has completed
            if (more) first_stage(sn, hh);
          }
          __syncwarp();
        }
        sj = sn;
      }
    }
  } else {
    setmaxnreg_inc<kKvComputeRegs>();
    const int quarter = warp & 3, half = warp >> 2;
    const int r = quarter * 32 + lane, p = key0 + r, g = r / s.Bk;
    const bool row_ok = p < s.L, row_valid = row_ok && p >= pad0;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const float sc2 = s.scale * kLog2e;

    // Half hh of every pair (32 queries) belongs to the four warps of group hh = half, which have a buffer of
    // their own: a thread takes all 32 columns, in two passes of 16.
    const uint32_t tb = tmem_base + 64 * half + lane_off;
    const int q0 = 32 * half;
    int li = 0;
    for (int i = 0; i < nvis; ++i) {
      if (li == nlist) li = 0;
      const uint8_t *cls2 = kcls + li * 16 + 8 * half + quarter;  // classes of the half tile's two column halves
      const int cls0 = cls2[0], cls1 = cls2[4];
      uint32_t hL = 0u, hS = 0u;
      const bool masked = ((cls0 | cls1) & 8) || (cls0 & 3) == 3 || (cls1 & 3) == 3;
      if ((cls0 | cls1) & 8) {  // a mixed half: per-lane column masks
        if (row_valid) {
          const int hx = list[2 * li + half], f = lflags[2 * li + half], qt = hx >> 1, col = 32 * (hx & 1), t0 = 32 * hx;
          const uint32_t mc = cols32_ge((causal ? p : pad0) - t0) & cols32_le(s.L - 1 - t0);
          if (f & 1) hL = mc & (pq ? (uint32_t)(inv64[g * nT + qt] >> col) : expand_block_bits32(invb[g * nT + qt], s.Bk, col));
          if (f & 2) hS = mc & (uint32_t)(st_query_cols(s, p, qt * 64, causal) >> col);
        }
      } else if (masked) {
        hL = (cls0 & 1 ? 0xffffu : 0u) | (cls1 & 1 ? 0xffff0000u : 0u);
        hS = (cls0 & 2 ? 0xffffu : 0u) | (cls1 & 2 ? 0xffff0000u : 0u);
      }
      ++li;
      mbar_wait(b_full + 8 * (i % STAGES), (i / STAGES) & 1, &abort_flag, 216);  // the row records have landed
      const float4 *stt = reinterpret_cast<const float4 *>(qg_tiles + (i % STAGES) * kStageBytes + 2 * C::kSmallBytes);
      mbar_wait(b_sfull + 8 * half, i & 1, &abort_flag, 217);
      __syncwarp();
      tc_fence_after();
      // W^T and dS^T of the 16 columns of a pass go, as bf16 pairs, over the first 8 of them in S^T / dP^T.
      auto pass = [&](auto full_tag, int ps, bool anyL, bool anyS, uint32_t xL, uint32_t xS) {
        constexpr bool FULL = decltype(full_tag)::value;
        uint32_t ww[8], dw[8];
        if (anyL || anyS) {
          float sv[16], dp[16];
          tmem_ld16(tb + 16 * ps, sv);
          tmem_ld16(tb + 32 + 16 * ps, dp);
          tmem_wait_ld();
          const float4 *sq = stt + q0 + 16 * ps;  // 8 pairs x 2 float4
          if (!FULL && (PLAIN || (anyL && anyS))) dkdv_tile<true, FULL>(sv, dp, xL, xS, sc2, sq, ww, dw);
          else dkdv_tile<false, FULL>(sv, dp, anyL ? xL : xS, 0u, sc2, sq + (anyL ? 0 : 1), ww, dw);
        } else {
#pragma unroll
          for (int c = 0; c < 8; ++c) { ww[c] = 0u; dw[c] = 0u; }
        }
        tmem_st8u(tb + 16 * ps, ww);
        tmem_st8u(tb + 32 + 16 * ps, dw);
      };
      if (masked) {
#pragma unroll 2
        for (int ps = 0; ps < 2; ++ps) {
          const uint32_t xL = (hL >> (16 * ps)) & 0xffffu, xS = (hS >> (16 * ps)) & 0xffffu;
          pass(std::false_type(), ps, __any_sync(0xffffffffu, xL != 0u), __any_sync(0xffffffffu, xS != 0u), xL, xS);
        }
      } else {
        pass(std::true_type(), 0, cls0 & 1, cls0 & 2, 0u, 0u);
        pass(std::true_type(), 1, cls1 & 1, cls1 & 2, 0u, 0u);
      }
      tmem_wait_st();
      tc_fence_before();
      warp_arrive(b_tfull + 8 * half, lane);
    }

    if (nvis > 0) {
      mbar_wait(b_all, 0, &abort_flag, 218);
      __syncwarp();
      tc_fence_after();
    }
    float ov[OC], okk[OC];
    if (nvis > 0) {
      tmem_ld<OC>(tmem_dv + lane_off + half * OC, ov);
      tmem_ld<OC>(tmem_dk + lane_off + half * OC, okk);
      tmem_wait_ld();
    }
    const bool live = nvis > 0 && row_valid;
    if (hs > 1) {
      // this CTA's sums in fp32, in the (now free) Q/dO stages: [dV, dK][128 rows][D + 4]
      float *acc = reinterpret_cast<float *>(qg_tiles) + r * (D + 4) + half * OC;
#pragma unroll
      for (int c = 0; c < OC; c += 4) {
        *reinterpret_cast<float4 *>(acc + c) =
            live ? make_float4(ov[c], ov[c + 1], ov[c + 2], ov[c + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
        *reinterpret_cast<float4 *>(acc + 128 * (D + 4) + c) =
            live ? make_float4(okk[c], okk[c + 1], okk[c + 2], okk[c + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    } else {
      // staged in the (now free) Q/dO stages, then two whole-line bulk stores clipped at L
      uint8_t *sv_t = qg_tiles, *sk_t = qg_tiles + C::kBigBytes;
#pragma unroll
      for (int ch = 0; ch < OC / 8; ++ch) {
        uint32_t wv[4], wk[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int c = ch * 8 + e * 2;
          wv[e] = live ? pack_bf16(ov[c], ov[c + 1]) : 0u;
          wk[e] = live ? pack_bf16(okk[c] * s.scale, okk[c + 1] * s.scale) : 0u;
        }
        if (ADDS && accumulate && live) {
          const int64_t off = row_offset_kv(s, n, hk, p) + half * OC + ch * 8;
          add_row_chunk(wv, dv + off);
          add_row_chunk(wk, dk + off);
        }
        store_row_chunk<D>(sv_t, r, half * (OC / 8) + ch, make_uint4(wv[0], wv[1], wv[2], wv[3]));
        store_row_chunk<D>(sk_t, r, half * (OC / 8) + ch, make_uint4(wk[0], wk[1], wk[2], wk[3]));
      }
      fence_async_smem();
      named_bar_sync(5, kComputeWarps * 32);
      if (tid == 0) {
        tma_store_4d(&tmdv, smem_u32(sv_t), 0, key0, hk, n);
        tma_store_4d(&tmdk, smem_u32(sk_t), 0, key0, hk, n);
        tma_store_commit_and_wait();
      }
    }
  }
  if (hs > 1) {
    // every CTA of the cluster adds its share of the rows over the cluster, in rank order
    static_assert(2 * 128 * (D + 4) * 4 <= STAGES * kStageBytes, "the fp32 sums fit in the stages");
    cg::cluster_group cluster = cg::this_cluster();
    __syncwarp();
    cluster.sync();
    if (warp < kComputeWarps) {
      const int rows = 128 / hs;
      float *own = reinterpret_cast<float *>(qg_tiles);
      for (int i = tid; i < 2 * rows * (D / 8); i += kComputeWarps * 32) {
        const int ch = i % (D / 8), lr = (i / (D / 8)) % rows, which = i / (rows * (D / 8));
        const int rr = rank * rows + lr, p = key0 + rr;
        if (p >= s.L) continue;
        float x[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        for (int k = 0; k < hs; ++k) {
          const float4 *o = reinterpret_cast<const float4 *>(cluster.map_shared_rank(own, k) +
                                                             (which * 128 + rr) * (D + 4) + ch * 8);
          const float4 a = o[0], b = o[1];
          x[0] += a.x; x[1] += a.y; x[2] += a.z; x[3] += a.w; x[4] += b.x; x[5] += b.y; x[6] += b.z; x[7] += b.w;
        }
        const float f = which ? s.scale : 1.f;
        __nv_bfloat16 *row = (which ? dk : dv) + row_offset_kv(s, n, hk, p) + ch * 8;
        uint32_t w[4] = {pack_bf16(x[0] * f, x[1] * f), pack_bf16(x[2] * f, x[3] * f), pack_bf16(x[4] * f, x[5] * f),
                         pack_bf16(x[6] * f, x[7] * f)};
        if (ADDS && accumulate) add_row_chunk(w, row);
        *reinterpret_cast<uint4 *>(row) = make_uint4(w[0], w[1], w[2], w[3]);
      }
    }
    __syncwarp();
    cluster.sync();  // nobody leaves while its sums are being read
  }
  if (nvis == 0 && tid == 0) mbar_wait(b_res, 0, &abort_flag, 222);  // no load may outlive the CTA
  finish(warp, tmem_base, kBwdTmemCols, &abort_flag, status);
  if (tid == 0) grid_wait();  // (see grid_wait: by now the dQ kernel has mostly completed)
}

}  // namespace

// Grouped heads: a CTA walks its tile list once per head, so with few CTAs the one with the first keys is the kernel's
// time (170 us at B 8, 8 heads on 2, L 1500, 192 CTAs): the heads are split over clusters of 2 and 4 while the CTAs fit the
// chip's places or a CTA's walk (key tiles times heads) is long against what it costs outside it.  With lengths, CTAs that
// hold padding alone end at once, so more of them are split.  The lines, from whole backward passes of 3834 shapes (two to eight
// heads a group, L 330 - 4000, 100 - 590 CTAs, every mask and option; 1514 of them with lengths down to 1, L / 10, L / 4 and
// L / 2): 0.4 % off the best split on average, at worst 14 (lengths: 19) %; one line for both was 1.9 % off, at worst 49 %.
// us with 1 / 2 / 4 CTAs, D 64, four heads a group: L 700, 108 CTAs 63 / 47 / 56, 360 111 / 125 / 156; L 2048, 160 147 / 103 /
// 113; two heads: L 1400, 352 CTAs 82 / 94; L 4000, 512 182 / 197 with links, L 1280, 420 with lengths from 320 82 / 74.
int dkdv_split(const Shape &s, bool lengths) {
  const int64_t nST = (s.L + 127) / 128, ctas = nST * s.B * s.Hkv;
  const int64_t walk = lengths ? 16 : 6, fixed = lengths ? 100 : 120, most = lengths ? 1000 : 592;
  int hs = 1;
  while (hs < 4 && s.G % (2 * hs) == 0 && ctas * hs < most && ctas * hs <= walk * nST * (s.G / hs) + fixed) hs *= 2;
  return hs;
}

template <int D>
int launch_bwd_tc_t(const Shape &s, const void *q, const void *k, const void *v, const float *gate,
                    const int32_t *seq_lens, const int32_t *idx, const void *out_lt,
                    const void *out_st, const float *lse, const void *dout, void *dq, void *dk,
                    void *dv, float *dgate, const Workspace &ws, cudaStream_t st, int branches, const float4 *records) {
  typedef __nv_bfloat16 bf;
  using C = Cfg<D>;
  CUtensorMap q128, k64, v64, g128, q64, k128, v128, g64, tdq, tdk, tdv, k32, v32, q32, g32;
  // (head-packed dQ kernel: a query-side box is 64 positions of two heads)
  const int qrows = s.pack ? 64 : 128, qheads = s.pack ? 2 : 1;
  if (make_tensor_map(&q128, q, s, qrows, false, qheads) || make_tensor_map(&k64, k, s, 64, true) ||
      make_tensor_map(&v64, v, s, 64, true) || make_tensor_map(&g128, dout, s, qrows, false, qheads) ||
      make_tensor_map(&q64, q, s, 64) || make_tensor_map(&k128, k, s, 128, true) ||
      make_tensor_map(&v128, v, s, 128, true) || make_tensor_map(&g64, dout, s, 64) ||
      make_tensor_map(&tdq, dq, s, qrows, false, qheads) || make_tensor_map(&tdk, dk, s, 128, true) ||
      make_tensor_map(&tdv, dv, s, 128, true) || make_tensor_map(&k32, k, s, 32, true) ||
      make_tensor_map(&v32, v, s, 32, true) || make_tensor_map(&q32, q, s, 32) || make_tensor_map(&g32, dout, s, 32))
    return BLOSSOM_ERR_CUDA;
  const int nT = (s.L + 63) / 64, nST = (s.L + 127) / 128;
  const unsigned grid = (unsigned)nST * (unsigned)(s.B * s.H);
  const size_t lists = meta_layout(nT, s.pq).bwd;
  const size_t smem_dq = 1024 + 2 * C::kBigBytes + kDqStages * 2 * C::kSmallBytes + lists;
  const size_t smem_kv = 1024 + 2 * C::kBigBytes + kKvStages * (2 * C::kSmallBytes + kStatBytes) + lists;
  auto kern_dq = bwd_dq_tc_kernel<D, kGeneral, false>;
  auto kern_kv = bwd_dkdv_tc_kernel<D, kGeneral>;
  if (branches != 3) {
    kern_dq = s.pack ? bwd_dq_tc_kernel<D, kPass, true> : bwd_dq_tc_kernel<D, kPass, false>;
    kern_kv = bwd_dkdv_tc_kernel<D, kPass>;
  } else if (s.causal && !s.pq) {
    kern_dq = s.pack ? bwd_dq_tc_kernel<D, kPlain, true> : bwd_dq_tc_kernel<D, kPlain, false>;
    kern_kv = bwd_dkdv_tc_kernel<D, kPlain>;
  } else if (s.pack) {
    kern_dq = bwd_dq_tc_kernel<D, kGeneral, true>;
  }
  if (!allow_smem(kern_dq, smem_dq) || !allow_smem(kern_kv, smem_kv)) return BLOSSOM_ERR_CUDA;
  if (!records && !s.reuse_lists)  // (the passes of the input-dependent gate have got theirs)
    if (int rc = launch_tc_meta(s, seq_lens, idx, ws.qmeta, ws.kmeta, st, ws.status + kTicketWord, branches)) return rc;
  const float4 *rec = records ? records : ws.qstats;
  if (!records) {
    LaunchScope ls(K_BWD_PREP, st);
    const int Lpad = nT * 64;
    const dim3 gp((unsigned)(s.B * s.H), (unsigned)((Lpad + prep_rows<D>() - 1) / prep_rows<D>()));
    launch_chained(bwd_prep_kernel<D>, gp, dim3(256), 0, st, s, gate, seq_lens, (const bf *)out_lt,
                   (const bf *)out_st, lse, (const bf *)dout, ws.qstats, Lpad, ws.status_bwd);
  }
  {
    LaunchScope ls(K_BWD_DQ_TC, st);
    const unsigned grid_q = s.pack ? (unsigned)nT * (unsigned)(s.B * (s.H / 2)) : grid;
    launch_chained(kern_dq, dim3(grid_q), dim3(kKvThreads), smem_dq, st, q128, k64, v64, g128, s, gate, seq_lens, lse,
                   (const uint8_t *)ws.qmeta, tdq, k32, v32, rec, ws.dalpha, ws.status_bwd, nT,
                   branches == 2 ? (const bf *)dq : nullptr);
  }
  if (dgate && branches != 3)  // between the two: it depends on neither, and its latency disappears
    if (int rc = launch_gate_param_grad(s, ws, dgate, st, 1)) return rc;
  float *dgate_here = branches == 3 ? dgate : nullptr;
  {
    LaunchScope ls(K_BWD_DKDV_TC, st);
    const unsigned ctas = (unsigned)nST * (unsigned)(s.B * s.Hkv);
    const unsigned hs = (unsigned)dkdv_split(s, seq_lens != nullptr);
    const dim3 grid_k((ctas + (dgate_here ? 1 : 0)) * hs);
    if (hs > 1)
      launch_chained_cluster(kern_kv, grid_k, dim3(kKvThreads), smem_kv, hs, st, q64, k128, v128, g64, s, seq_lens,
                             (const uint8_t *)ws.kmeta, rec, tdk, tdv, q32, g32, ws.status_bwd, nT, (int)hs, (bf *)dk, (bf *)dv, gate,
                             (const double *)ws.dalpha, dgate_here, branches == 2);
    else
      launch_chained(kern_kv, grid_k, dim3(kKvThreads), smem_kv, st, q64, k128, v128, g64, s, seq_lens,
                     (const uint8_t *)ws.kmeta, rec, tdk, tdv, q32, g32, ws.status_bwd, nT, 1, (bf *)dk, (bf *)dv, gate,
                     (const double *)ws.dalpha, dgate_here, branches == 2);
  }
  return cudaGetLastError() == cudaSuccess ? BLOSSOM_OK : BLOSSOM_ERR_CUDA;
}

template int launch_bwd_tc_t<32>(const Shape &, const void *, const void *, const void *, const float *,
                                 const int32_t *, const int32_t *, const void *, const void *,
                                 const float *, const void *, void *, void *, void *, float *, const Workspace &,
                                 cudaStream_t, int, const float4 *);
template int launch_bwd_tc_t<64>(const Shape &, const void *, const void *, const void *, const float *,
                                 const int32_t *, const int32_t *, const void *, const void *,
                                 const float *, const void *, void *, void *, void *, float *, const Workspace &,
                                 cudaStream_t, int, const float4 *);

}  // namespace tc
}  // namespace blossom
