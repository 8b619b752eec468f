// Tensor-core forward of the fused two-branch attention (bf16 storage, fp32 accumulate).
//
// A CTA owns 128 query rows (128 / Bk query blocks) and walks a list of items, two half tiles of 32 keys of
// one branch each (any two: tc_meta_kernel lists only those that some row needs): first what any of its query blocks
// selected (Eq. 14, 16), then what its rows reach through the window (Eq. 15, 17).  Keys that belong to both branches are visited
// once per phase.  With grouped heads (an even number per key/value head) the 128 rows are instead
// the same 64 positions of two heads of a group, which share their selection (Eq. 12), their window
// tiles and their K/V: every tile on the list then has work for every row (template flag PACK).
//
// The kernel is persistent: two CTAs on every SM take 128-row tiles, long rows first, from a counter
// until none is left.  A tile's fixed part (its lists, queries and first keys to wait for, the merges,
// the staged rows to be read by the bulk stores, launching a CTA) was most of the time of a kernel with
// a CTA per tile: with four items a tile 146 us for 4096 tiles of D 64, 98 - 104 us so; 11.5 items
// 228 -> 204 us, 27 items (L 4096) 388 -> 365 us, D 32 97 -> 91 us.  The roles therefore run on from
// tile to tile (item counters, stages and barrier phases continue), each as far ahead as its own inputs
// allow, while the softmax warps merge.  What is left is bound by the softmax warps' instructions, four warps a
// scheduler: issue slots 57 %, tensor pipe 34 % busy (B 4, H 8, L 4096, D 64).
//
// One warp issues both products of an item.  With a warp for each, S(i + 2) waited for the products of item
// i to be reported complete; in the order that products of one thread are taken to run in (tc_common.cuh) it follows
// them at once.  That, and roles, loop bounds and addresses in uniform registers (tc_common.cuh), took the kernel
// from 199 to 179 us at B 128, H 4, L 1024, D 64 and from 360 to 332 at B 16, H 8, L 4096.
// One code serves all items, masked or not, and both phases' ends: the logits that a row does not see become
// -infinity before the maximum is taken.  With variants for masked items, a vote which to take and the merge inlined three
// times the instructions did not come fast enough: 176 -> 165 us, 330 -> 310, D 32 78 -> 74, a selection per position
// at B 8, L 1500 51 -> 45 (2 - 4 us of each by classes per half of the keys, which leave out masks where one of two
// blocks of 32 was selected).
//
// CTA = 384 threads.  Warps 0..7 are softmax warps: a query row (= TMEM lane) is shared by two
// threads, warp w and warp w + 4, which split the KEYS of every item: group 0 (warps 0..3) takes
// the first half, group 1 the second.  Each group keeps its own running maximum and sum and its own
// accumulator (O_A += P[:, 0:32] V[0:32], O_B += P[:, 32:64] V[32:64]), so the two threads of a row
// never exchange anything inside the loop; the two partial results are merged, exactly as two
// halves of an online softmax, when a phase ends.  Sixteen softmax warps per SM instead of eight
// hide the latency of a thread's dependent chain (load, maximum, exponentials, store).
// Warps 8 and 9 stay converged; one elected lane of the first loads K/V tiles (TMA), one of the second issues
// S = Q K^T and the two O += P V products with P read from tensor memory.  Warp 11 stores the
// finished rows and fetches the next tile's lists and queries (warp 10 is spare).
//
// Tensor memory (256 columns): two logits / probability buffers [0,64) [64,128), O_A [128,128+D),
// O_B [192,192+D).  Item i uses buffer i % 2: S(i) lands there as fp32, a softmax thread reads its
// 32 logits and writes their probabilities (bf16 pairs) over the first 16 of them, from where the
// products read their first operand:
//
//   loader   : stage j <- K, V of item j once the products of item j - STAGES have completed
//   softmax  : wait s_full -> tcgen05.ld 32 logits -> online softmax of the half row (maximum
//              raised, and the group's accumulator rescaled, only when it grows by > 2^8) ->
//              tcgen05.st P -> arrive t_full[group][i%2]
//   issuer   : (S(0) -> s_full[0], S(1) -> s_full[1] of a tile;) wait t_full[0] -> O_A += P_A V[0:32];
//              wait t_full[1] -> O_B += P_B V[32:64] -> commit done[i%2], release the stage; wait
//              K(i+2) -> S(i+2) into the same buffer -> s_full[i%2]
//
// When the long-term phase ends the merged, normalised rows go (as bf16) to a staging tile in
// shared memory, from where they are stored; the short-term phase then starts both accumulators
// afresh.  At its end the staged rows are read back for the gate mix (Eq. 19) and replaced by the
// short-term rows; the mix goes over the tile's queries, which no product reads any more (the next
// tile's lie in a second buffer).  Whole-line TMA stores; lse directly.  Every wait is bounded
// (tc_common.cuh); the softmax warps, which meet at named barriers, agree on every tile they start.
#include "tc_common.cuh"

#include <cfloat>

namespace blossom {
namespace tc {
namespace {

constexpr float kRescaleThreshold = 8.0f;  // log2 units
constexpr int kFwdThreads = 384;  // warps 0..7 softmax; 8 loader, 9 issuer of the products, 11 storer
constexpr int kSoftmaxWarps = 8;
// The kernel is compiled for 80 registers per thread (two CTAs of 384 threads per SM): the pool of
// a CTA is 384 * 80 = 30720, and the two register counts must fit in it or the increase would
// wait for registers that never come: 256 * 96 + 128 * 40 = 29696.
constexpr int kProducerRegs = 40, kSoftmaxRegs = 96;
static_assert(256 * kSoftmaxRegs + 128 * kProducerRegs <= kFwdThreads * 80, "register pool of a CTA");
constexpr uint32_t kFwdTmemCols = 256;
__host__ __device__ constexpr int fwd_stages(int D) { return D == 64 ? 3 : 4; }
// Two logits / probability buffers take turns: the next item's and its phase, and those of the item before.  The issuer
// and the softmax warps count for themselves (with the loader's counter for the issuer too: L 4096, B 1, H 8 70.4 -> 71.4 us;
// D 32, L 1024 286 -> 284).
struct Turn {
  int x = 0;
  __device__ __forceinline__ int buffer() const { return x & 1; }
  __device__ __forceinline__ int phase() const { return (x >> 1) & 1; }
  __device__ __forceinline__ int last_buffer() const { return (x - 1) & 1; }
  __device__ __forceinline__ int last_phase() const { return ((x - 1) >> 1) & 1; }
  __device__ __forceinline__ void step() { ++x; }
};

// maximum of 32 logits
__device__ __forceinline__ float half_row_max(const float (&v)[32]) {
  float a[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) a[e] = fmaxf(v[2 * e], v[2 * e + 1]);
#pragma unroll
  for (int c = 8; c < 32; c += 8)
#pragma unroll
    for (int e = 0; e < 4; ++e) a[e] = max3(a[e], v[c + 2 * e], v[c + 2 * e + 1]);
  return fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3]));
}

// probabilities of 32 logits relative to the running maximum (nm = -m, log2 units), packed as
// bf16 pairs; their sum is added to l.  Two logits per FMA / ADD instruction.
__device__ __forceinline__ void half_row_probs(const float (&sv)[32], float sc2, float nm, float &l, uint32_t (&pk)[16]) {
  const float2 sc = make_float2(sc2, sc2), nn = make_float2(nm, nm);
  float2 s0 = make_float2(0.f, 0.f), s1 = make_float2(0.f, 0.f);
#pragma unroll
  for (int c = 0; c < 32; c += 4) {
    const float2 x0 = ffma2(make_float2(sv[c], sv[c + 1]), sc, nn);
    const float2 x1 = ffma2(make_float2(sv[c + 2], sv[c + 3]), sc, nn);
    const float2 e0 = make_float2(exp2f(x0.x), exp2f(x0.y)), e1 = make_float2(exp2f(x1.x), exp2f(x1.y));
    s0 = fadd2(s0, e0);
    s1 = fadd2(s1, e1);
    pk[c >> 1] = pack_bf16(e0.x, e0.y);
    pk[(c >> 1) + 1] = pack_bf16(e1.x, e1.y);
  }
  l += (s0.x + s0.y) + (s1.x + s1.y);
}

// multiply the row's accumulator by fac (all lanes of the warp take part)
template <int D>
__device__ __forceinline__ void rescale_acc(uint32_t taddr, float fac) {
#pragma unroll
  for (int c0 = 0; c0 < D; c0 += 32) {
    float o[32];
    tmem_ld32(taddr + c0, o);
    tmem_wait_ld();
#pragma unroll
    for (int c = 0; c < 32; ++c) o[c] *= fac;
    tmem_st32(taddr + c0, o);
  }
  tmem_wait_st();
}

// 16-byte chunk ch of row r of a staged D-wide bf16 tile (the layout of store_row_chunk)
template <int D>
__device__ __forceinline__ uint4 load_row_chunk(const uint8_t *tile, int r, int ch) {
  if constexpr (D == 64) return *reinterpret_cast<const uint4 *>(tile + r * 128 + ((ch ^ (r & 7)) << 4));
  else return *reinterpret_cast<const uint4 *>(tile + r * 64 + ((ch ^ ((r >> 1) & 3)) << 4));
}

// PLAIN: the causal mask and one selection per query block (the measured path): the other modes'
// tests fold away at compile time.
// PACK: rows 0..63 and 64..127 of the CTA are the same 64 positions of two query heads with a common
// key/value head: by Eq. 12 they selected the same blocks and their windows reach the same tiles,
// so every tile the CTA loads has work for all its rows.
template <int D, bool PLAIN, bool PACK>
__global__ void __launch_bounds__(kFwdThreads, 2) fwd_tc_kernel(
    const __grid_constant__ CUtensorMap tmq, const __grid_constant__ CUtensorMap tmk,
    const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmo,
    const __grid_constant__ CUtensorMap tmol, const __grid_constant__ CUtensorMap tmos,
    const __grid_constant__ CUtensorMap tmk32, const __grid_constant__ CUtensorMap tmv32, Shape s,
    const float *__restrict__ gate, const int32_t *__restrict__ seq_lens,
    const uint8_t *__restrict__ qmeta, int training, float *__restrict__ lse,
    int32_t *__restrict__ status, int32_t *__restrict__ tickets, int nT, int n_tiles, int n_meta, int image_bytes, MetaLayout ml) {
  grid_chain_enter();
  using C = Cfg<D>;
  constexpr int STAGES = fwd_stages(D);
  constexpr int DC = D / 2;  // output columns a softmax thread merges and stages
  extern __shared__ uint8_t smem_raw[];
  // barriers: full[STAGES], empty[STAGES], then by tile res[2], meta[2], roles[2], then staged, stored, then per buffer
  // s_full[2], t_full[group][2], done[2]
  __shared__ __align__(8) uint64_t bars[2 * STAGES + 16];
  __shared__ int softmax_tile, tile_id[2];  // the tile whose lists lie (or are about to) behind meta[.]; -1: no more
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_flag;
  __shared__ float2 stat[2][128];  // (maximum, sum) of each group's half of every row, exchanged at a phase end

  const int tid = threadIdx.x, warp = uniform(tid >> 5), lane = tid & 31;
  const int nST = (s.L + 127) >> 7;
  // long rows first, tile-major: every unit's last tile, then every unit's last but one, ...
  // (PACK: a unit is a pair of heads, a tile 64 positions; h = the pair's first head)
  const int nU = PACK ? s.B * (s.H / 2) : s.B * s.H, nQT = PACK ? nT : nST;
  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t *tiles = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  uint8_t *q_tiles = tiles;                                  // [2]: the tile's queries, then its staged rows of out
  uint8_t *kv_tiles = q_tiles + 2 * C::kBigBytes;            // [stage][K, V]
  uint8_t *sl = kv_tiles + STAGES * 2 * C::kSmallBytes;      // staged rows: the long-term branch, then the short-term one
  uint8_t *metas = sl + C::kBigBytes;                        // [n_meta] the forward's part of an image built by tc_meta_kernel
  const bool causal = PLAIN || s.causal;
  const int pq = PLAIN ? 0 : s.pq;
  const int meta_step = n_meta == 2 ? ml.bytes : 0;
  // tile x of this grid: its rows (tile st of unit u; long rows first, every unit's last tile, then every
  // unit's last but one, ...) and heads
  auto tile_unit = [&](int x) { return x % nU; };
  auto tile_row0 = [&](int x) { return (nQT - 1 - x / nU) * (PACK ? 64 : 128); };
  auto unit_batch = [&](int u) { return PACK ? u / (s.H / 2) : u / s.H; };
  auto unit_head = [&](int u) { return PACK ? 2 * (u % (s.H / 2)) : u % s.H; };
  const uint32_t b_full = smem_u32(&bars[0]), b_empty = smem_u32(&bars[STAGES]);
  const uint32_t b_res = smem_u32(&bars[2 * STAGES]), b_meta = smem_u32(&bars[2 * STAGES + 2]);
  const uint32_t b_roles = smem_u32(&bars[2 * STAGES + 4]);
  const uint32_t b_staged = smem_u32(&bars[2 * STAGES + 6]), b_stored = smem_u32(&bars[2 * STAGES + 7]);
  const uint32_t b_sfull = smem_u32(&bars[2 * STAGES + 8]), b_tfull = b_sfull + 16;  // [group][buffer]
  const uint32_t b_done = b_tfull + 32;
  // one thread: the lists (and which tile's they are) and the queries of this CTA's k-th tile, number x
  auto fetch_meta = [&](int k, int x) {
    tile_id[k & 1] = x;
    const uint32_t bar = b_meta + 8 * (k & 1);
    if (x < 0) {
      mbar_arrive(bar);
    } else {
      mbar_expect_tx(bar, (uint32_t)ml.bytes);
      bulk_load(smem_u32(metas) + (k & 1) * meta_step,
                qmeta + ((size_t)tile_unit(x) * nQT + x / nU) * image_bytes, (uint32_t)ml.bytes, bar);
    }
  };
  auto fetch_queries = [&](int k, int x) {
    const int u = tile_unit(x);
    const uint32_t bar = b_res + 8 * (k & 1);
    mbar_expect_tx(bar, C::kBigBytes);
    tma_load_4d(smem_u32(q_tiles) + (k & 1) * C::kBigBytes, &tmq, bar, 0, tile_row0(x), unit_head(u), unit_batch(u));
  };

  if (tid == 0) {
    abort_flag = (*status != 0) ? 1 : 0;  // an earlier CTA timed out: do not wait again
    tma_prefetch_desc(&tmq);
    tma_prefetch_desc(&tmk);
    tma_prefetch_desc(&tmv);
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(b_full + 8 * i, 1);
      mbar_init(b_empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_res + 8 * i, 1);
      mbar_init(b_meta + 8 * i, 1);
      mbar_init(b_roles + 8 * i, 2);
      mbar_init(b_sfull + 8 * i, 1);
      mbar_init(b_tfull + 8 * i, kSoftmaxWarps / 2);        // group 0
      mbar_init(b_tfull + 8 * (2 + i), kSoftmaxWarps / 2);  // group 1
      mbar_init(b_done + 8 * i, 1);
    }
    mbar_init(b_staged, kSoftmaxWarps);
    mbar_init(b_stored, 1);
    mbar_fence_init();
    fetch_meta(0, (int)blockIdx.x);
    fetch_queries(0, (int)blockIdx.x);
  }
  if (warp == 0) {
    __syncwarp();
    tmem_alloc(smem_u32(&tmem_slot), kFwdTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = (uint32_t)uniform((int)tmem_slot);
  const uint32_t tmem_oa = tmem_base + 128, tmem_ob = tmem_base + 192;  // buffers at tmem_base + 64 * (item % 2)

  if (warp >= kSoftmaxWarps) {
    // ===================== three single-thread roles, one warp each (warp 10 is spare) =====================
    setmaxnreg_dec<kProducerRegs>();
    if (warp == kSoftmaxWarps + 3) {
      // ---- storer: the staged rows of a tile as whole-line bulk stores (rows past L are clipped by the
      // hardware, padded rows were staged as zeros).  When the long-term rows are there it takes the CTA's
      // next tile and fetches that one's lists and queries: late enough for the CTAs that are behind to take
      // fewer tiles (taken a tile earlier, 768 tiles of L 1500: 72 us), early enough for both to be there
      // when the last items are done ----
      if (lane == 0) {
        int cur = (int)blockIdx.x;
        for (int k = 0; cur >= 0 && !*(volatile int *)&abort_flag; ++k) {
          const int u = tile_unit(cur), row0 = tile_row0(cur), h = unit_head(u), n = unit_batch(u);
          mbar_wait(b_staged, 0, &abort_flag, 114);
          if (training) {
            tma_store_4d(&tmol, smem_u32(sl), 0, row0, h, n);
            tma_store_commit();
          }
          int next = (int)gridDim.x + atomicAdd(tickets, 1);
          next = next < n_tiles ? next : -1;
          if (n_meta == 2) fetch_meta(k + 1, next);
          if (next >= 0) fetch_queries(k + 1, next);
          if (training) tma_store_wait_read();
          mbar_arrive(b_stored);
          mbar_wait(b_staged, 1, &abort_flag, 115);
          mbar_wait(b_roles + 8 * (k & 1), (k >> 1) & 1, &abort_flag, 116);  // (of a tile without items nobody else waits for them)
          if (n_meta == 1) fetch_meta(k + 1, next);
          tma_store_4d(&tmo, smem_u32(q_tiles) + (k & 1) * C::kBigBytes, 0, row0, h, n);
          if (training) tma_store_4d(&tmos, smem_u32(sl), 0, row0, h, n);
          tma_store_commit();
          tma_store_wait_read();
          mbar_arrive(b_stored);
          cur = next;
        }
      }
      __syncwarp();
    } else if (warp < kSoftmaxWarps + 2) {
      int it = 0;              // items of the tiles before
      int sj = 0, sph = 0;     // their stage and its phase
      Turn turn;               // (the issuer's)
      auto step = [&] { if (++sj == STAGES) { sj = 0; sph ^= 1; } };
      for (int k = 0;; ++k) {
        mbar_wait(b_meta + 8 * (k & 1), (k >> 1) & 1, &abort_flag, 113);
        const int x = uniform(*(volatile int *)&abort_flag ? -1 : *(volatile int *)&tile_id[k & 1]);
        if (x < 0) break;
        const uint8_t *meta = metas + (k & 1) * meta_step;
        const uint16_t *items = reinterpret_cast<const uint16_t *>(meta + ml.items);  // [2 nT][2]
        const int *counts = reinterpret_cast<const int *>(meta + ml.counts);
        const int nL = uniform(counts[1]), nI = nL + uniform(counts[2]);
        if (warp == kSoftmaxWarps) {
          // ---- loader: K/V tiles, up to STAGES ahead of their consumers ----
          const int u = tile_unit(x), n = unit_batch(u), hk = unit_head(u) / s.G;
          bool go = true;
          for (int j = 0; j < nI; ++j, ++it, step()) {
            const uint32_t pair = reinterpret_cast<const uint32_t *>(items)[j];
            const int row0 = (int)(pair & 0xffffu) * 32, row1 = (int)(pair >> 16) * 32;
            if (it >= STAGES) go = mbar_wait(b_empty + 8 * sj, sph ^ 1, &abort_flag, 105) && go;
            const uint32_t bar = b_full + 8 * sj;
            const uint32_t kt = smem_u32(kv_tiles + sj * 2 * C::kSmallBytes);
            if (elect_one() && go) {
              mbar_expect_tx(bar, 2 * C::kSmallBytes);
              tma_load_halves(kt, C::kSmallBytes / 2, &tmk, &tmk32, bar, row0, row1, hk, n);  // (the key/value head of this query head)
              tma_load_halves(kt + C::kSmallBytes, C::kSmallBytes / 2, &tmv, &tmv32, bar, row0, row1, hk, n);
            }
            __syncwarp();
          }
        } else {
          // ---- S(i) = Q K^T into buffer i % 2; once a group's probabilities of item i are in tensor memory,
          // O_A += P(i)[:, 0:32] V[0:32], O_B += P(i)[:, 32:64] V[32:64], and behind them S(i + 2) into the same
          // buffer, without a wait for the probabilities to have been read (the order assumed in tc_common.cuh) ----
          constexpr uint32_t idesc_s = instr_desc(128, 64, 0, 0), idesc_pv = instr_desc(128, D, 0, 1);
          const uint64_t dq = smem_desc(smem_u32(q_tiles) + (k & 1) * C::kBigBytes, 16, C::kAtomBytes, C::kSwizzle);
          auto logits = [&](int b, int stage, int phase) {
            mbar_wait(b_full + 8 * stage, phase, &abort_flag, 102);
            const uint64_t dk = smem_desc(smem_u32(kv_tiles + stage * 2 * C::kSmallBytes), 16, C::kAtomBytes, C::kSwizzle);
            if (elect_one()) {
#pragma unroll
              for (int c = 0; c < D / 16; ++c) umma_bf16(tmem_base + 64 * b, dq + 2 * c, dk + 2 * c, idesc_s, c > 0);
              umma_commit(b_sfull + 8 * b);
            }
            __syncwarp();
          };
          mbar_wait(b_res + 8 * (k & 1), (k >> 1) & 1, &abort_flag, 101);
          tc_fence_after();
          int ss = sj, sp = sph;  // stage and phase of the next logits
          auto step_s = [&] { if (++ss == STAGES) { ss = 0; sp ^= 1; } };
          Turn ahead = turn;
          for (int i = 0; i < 2 && i < nI; ++i, step_s(), ahead.step()) logits(ahead.buffer(), ss, sp);
          for (int i = 0; i < nI; ++i, step()) {
            const int b = turn.buffer(), ph = turn.phase();
            turn.step();
            const uint64_t dv = smem_desc(smem_u32(kv_tiles + sj * 2 * C::kSmallBytes + C::kSmallBytes),
                                          C::kSmallBytes, C::kAtomBytes, C::kSwizzle);
            const uint32_t tp = tmem_base + 64 * b;
            const uint32_t first = (i == 0 || i == nL) ? 0u : 1u;  // a phase starts the accumulators afresh
            mbar_wait(b_tfull + 8 * b, ph, &abort_flag, 104);
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int c = 0; c < 2; ++c)
                umma_bf16_ts(tmem_oa, tp + 8 * c, dv + c * C::kKStep, idesc_pv, (first | (uint32_t)c) != 0u);
            }
            __syncwarp();
            mbar_wait(b_tfull + 8 * (2 + b), ph, &abort_flag, 109);
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int c = 0; c < 2; ++c)
                umma_bf16_ts(tmem_ob, tp + 32 + 8 * c, dv + (2 + c) * C::kKStep, idesc_pv, (first | (uint32_t)c) != 0u);
              umma_commit(b_done + 8 * b);
              umma_commit(b_empty + 8 * sj);  // S(i) completed before the softmax warps read it
            }
            __syncwarp();
            if (i + 2 < nI) {
              logits(b, ss, sp);
              step_s();
            }
          }
        }
        warp_arrive(b_roles + 8 * (k & 1), lane);  // done with the lists
      }
    }
  } else {
    // ================================ softmax =================================
    setmaxnreg_inc<kSoftmaxRegs>();
    const int quarter = warp & 3, grp = warp >> 2;  // TMEM lane quarter; key half of every tile
    const int r = quarter * 32 + lane, g = r / s.Bk;
    const uint32_t lane_off = (uint32_t)(quarter * 32) << 16;
    const uint32_t acc_own = (grp ? tmem_ob : tmem_oa) + lane_off;
    // (not zero, which a scale among the denormals is flushed to: a hidden logit, -infinity, times it has to stay so)
    const float sc2 = fmaxf(s.scale * kLog2e, FLT_MIN);
    Turn turn;
    for (int k = 0;; ++k) {
      if (warp == 0) {  // one warp decides for all: the named barriers below need every one of them
        mbar_wait(b_meta + 8 * (k & 1), (k >> 1) & 1, &abort_flag, 117);
        if (lane == 0) softmax_tile = *(volatile int *)&abort_flag ? -1 : *(volatile int *)&tile_id[k & 1];
      }
      named_bar_sync(2, kSoftmaxWarps * 32);
      const int x = uniform(*(volatile int *)&softmax_tile);
      if (x < 0) break;
      mbar_wait(b_meta + 8 * (k & 1), (k >> 1) & 1, &abort_flag, 120);  // (complete: makes the lists visible to this warp)
      const uint8_t *meta = metas + (k & 1) * meta_step;
      const uint8_t *selb = meta + ml.sel;
      const uint8_t *rowb = meta + ml.rows;  // (selection per query position) [128 rows][nT]
      const uint16_t *items = reinterpret_cast<const uint16_t *>(meta + ml.items);  // [2 nT][2]
      const uint8_t *icls = meta + ml.icls;                                         // [2 nT][4]
      const int *counts = reinterpret_cast<const int *>(meta + ml.counts);
      const int nL = uniform(counts[1]), nI = nL + uniform(counts[2]);
      const int u = tile_unit(x), n = unit_batch(u);
      const int pad0 = s.L - min(max(seq_lens ? seq_lens[n] : s.L, 0), s.L);
      const int t = tile_row0(x) + (PACK ? r & 63 : r);
      const int hr = unit_head(u) + (PACK ? r >> 6 : 0);  // this row's head
      const bool row_ok = t < s.L;
      // the last key this row may see (a padded row sees nothing; under the causal mask its keys lie behind t)
      const int t_last = row_ok && (causal || t >= pad0) ? (causal ? t : s.L - 1) : -1;
      float m = -INFINITY, l = 0.f;  // this group's running maximum (log2 units) and sum of the row
      const float alpha = gate_alpha(gate, hr), beta = 1.f - alpha;
      int hx_n = nI > 0 ? items[grp] : 0, cls_n = nI > 0 ? icls[quarter] : 0;
      uint8_t *so = q_tiles + (k & 1) * C::kBigBytes;  // the gate mix is staged over the queries, free by then

      // End of a phase: the two groups' halves of every row are merged (maxima, sums, accumulators),
      // normalised, and this thread's DC columns are staged: the long-term rows into sl; at the end of the
      // short-term phase, which finds the long-term rows there, its rows into sl and the gate mix (Eq. 19)
      // into so.  The caller has waited for the phase's last products and for sl to be free.
      auto merge = [&](bool final_phase) {
        stat[grp][r] = make_float2(m, l);
        named_bar_sync(1, kSoftmaxWarps * 32);
        const float2 oth = stat[grp ^ 1][r];
        const float mt = fmaxf(m, oth.x);
        const float fo = l > 0.f ? exp2f(m - mt) : 0.f, fp = oth.y > 0.f ? exp2f(oth.x - mt) : 0.f;
        const float lt = l * fo + oth.y * fp;
        const float inv = (lt > 0.f && row_ok && t >= pad0) ? 1.f / lt : 0.f;
        const float fa = (grp ? fp : fo) * inv, fb = (grp ? fo : fp) * inv;
        if (grp == 0 && row_ok && lse)
          lse[((int64_t)((final_phase ? s.B : 0) + n) * s.H + hr) * s.L + t] = lt > 0.f ? (mt + log2f(lt)) * kLn2 : 0.f;
#pragma unroll
        for (int c0 = 0; c0 < DC; c0 += 16) {
          float a[16], b[16];
          tmem_ld16(tmem_oa + lane_off + DC * grp + c0, a);
          tmem_ld16(tmem_ob + lane_off + DC * grp + c0, b);
          tmem_wait_ld();
#pragma unroll
          for (int ch = 0; ch < 2; ++ch) {
            const int chunk = (DC * grp + c0) / 8 + ch;
            float o[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) o[e] = inv > 0.f ? a[ch * 8 + e] * fa + b[ch * 8 + e] * fb : 0.f;
            if (final_phase) {
              const uint4 w = load_row_chunk<D>(sl, r, chunk);
              const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
              uint32_t wo[4];
#pragma unroll
              for (int e = 0; e < 4; ++e)
                wo[e] = pack_bf16(alpha * __uint_as_float(ww[e] << 16) + beta * o[2 * e],
                                  alpha * __uint_as_float(ww[e] & 0xffff0000u) + beta * o[2 * e + 1]);
              store_row_chunk<D>(so, r, chunk, make_uint4(wo[0], wo[1], wo[2], wo[3]));
            }
            store_row_chunk<D>(sl, r, chunk, make_uint4(pack_bf16(o[0], o[1]), pack_bf16(o[2], o[3]),
                                                         pack_bf16(o[4], o[5]), pack_bf16(o[6], o[7])));
          }
        }
        fence_async_smem();
        tc_fence_before();
        warp_arrive(b_staged, lane);
        // Both groups read both accumulators above, and the first product of the next phase (or tile)
        // overwrites an accumulator as soon as ITS group has stored the next probabilities: no warp may go
        // on before every warp has read.
        named_bar_sync(3, kSoftmaxWarps * 32);
        m = -INFINITY;
        l = 0.f;
      };
      // the products of the item before (of either phase) have completed
      // (A parity only tells a barrier's last two phases apart.  The one before, of the item two earlier, has passed: this warp
      // has seen the logits of the item before, which were issued behind those products and are taken to be reported behind them.)
      auto products_done = [&](int site) {
        mbar_wait(b_done + 8 * turn.last_buffer(), turn.last_phase(), &abort_flag, site);
        __syncwarp();
        tc_fence_after();
      };
      int i = 0;
#pragma unroll 1
      for (int phase = 0; phase < 2; ++phase) {  // the long-term items, the short-term items
        const int phase_end = phase ? nI : nL;
        const bool isL = phase == 0;
#pragma unroll 1
        for (; i < phase_end; ++i) {
          const int hx = hx_n, cls = (cls_n >> (2 * grp)) & 3;  // this group's half, 32 keys from 32 hx
          if (i + 1 < nI) {  // the next item's half and class, ahead of their use
            hx_n = items[2 * (i + 1) + grp];
            cls_n = icls[(i + 1) * 4 + quarter];
          }
          uint32_t hm = 0u;  // this thread's 32 keys of the tile that the row sees
          bool doB = cls == 1;
          if (cls == 2) {
            const int c0 = 32 * hx, jt = hx >> 1, col = 32 * (hx & 1);
            hm = cols32_le(t_last - c0) & cols32_ge(pad0 - c0);
            if (isL) hm &= expand_block_bits32(pq ? rowb[r * nT + jt] : selb[g * nT + jt], s.Bk, col);
            else hm &= s.stis_mode ? (uint32_t)(st_key_cols(s, t, jt * 64, causal) >> col) : st_window32(s, t, c0, causal);
            doB = __any_sync(0xffffffffu, hm != 0u);
          }
          const int b = turn.buffer();
          const uint32_t t_b = tmem_base + 64 * b + lane_off + 32 * grp;

          mbar_wait(b_sfull + 8 * b, turn.phase(), &abort_flag, 107);
          __syncwarp();
          tc_fence_after();
          uint32_t pk[16];
          if (doB) {
            float sv[32];
            tmem_ld32(t_b, sv);
            tmem_wait_ld();
            float fac = 1.f;
            if (cls == 2)  // (one code behind it for all items: the instructions have to be fetched, and that is felt)
#pragma unroll
              for (int c = 0; c < 32; ++c) sv[c] = (hm >> c) & 1u ? sv[c] : -INFINITY;
            const float mt = half_row_max(sv) * sc2;
            const bool need = mt > m + kRescaleThreshold;  // also true on the row's first keys, before which
            const bool scale_acc = need && l > 0.f;        // the accumulator holds sums of zero probabilities
            if (need) {
              fac = exp2f(m - mt);
              l *= fac;
              m = mt;
            }
            half_row_probs(sv, sc2, m == -INFINITY ? 0.f : -m, l, pk);  // (no key yet: all logits are -infinity)
            if (__any_sync(0xffffffffu, scale_acc)) {  // rescaling needs the products of item i-1
              products_done(108);
              rescale_acc<D>(acc_own, fac);
            }
          } else {
#pragma unroll
            for (int c = 0; c < 16; ++c) pk[c] = 0u;
          }
          tmem_st16u(t_b, pk);  // the probabilities replace this thread's logits
          tmem_wait_st();
          tc_fence_before();
          warp_arrive(b_tfull + 8 * (2 * grp + b), lane);  // the stores have completed (wait::st)
          turn.step();
        }

        if (phase_end > (phase ? nL : 0)) products_done(110 + phase);
        if (phase && nI == 0) mbar_wait(b_res + 8 * (k & 1), (k >> 1) & 1, &abort_flag, 112);  // (nothing else waited for the queries)
        // sl: the tile before has been stored (at once for the first); the long-term rows have been stored
        mbar_wait(b_stored, phase ^ 1, &abort_flag, 118 + phase);
        merge(phase == 1);
      }
    }
  }
  finish(warp, tmem_base, kFwdTmemCols, &abort_flag, status);
}

}  // namespace

template <int D>
int launch_fwd_tc_t(const Shape &s, const void *q, const void *k, const void *v, const float *gate,
                    const int32_t *seq_lens, const int32_t *idx, void *out, void *out_lt,
                    void *out_st, float *lse, const Workspace &ws, cudaStream_t st) {
  using C = Cfg<D>;
  CUtensorMap tq, tk, tv, to, tol, tos, tk32, tv32;
  const int training = out_lt != nullptr;
  // (head-packed: a query-side box is 64 positions of two heads)
  const int qrows = s.pack ? 64 : 128, qheads = s.pack ? 2 : 1;
  if (make_tensor_map(&tq, q, s, qrows, false, qheads) || make_tensor_map(&tk, k, s, 64, true) ||
      make_tensor_map(&tv, v, s, 64, true) || make_tensor_map(&tk32, k, s, 32, true) || make_tensor_map(&tv32, v, s, 32, true) || make_tensor_map(&to, out, s, qrows, false, qheads) ||
      make_tensor_map(&tol, training ? out_lt : out, s, qrows, false, qheads) ||
      make_tensor_map(&tos, training ? out_st : out, s, qrows, false, qheads))
    return BLOSSOM_ERR_CUDA;
  const int nT = (s.L + 63) / 64, nST = (s.L + 127) / 128;
  // Two CTAs share an SM (228 KB with 1 KB for each and its static part): a second buffer for the lists as long
  // as that stays so.
  // (The offsets go to the kernel as an argument: computed there they take registers of the softmax loop: 317 us instead of
  // 308 at B 16, H 8, L 4096, D 64.)
  const MetaLayout ml = meta_layout(nT, s.pq, false);
  const size_t tiles = 1024 + 3 * C::kBigBytes + fwd_stages(D) * 2 * C::kSmallBytes, list = ml.bytes,
               image = meta_layout(nT, s.pq).bytes;  // (of which the kernel reads the end)
  const size_t kPair = 110 * 1024;
  const int n_meta = tiles + 2 * list <= kPair ? 2 : 1;
  const size_t smem = tiles + n_meta * list;
  const bool plain = s.causal && !s.pq;
  auto kern = s.pack ? (plain ? fwd_tc_kernel<D, true, true> : fwd_tc_kernel<D, false, true>)
                     : (plain ? fwd_tc_kernel<D, true, false> : fwd_tc_kernel<D, false, false>);
  if (!allow_smem(kern, smem)) return BLOSSOM_ERR_CUDA;
  const int n_tiles = s.pack ? nT * (s.B * (s.H / 2)) : nST * (s.B * s.H);
  const int resident = 148 * (smem <= kPair ? 2 : 1);
  const unsigned grid = (unsigned)(n_tiles < resident ? n_tiles : resident);
  // A training call also builds the backward's tile lists (the same launch):
  // a backward call told to reuse them (blossom_params::reuse_tile_lists) then builds none.  (The backward of an
  // input-dependent gate takes lists of one branch at a time: it builds its own.)
  if (int rc = launch_tc_meta(s, seq_lens, idx, ws.qmeta, training && !s.gate_mode ? ws.kmeta : nullptr, st, ws.status + kTicketWord, 3, 1)) return rc;
  {
    LaunchScope ls(K_FWD_TC, st);
    launch_chained(kern, dim3(grid), dim3(kFwdThreads), smem, st, tq, tk, tv, to, tol, tos, tk32, tv32, s, gate, seq_lens,
                   (const uint8_t *)ws.qmeta + (image - list), training, lse, ws.status, ws.status + kTicketWord, nT, n_tiles, n_meta,
                   (int)image, ml);
  }
  return cudaGetLastError() == cudaSuccess ? BLOSSOM_OK : BLOSSOM_ERR_CUDA;
}

template int launch_fwd_tc_t<32>(const Shape &, const void *, const void *, const void *, const float *,
                                 const int32_t *, const int32_t *, void *, void *, void *, float *,
                                 const Workspace &, cudaStream_t);
template int launch_fwd_tc_t<64>(const Shape &, const void *, const void *, const void *, const float *,
                                 const int32_t *, const int32_t *, void *, void *, void *, float *,
                                 const Workspace &, cudaStream_t);

}  // namespace tc
}  // namespace blossom
