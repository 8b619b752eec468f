// Tile bookkeeping of the tensor-core attention kernels, built once per call.
//
// Which half tiles of 32 keys a 128-row query tile has to visit (the blocks its query blocks selected,
// Eq. 13, and what its window reaches, Eq. 15), in which order, two at a time, and which of its warps they
// concern, depends only on the block indices and the sequence lengths.  Building that inside the
// attention kernels cost every CTA several thousand cycles before its first product; here a warp
// (or four, see the kernel) per attention CTA builds the image of the bookkeeping the attention kernel wants in shared
// memory, and the attention kernel fetches it with one bulk copy while its first tiles load.
//
// Query-major image (forward and dQ kernel), see meta_layout():
//   list[2 nT], flags[2 nT]   (dQ) the halves any row of the CTA needs; bit 0: some selected
//                             block lies in the half, bit 1: the window of some row reaches it
//   jcls[nT][2][8]            (dQ) class of every (listed pair, half of it, compute warp)
//   [8][nT] selection bytes   bit c of byte (g, jt): query block g of the CTA selected key block
//                             jt * (64 / Bk) + c
//   counts                    {pairs on the list, long-term items, short-term items}
//   items[2 nT][2], icls[2 nT][4] (forward) the long-term halves, then the short-term halves, two an item, and the
//                             classes of every (item, row quarter), two bits per half
// The attention kernels work on 64 columns at a time, 32 for each group of their compute warps: any two halves
// make such a pair (an odd one out is paired with the half behind the last, which reads as zeros and has class 0).
// With tiles of 64 adjacent rows, halves of 32 that no row needs were worked through as well: with blocks of 32 and 128 rows
// a CTA 8 % of the items at L 1024 with 8 blocks each, 22 % at L 777 without the causal mask with 6.  us, forward + backward:
// B 128, H 4, L 1024, D 64 677 -> 654; H 2, D 32 293 -> 287; without the mask, B 16, H 4, L 777 117 -> 112.
// Head-packed variant (Shape::pack): the CTA's rows 0..63 and 64..127 are the same 64 positions of
// two query heads with a common key/value head, so both halves have the same selection bytes and
// every listed tile concerns both.
// With a selection per query position the key-major images would each have to scan the index rows
// of every later position; instead the query-major images, which read every index row once, set
// one bit per (key block, position) in a table in global memory (launch 1), and the key-major
// images copy the words of their key blocks from it (launch 2).
// Key-major image (dK/dV kernel): [8][nT] bytes: bit c of byte (g, qt): query block
// qt * (64 / Bk) + c selected key block g of the CTA; list / flags of the halves of 32 queries that
// visit the CTA's keys; jcls[nT][2][8] class of every (listed pair, half of it, compute warp);
// counts {pairs on the list}.
#include "tc_common.cuh"

#include <type_traits>

namespace blossom {
namespace tc {
namespace {

constexpr int kMetaWarps = 4;  // warps per CTA

// NW warps build one image.  One: no block-wide barrier anywhere, so the images of a large launch are in
// flight at once and the issue slots are what counts.  Four: an image's loops are a chain of loads and
// atomics that one warp takes 8 - 25 us for (the selection per position has 128 index rows to go through),
// so a launch of few images is shorter with the loops split.  The compactions stay with the first warp.
// PLAIN: the causal mask, one selection per query block, a window: the other modes' tests fold away, and their code out of
// the instruction cache (22.7 -> 20.7 us for the 8192 images of B 128, H 4, L 1024, 17.0 -> 14.6 at H 2, 33.2 -> 29.5 at B 16, H 8, L 4096).
// WHOLE (blocks of 64): a block is needed whole, so the lists' unit is a tile, i.e. its two halves in one word: half as much to
// list, class and order, and both halves of every pair adjacent.  us with lists of halves -> of tiles, H 8, D 64, 16 blocks:
// forward at B 1, L 4096 70.2 -> 69.1; forward + backward at B 16, L 4096 1254 -> 1248, at B 1, L 10240 461 -> 457.
template <int NW, bool PLAIN, bool WHOLE>
__global__ void __launch_bounds__(kMetaWarps * 32) tc_meta_kernel(Shape s, const int32_t *__restrict__ seq_lens,
                                                                  const int32_t *__restrict__ idx,
                                                                  uint8_t *__restrict__ qmeta,
                                                                  uint8_t *__restrict__ kmeta, int nT,
                                                                  int n_query_ctas, int image0, int image_end,
                                                                  int branches, int with_fwd,
                                                                  uint32_t *__restrict__ inv_bits,
                                                                  int32_t *__restrict__ tickets,
                                                                  uint8_t *qmeta2, uint8_t *kmeta2, int release_late,
                                                                  const MetaLayout ml) {
  if (!release_late) grid_release();
  grid_wait();
  if (release_late) grid_release();
  if (blockIdx.x == 0 && threadIdx.x == 0) *tickets = 0;  // of the persistent kernel behind
  constexpr int NT = 32 * NW;  // threads per image
  const bool causal = PLAIN || s.causal;
  const int pq = PLAIN ? 0 : s.pq;
  // may a query of [t0, t1] see a key of [p0, p1] through the short-term branch?
  auto touch = [&](int t0, int t1, int p0, int p1) { return PLAIN ? t0 - p1 < s.window : st_ranges_touch(s, t0, t1, p0, p1); };
  auto sync = [] {
    if (NW == 1) __syncwarp();
    else __syncthreads();
  };
  extern __shared__ __align__(16) uint8_t meta_all[];
  const int lane = threadIdx.x & 31, tid = threadIdx.x % NT, sub = threadIdx.x / NT;
  const bool scans = tid < 32;  // the warp that compacts
  int image = image0 + (int)blockIdx.x * (kMetaWarps / NW) + sub;  // this launch builds [image0, image_end)
  if (image >= image_end) return;
  if (qmeta2) {  // one set of images per branch
    branches = image < image_end / 2 ? 1 : 2;
    if (branches == 2) image -= image_end / 2, qmeta = qmeta2, kmeta = kmeta2;
  }
  const int Lw = (s.L + 31) >> 5;  // words per key block of the bit table
  uint8_t *meta = meta_all + (size_t)sub * ml.bytes;
  const int nST = (s.L + 127) >> 7;
  const bool key_major = image >= n_query_ctas;
  const int cta = key_major ? image - n_query_ctas : image;
  // query-major CTAs count (batch, query head) pairs, key-major CTAs (batch, key/value head) pairs;
  // uk = the (batch, key/value head) pair whose selection the image is built from
  // (head-packed query-major CTAs count (batch, pair of query heads) pairs, one CTA per 64 positions)
  const bool pack = !key_major && s.pack;
  const int u = pack ? cta / nT : cta / nST;
  const int n = key_major ? u / s.Hkv : (pack ? u / (s.H / 2) : u / s.H);
  const int uk = key_major ? u : n * s.Hkv + (pack ? 2 * (u % (s.H / 2)) : u % s.H) / s.G;
  int len = seq_lens ? seq_lens[n] : s.L;
  len = min(max(len, 0), s.L);
  const int pad0 = s.L - len;
  uint32_t *selw = reinterpret_cast<uint32_t *>(meta + ml.sel);
  uint8_t *selb = meta + ml.sel;
  constexpr int PER = WHOLE ? 1 : 2;  // entries of a list, or of the items, in a pair of halves
  using Entry = std::conditional_t<WHOLE, uint32_t, uint16_t>;
  using Flag = std::conditional_t<WHOLE, uint16_t, uint8_t>;
  auto entry = [](int hx) { return (Entry)(WHOLE ? hx | (hx + 1) << 16 : hx); };
  Entry *list = reinterpret_cast<Entry *>(meta + ml.list), *items = reinterpret_cast<Entry *>(meta + ml.items);
  Flag *lflags = reinterpret_cast<Flag *>(meta + ml.flags);
  const uint16_t *list_half = reinterpret_cast<const uint16_t *>(list), *item_half = reinterpret_cast<const uint16_t *>(items);
  const uint8_t *flags_half = meta + ml.flags;
  uint8_t *icls = meta + ml.icls;
  uint8_t *jcls = meta + ml.jcls;
  int *counts = reinterpret_cast<int *>(meta + ml.counts);
  const unsigned lt = (1u << lane) - 1u;
  const int bk_shift = WHOLE ? 6 : __ffs(s.Bk) - 1, nb_shift = 6 - bk_shift;  // Bk is a power of two
  const int G = 128 >> bk_shift, nb = 1 << nb_shift;  // query blocks of a CTA, blocks of a tile
  // index rows: entry i of a run is slot i % topk of row i / topk; a thread's next entry lies NT further
  const int step_row = NT / s.topk, step_slot = NT % s.topk;
  auto next_entry = [&](int &row, int &slot) {
    row += step_row;
    slot += step_slot;
    if (slot >= s.topk) slot -= s.topk, ++row;
  };
  const int row_0 = tid / s.topk, slot_0 = tid % s.topk;

  // place of the k-th of n entries of one kind among those of both kinds: a pair of the first, a pair of the second, and so
  // on while there are pairs of both, then what is left
  auto alternate = [](int k, int second, int n, int other) {
    const int m = min(n, other) / PER * PER;
    if (k < m) return 2 * (k / PER * PER) + k % PER + PER * second;
    return second ? k + other : k + m;
  };
  // one warp: the list of n entries becomes one of pairs
  auto pad_list = [&](int n) {
    if (lane == 0) {
      if (n % PER) {
        list[n] = (Entry)(2 * nT);
        lflags[n] = 0;
      }
      counts[0] = (n + PER - 1) / PER;
    }
  };
  // One warp: the halves hx_min ... hx_max (or their tiles) that the CTA's rows (or keys) lo ... hi need, ascending, a lane
  // per tile of two.
  // selected(jt, first, second): bits of tile jt's selections by the first and by the other 64 rows.  In a query-major
  // image the flags also hold which of the two 64-row halves need it, through the long-term branch (bits 2, 3) and at all
  // (bits 4, 5, of a backward's image); n_long, n_all count them by that class.
  auto half_row0 = [&](int row0, int hf) { return pack ? row0 : row0 + 64 * hf; };
  int n_long[4] = {0, 0, 0, 0}, n_all[4] = {0, 0, 0, 0};
  auto list_halves = [&](int hx_min, int hx_max, bool live, int lo, int hi, auto by_key, auto selected) {
    constexpr bool KEYS = decltype(by_key)::value;
    int nv = 0;
    uint32_t one_long = 0u, both_long = 0u, one_all = 0u;  // this lane's counts of classes 1 and 2 (low, high half), of class 3
    for (int base = hx_min >> 1; live && base <= hx_max >> 1; base += 32) {
      const int jt = base + lane;
      uint32_t first[2] = {0u, 0u}, second[2] = {0u, 0u};
      if (jt <= hx_max >> 1) selected(jt, first, second);
      int f[2] = {0, 0};
#pragma unroll
      for (int x = 0; x < PER; ++x) {
        const int hx = 2 * jt + x, p0 = hx * 32, p1 = p0 + 64 / PER - 1;
        if (hx >= hx_min && hx <= hx_max && p1 >= pad0) {
          if (KEYS ? touch(p0, min(p1, s.L - 1), lo, hi) : touch(lo, hi, p0, p1)) f[x] = 2;
          int c = ((WHOLE ? first[0] | first[1] : first[x]) ? 1 : 0) | ((WHOLE ? second[0] | second[1] : second[x]) ? 2 : 0);
          f[x] = (f[x] | (c ? 1 : 0)) & branches;
          if (!KEYS) {
            if (!(f[x] & 1)) c = 0;
            f[x] |= c << 2;
            if ((f[x] & 2) && kmeta)
              for (int hf = 0; hf < 2; ++hf)
                if ((p0 <= half_row0(lo, hf) + 63 || !causal) && touch(half_row0(lo, hf), half_row0(lo, hf) + 63, p0, p1)) c |= 1 << hf;
            if (f[x] && kmeta) f[x] |= (c ? c : 3) << 4;
          }
        }
        if (!KEYS) {
          const int cl = (f[x] >> 2) & 3, ca = f[x] >> 4;
          one_long += cl == 1 ? 1u : cl == 2 ? 0x10000u : 0u;
          both_long += cl == 3 ? 1u : 0u;
          one_all += ca == 1 ? 1u : ca == 2 ? 0x10000u : 0u;
        }
      }
      const unsigned b0 = __ballot_sync(0xffffffffu, f[0] != 0), b1 = WHOLE ? 0u : __ballot_sync(0xffffffffu, f[1] != 0);
      int pos = nv + __popc(b0 & lt) + __popc(b1 & lt);
#pragma unroll
      for (int x = 0; x < 2; ++x)
        if (f[x]) {
          list[pos] = entry(2 * jt + x);
          lflags[pos++] = (Flag)(WHOLE ? f[x] * 0x101 : f[x]);
        }
      nv += __popc(b0) + __popc(b1);
    }
    if (!KEYS) {
      one_long = __reduce_add_sync(0xffffffffu, one_long);
      n_long[1] = (int)(one_long & 0xffffu);
      n_long[2] = (int)(one_long >> 16);
      n_long[3] = (int)__reduce_add_sync(0xffffffffu, both_long);
      one_all = __reduce_add_sync(0xffffffffu, one_all);
      n_all[1] = (int)(one_all & 0xffffu);
      n_all[2] = (int)(one_all >> 16);
      n_all[3] = nv - n_all[1] - n_all[2];
    }
    return nv;
  };
  // One warp: the list's entries in the order both 64-row halves, then alternately a pair of the first and one of the second,
  // by the class in the flags from bit `shift`; place(entry, position) takes them down.
  auto order = [&](int nv, int shift, const int (&n)[4], auto place) {
    int c1 = 0, c2 = 0, c3 = 0;
    for (int base = 0; base < nv; base += 32) {
      const int j = base + lane, c = j < nv ? (lflags[j] >> shift) & 3 : 0;
      const unsigned b1 = __ballot_sync(0xffffffffu, c == 1), b2 = __ballot_sync(0xffffffffu, c == 2), b3 = __ballot_sync(0xffffffffu, c == 3);
      if (c)
        place(j, c == 3 ? c3 + __popc(b3 & lt)
                        : n[3] + (c == 1 ? alternate(c1 + __popc(b1 & lt), 0, n[1], n[2]) : alternate(c2 + __popc(b2 & lt), 1, n[2], n[1])));
      c1 += __popc(b1);
      c2 += __popc(b2);
      c3 += __popc(b3);
    }
  };

  for (int i = ml.sel / 4 + tid; i < ml.bwd / 4; i += NT) reinterpret_cast<uint32_t *>(meta)[i] = 0u;  // what is not written throughout
  sync();

  if (!key_major) {
    const int st = pack ? nT - 1 - cta % nT : nST - 1 - cta % nST;  // the attention kernels take long rows first
    const int row0 = pack ? st * 64 : st * 128, row_last = min(s.L - 1, row0 + (pack ? 63 : 127));
    // first position of the 32 rows of TMEM lane quarter w, and of the 64-row half hf
    auto quarter_row0 = [&](int w) { return row0 + 32 * (pack ? (w & 1) : w); };
    if (pq) {
      // a selection per query position: every row's own bytes, and their union per query block
      // (which is what the tile list and the item order below are built from)
      uint32_t *roww = reinterpret_cast<uint32_t *>(meta + ml.rows);
      // the bit table is per key/value head: the group's first query head (or pair of heads) fills it
      const bool fills = inv_bits && (pack ? (2 * (u % (s.H / 2))) % s.G == 0 : (u % s.H) % s.G == 0);
      for (int r = row_0, slot = slot_0; r < 128; next_entry(r, slot)) {
        const int t = pack ? row0 + (r & 63) : row0 + r;
        if (t < s.L) {
          const int blk = idx[((int64_t)uk * s.L + t) * s.topk + slot];
          if (blk >= 0 && blk <= (t >> bk_shift)) {
            const int a = (r >> bk_shift) * nT + (blk >> nb_shift), b2 = r * nT + (blk >> nb_shift);
            atomicOr(&selw[a >> 2], (1u << (blk & (nb - 1))) << ((a & 3) * 8));
            atomicOr(&roww[b2 >> 2], (1u << (blk & (nb - 1))) << ((b2 & 3) * 8));
            if (fills && (!pack || r < 64))
              atomicOr(&inv_bits[((int64_t)uk * s.M + blk) * Lw + (t >> 5)], 1u << (t & 31));
          }
        }
      }
    } else {
    for (int g = row_0, slot = slot_0; g < G; next_entry(g, slot)) {  // the selections of the CTA's query blocks
      const int qb = pack ? st * nb + (g & (nb - 1)) : st * G + g;
      if (qb < s.M) {
        const int blk = idx[((int64_t)uk * s.M + qb) * s.topk + slot];
        if (blk >= 0 && blk < s.M && (blk <= qb || !causal)) {
          const int a = g * nT + (blk >> nb_shift);
          atomicOr(&selw[a >> 2], (1u << (blk & (nb - 1))) << ((a & 3) * 8));
        }
      }
    }
    }
    sync();
    if (scans) {  // the halves any row of the CTA needs, ascending
      const int nv = list_halves(0, (causal ? row_last : s.L - 1) >> 5, row_last >= pad0, row0, row_last, std::false_type(),
                                 [&](int jt, uint32_t (&first)[2], uint32_t (&second)[2]) {
        for (int g = 0; g < G / 2; ++g) {
          first[0] |= selb[g * nT + jt];
          second[0] |= selb[(g + G / 2) * nT + jt];
        }
        first[1] = first[0] & half_bits(1, bk_shift);
        first[0] &= half_bits(0, bk_shift);
        second[1] = second[0] & half_bits(1, bk_shift);
        second[0] &= half_bits(0, bk_shift);
      });
      if (lane == 0) counts[0] = nv;
    }
    sync();
    const int nv = counts[0];
    if (with_fwd) {
    if (scans) {  // ---- the forward's items and their classes ----
    // Long-term items: the halves that rows of both 64-row halves of the CTA need, then alternately a pair that only
    // rows 0..63 need and a pair that only rows 64..127 need.  A softmax warp may run ahead of the
    // slowest one, so with alternating items both pairs of warps have work at once.
    order(nv, 2, n_long, [&](int j, int pos) { items[pos] = list[j]; });
    const int n_lt = n_long[1] + n_long[2] + n_long[3], nl = (n_lt + PER - 1) / PER * PER;
    if (lane == 0 && nl > n_lt) items[nl - 1] = (Entry)(2 * nT);
    int count = nl;
    for (int base = 0; base < nv; base += 32) {  // short-term items in ascending order
      const int j = base + lane;
      const bool on = j < nv && (lflags[j] & 2);
      const unsigned bal = __ballot_sync(0xffffffffu, on);
      if (on) items[count + __popc(bal & lt)] = list[j];
      count += __popc(bal);
    }
    if (lane == 0) {
      if (count % PER) items[count++] = (Entry)(2 * nT);
      counts[1] = nl / PER;
      counts[2] = (count - nl) / PER;
    }
    }
    sync();
    const int nl = counts[1], count = nl + counts[2];
    // Class of every (item, row quarter, key half), two bits each in a byte per (item, quarter): 0 = no row of the
    // quarter needs the 32 keys, 1 = every row sees all of them, 2 = mixed (the warp builds per-lane column masks).
    const bool uni = s.Bk >= 32;  // a quarter's 32 rows share one query block
    for (int e = tid; e < count * 4; e += NT) {
      const int it = e >> 2, w = e & 3;
      const int t_lo = quarter_row0(w), t_hi = t_lo + 31;
      const bool rows = t_hi >= pad0 && t_lo < s.L, rows_in = t_lo >= pad0 && t_hi < s.L;
      int cls = 0;
#pragma unroll 1
      for (int hf = 0; hf < 2; ++hf) {
        const int hx = item_half[2 * it + hf], k_lo = hx * 32, k_hi = k_lo + 31;
        int c = 0;
        if (rows && (k_lo <= t_hi || !causal) && k_hi >= pad0 && k_lo < s.L) {
          // every row of the quarter may see every key of the half as far as validity and causality go
          const bool inner = rows_in && k_lo >= pad0 && (causal ? k_hi <= t_lo : k_hi < s.L);
          if (it < nl) {
            if (!uni) c = 2;
            else if (selb[((w * 32) >> bk_shift) * nT + (hx >> 1)] & half_bits(hx, bk_shift)) c = !pq && inner ? 1 : 2;  // (per position: the rows differ)
          } else if (touch(t_lo, t_hi, k_lo, k_hi)) {
            c = (inner && k_lo >= t_hi - s.window + 1 && (causal || k_hi <= t_lo + s.window - 1)) ? 1 : 2;  // 1: inside every row's window
          }
        }
        cls |= c << (2 * hf);
      }
      icls[e] = (uint8_t)cls;
    }
    }  // the forward's part
    sync();
    // The dQ kernel walks `list` itself (a half serves both branches there).  Same idea as above:
    // what both 64-row halves need first, then alternately a pair that only rows 0..63 need and one
    // only rows 64..127 need, so that the two halves' warps work on neighbouring pairs at once.
    // (Backward call only; the forward reads `items`.)
    if (kmeta && scans) {
      Entry *tlist = reinterpret_cast<Entry *>(jcls);  // (the classes come later)
      Flag *tflags = reinterpret_cast<Flag *>(jcls + 4 * nT);
      order(nv, 4, n_all, [&](int j, int pos) {
        tlist[pos] = list[j];
        tflags[pos] = lflags[j];
      });
      __syncwarp();
      for (int j = lane; j < nv; j += 32) {
        list[j] = tlist[j];
        lflags[j] = tflags[j];
      }
    }
    if (scans) pad_list(nv);
    sync();
    // dQ kernel: class of every (listed pair, half of 32 keys, compute warp).  Warp w works
    // on rows 32 (w % 4) ... and keys 16 (w / 4) ... of the half.  Bit 0 / bit 1: every row of
    // the warp sees all 16 keys through the long-term / short-term branch and no row sees only a
    // part of them; 8: mixed, the warp builds per-lane column masks.  (A forward-only call has no
    // use for them.)
    for (int e = tid; e < (kmeta ? (nv + PER - 1) / PER * 16 : 0); e += NT) {
      const int j = e >> 3, w = e & 7, qtr = w & 3, c = w >> 2;
      const int hx = list_half[j], f = flags_half[j], jt = hx >> 1;
      const int k_lo = hx * 32 + 16 * c, k_hi = k_lo + 15, t_lo = quarter_row0(qtr), t_hi = t_lo + 31;
      const bool rows_in = t_lo >= pad0 && t_hi < s.L, rows_none = t_hi < pad0 || t_lo >= s.L;
      const bool past = rows_in && k_lo >= pad0 && (causal ? k_hi <= t_lo : k_hi < s.L);  // every key visible to every row (validity, causality)
      const bool reach = !rows_none && (k_lo <= t_hi || !causal) && k_hi >= pad0 && k_lo < s.L;  // some key may be visible to some row
      int cL = 0, cS = 0;  // 0 none, 1 all, 2 mixed
      if ((f & 1) && reach) {
        const int kb = (32 * (hx & 1) + 16 * c) >> bk_shift;  // key block within the tile
        bool any_sel = false, all_sel = true;
        for (int gq = (qtr * 32) >> bk_shift; gq <= (qtr * 32 + 31) >> bk_shift; ++gq) {
          const bool sel = (selb[gq * nT + jt] >> kb) & 1u;
          any_sel |= sel;
          all_sel &= sel;
        }
        if (any_sel) cL = (all_sel && past && !pq) ? 1 : 2;
      }
      if ((f & 2) && reach && touch(t_lo, t_hi, k_lo, k_hi))
        cS = (past && k_lo >= t_hi - s.window + 1 && (causal || k_hi <= t_lo + s.window - 1)) ? 1 : 2;  // 1: inside every row's window
      jcls[e] = (uint8_t)((cL == 2 || cS == 2) ? 8 : (cL | (cS << 1)));
    }
  } else {
    const int kt = cta % nST;  // the dK/dV kernel takes early keys first
    const int key0 = kt * 128, key_last = min(s.L - 1, key0 + 127);
    if (pq) {
      // a selection per query position: which positions selected each of this CTA's key blocks
      // (one bit per position), and per 64-query tile which query blocks hold such a position
      // (the words of this CTA's key blocks from the bit table the query-major images filled: word w
      // of a block holds positions 32 w ...; a position before the block never selected it)
      uint32_t *invw = reinterpret_cast<uint32_t *>(meta + ml.rows);
      const int qb0 = kt * G, w_lo = key0 >> 5;
      for (int i = tid; i < G * (Lw - w_lo); i += NT) {
        const int g = i / (Lw - w_lo), w = w_lo + i % (Lw - w_lo);
        if (qb0 + g >= s.M) continue;
        const uint32_t bits = inv_bits[((int64_t)uk * s.M + qb0 + g) * Lw + w];
        if (!bits) continue;
        const int a = g * nT + (w >> 1);
        invw[2 * a + (w & 1)] = bits;
        // the 32 positions lie in one query block (Bk >= 32) or in two (Bk = 16)
        uint32_t qbits;
        if (s.Bk >= 32) qbits = 1u << (((w & 1) * 32) >> bk_shift);
        else qbits = (((bits & 0xffffu) ? 1u : 0u) | ((bits >> 16) ? 2u : 0u)) << ((w & 1) * 2);
        atomicOr(&selw[a >> 2], qbits << ((a & 3) * 8));
      }
    } else {  // which query blocks selected each of this CTA's key blocks, per 64-query tile
      // (the index rows of query blocks qb0 .. M-1 are contiguous; eight loads in flight per lane)
      // (without the causal mask every query block may have selected them: the rows start at block 0)
      const int qb0 = kt * G, qb_first = causal ? qb0 : 0, total = (s.M - qb_first) * s.topk;
      const int32_t *rows = idx + ((int64_t)uk * s.M + qb_first) * s.topk;
      int row = row_0, slot = slot_0;
      for (int base = 0; base < total; base += 8 * NT) {
        int blk[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int i = base + e * NT + tid;
          blk[e] = i < total ? rows[i] : -1;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const int qb = qb_first + row;
          next_entry(row, slot);
          if (blk[e] >= qb0 && blk[e] < qb0 + G && (blk[e] <= qb || !causal)) {
            const int a = (blk[e] - qb0) * nT + (qb >> nb_shift);
            atomicOr(&selw[a >> 2], (1u << (qb & (nb - 1))) << ((a & 3) * 8));
          }
        }
      }
    }
    sync();
    if (scans) {
      const int count = list_halves(causal ? key0 >> 5 : 0, (s.L - 1) >> 5, key_last >= pad0, key0, key_last, std::true_type(),
                                    [&](int qt, uint32_t (&sel)[2], uint32_t (&)[2]) {
        for (int g = 0; g < G; ++g) {
          if (pq) {
            const uint32_t *w = reinterpret_cast<const uint32_t *>(meta + ml.rows) + 2 * (g * nT + qt);
            sel[0] |= w[0];
            sel[1] |= w[1];
          } else {
            sel[0] |= selb[g * nT + qt];
          }
        }
        if (!pq) {
          sel[1] = sel[0] & half_bits(1, bk_shift);
          sel[0] &= half_bits(0, bk_shift);
        }
      });
      __syncwarp();
      pad_list(count);
    }
    sync();
    const int count = 2 * counts[0];
    // dK/dV kernel: class of every (listed pair, half of 32 queries, compute warp).  Warp w
    // works on key rows 32 (w % 4) ... of the CTA and on query columns 16 (w / 4) ... of the half.  Same code as for the dQ kernel: bit 0 / bit 1 = every key row of the warp is seen in
    // full by all 16 queries through the long-term / short-term branch and none in part; 8 = mixed.
    for (int e = tid; e < count * 8; e += NT) {
      const int j = e >> 3, w = e & 7, qtr = w & 3, hf = w >> 2;
      const int hx = list_half[j], qt = hx >> 1, f = flags_half[j], c_lo = 32 * (hx & 1) + 16 * hf;
      const int p_lo = key0 + 32 * qtr, p_hi = p_lo + 31, t_lo = qt * 64 + c_lo, t_hi = t_lo + 15;
      const bool rows_in = p_lo >= pad0 && p_hi < s.L, rows_none = p_hi < pad0 || p_lo >= s.L;
      const bool past = rows_in && t_hi < s.L && (causal ? t_lo >= p_hi : t_lo >= pad0);  // every query sees every key (validity, causality)
      const bool reach = !rows_none && (t_hi >= p_lo || !causal) && t_hi >= pad0 && t_lo < s.L;  // some query may see some key
      int cL = 0, cS = 0;  // 0 none, 1 all, 2 mixed
      if ((f & 1) && reach) {
        bool any_sel = false, all_sel = true;
        for (int gk = (qtr * 32) >> bk_shift; gk <= (qtr * 32 + 31) >> bk_shift; ++gk) {
          const uint32_t bits = selb[gk * nT + qt];
          for (int c = c_lo >> bk_shift; c <= (c_lo + 15) >> bk_shift; ++c) {
            const bool sel = (bits >> c) & 1u;
            any_sel |= sel;
            all_sel &= sel;
          }
        }
        if (any_sel) cL = (all_sel && past && !pq) ? 1 : 2;
      }
      if ((f & 2) && reach && touch(t_lo, min(t_hi, s.L - 1), p_lo, min(p_hi, s.L - 1)))
        cS = (past && p_lo >= t_hi - s.window + 1 && (causal || p_hi <= t_lo + s.window - 1)) ? 1 : 2;  // 1: inside every query's window
      jcls[e] = (uint8_t)((cL == 2 || cS == 2) ? 8 : (cL | (cS << 1)));
    }
  }
  sync();
  // the parts that this call's kernels read (see MetaLayout)
  uint4 *dst = reinterpret_cast<uint4 *>(key_major ? kmeta + (size_t)cta * ml.bwd : qmeta + (size_t)cta * ml.bytes);
  const uint4 *src = reinterpret_cast<const uint4 *>(meta);
  const int begin = kmeta ? 0 : ml.sel, end = key_major || !with_fwd ? ml.bwd : ml.bytes;
  for (int i = begin / 16 + tid; i < end / 16; i += NT) dst[i] = src[i];
}

}  // namespace

int launch_tc_meta(const Shape &s, const int32_t *seq_lens, const int32_t *idx, uint8_t *qmeta,
                   uint8_t *kmeta, cudaStream_t st, int32_t *tickets, int branches, int with_fwd, uint8_t *qmeta2,
                   uint8_t *kmeta2, bool release_late) {
  if (with_fwd < 0) with_fwd = kmeta == nullptr;
  if (qmeta2 && s.pq) {  // (a selection per position takes two launches for each set)
    if (int rc = launch_tc_meta(s, seq_lens, idx, qmeta, kmeta, st, tickets, 1, with_fwd)) return rc;
    return launch_tc_meta(s, seq_lens, idx, qmeta2, kmeta2, st, tickets, 2, with_fwd, nullptr, nullptr, release_late);
  }
  const int nT = (s.L + 63) / 64, nST = (s.L + 127) / 128;
  const int nq = s.pack ? nT * s.B * (s.H / 2) : nST * s.B * s.H, n_images = kmeta ? nq + nST * s.B * s.Hkv : nq;
  // Four warps per image while its loops are long (a selection per position) or the images do not fill the SMs.  us with
  // one | four, by the number of images: L 1024, blocks of 32, 1024 12.0 | 10.6, 2048 12.5 | 14.1, 8192 20.7 | 32.5; L 4096,
  // blocks of 64, 1024 14.8 | 11.7, 2048 16.5 | 14.4, 4096 20.0 | 21.6; a selection per position, both launches, L 1500 960
  // 46.6 | 31.4, 3840 54.2 | 54.3, 7680 79 | 86, L 400 1152 31.6 | 25.5, 4608 39.9 | 45.1.
  const bool wide = n_images * (qmeta2 ? 2 : 1) <= 148 * (s.pq ? 48 : 8);
  const int per_cta = wide ? 1 : kMetaWarps;
  // (an argument of the kernel: computed there the offsets cost launches of few images 0.5 to 1.5 of their 9 to 12 us)
  const MetaLayout ml = meta_layout(nT, s.pq);
  const size_t smem = (size_t)per_cta * ml.bytes;
  const bool plain = s.causal && !s.pq && s.stis_mode == 0;
  auto of = [&](auto whole) {
    constexpr bool W = decltype(whole)::value;
    return wide ? (plain ? tc_meta_kernel<kMetaWarps, true, W> : tc_meta_kernel<kMetaWarps, false, W>)
                : (plain ? tc_meta_kernel<1, true, W> : tc_meta_kernel<1, false, W>);
  };
  auto kern = s.Bk == 64 ? of(std::true_type()) : of(std::false_type());
  if (!allow_smem(kern, smem)) return BLOSSOM_ERR_CUDA;
  auto launch = [&](int image0, int image_end, uint32_t *inv_bits) {
    LaunchScope ls(K_TC_META, st);
    launch_chained(kern, dim3((unsigned)((image_end - image0 + per_cta - 1) / per_cta)), dim3(kMetaWarps * 32), smem, st, s,
                   seq_lens, idx, qmeta, kmeta, nT, nq, image0, image_end, branches, with_fwd, inv_bits, tickets, qmeta2,
                   kmeta2, (int)release_late, ml);
  };
  if (s.pq && kmeta) {
    // selection per position: the query-major images fill the bit table, then the key-major ones read it
    uint32_t *inv_bits = reinterpret_cast<uint32_t *>(kmeta + tc_key_meta_bytes(s));
    if (cudaMemsetAsync(inv_bits, 0, tc_inv_bits_bytes(s), st) != cudaSuccess) return BLOSSOM_ERR_CUDA;
    launch(0, nq, inv_bits);
    launch(nq, n_images, inv_bits);
  } else {
    launch(0, n_images * (qmeta2 ? 2 : 1), nullptr);
  }
  return cudaGetLastError() == cudaSuccess ? BLOSSOM_OK : BLOSSOM_ERR_CUDA;
}

}  // namespace tc
}  // namespace blossom
