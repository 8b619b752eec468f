// Building blocks of the short-history kernels: warp-level bf16 matrix products out of swizzled
// shared-memory tiles, chunk masks, row stores.
#pragma once
#include "select_geom.cuh"

namespace blossom {
namespace sh {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// byte offset of 16-byte chunk ch of row r in a [rows][D] bf16 tile: the eight rows of an 8x8 matrix
// land in eight different 16-byte bank groups
template <int D>
__device__ __forceinline__ uint32_t tile_off(int r, int ch) {
  if constexpr (D == 64) return (uint32_t)(r * 128 + ((ch ^ (r & 7)) << 4));
  else return (uint32_t)(r * 64 + ((ch ^ ((r >> 1) & 3)) << 4));
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void stsm4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
               "r"(d) : "memory");
}
// c[16 x 8] += a[16 x 16] b[16 x 8], bf16 inputs, fp32 accumulators
__device__ __forceinline__ void mma16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ uint32_t pack2(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&h);
}
__device__ __forceinline__ float lo_bf(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float hi_bf(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// First operand (16 rows) of a product straight from global memory: rows t0 .. t0 + 15 of a
// [.][D] tensor with row stride `sl`; rows outside [lo, hi) are zeros.  a[k] = the k-th 16 columns.
template <int D>
__device__ __forceinline__ void load_a_rows(const __nv_bfloat16 *base, int64_t sl, int t0, int lo, int hi, int lane,
                                            uint32_t (&a)[D / 16][4]) {
  const int r0 = t0 + (lane >> 2), r1 = r0 + 8, c = (lane & 3) * 2;
  const bool ok0 = r0 >= lo && r0 < hi, ok1 = r1 >= lo && r1 < hi;
  const __nv_bfloat16 *p0 = base + (int64_t)r0 * sl + c, *p1 = base + (int64_t)r1 * sl + c;
#pragma unroll
  for (int k = 0; k < D / 16; ++k) {
    a[k][0] = ok0 ? *reinterpret_cast<const uint32_t *>(p0 + 16 * k) : 0u;
    a[k][1] = ok1 ? *reinterpret_cast<const uint32_t *>(p1 + 16 * k) : 0u;
    a[k][2] = ok0 ? *reinterpret_cast<const uint32_t *>(p0 + 16 * k + 8) : 0u;
    a[k][3] = ok1 ? *reinterpret_cast<const uint32_t *>(p1 + 16 * k + 8) : 0u;
  }
}

// c = a b (no accumulator read)
__device__ __forceinline__ void mma16816_0(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// A lane's row and piece of the 8x8 matrices of a 16-row chunk, as an offset from the chunk's first
// byte.  Chunks start at multiples of 16 rows, so the swizzle depends on the lane alone, and the k-th
// 16 columns are one XOR away (offset ^ 32 k).
//   nt (product over D):         (rows 0-7, columns 0-7), (0-7, 8-15), (8-15, 0-7), (8-15, 8-15)
//   nn (product over the rows):  (rows 0-7, columns 0-7), (8-15, 0-7), (0-7, 8-15), (8-15, 8-15)
template <int D>
__device__ __forceinline__ uint32_t lane_off_nt(int lane) { return tile_off<D>((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1); }
template <int D>
__device__ __forceinline__ uint32_t lane_off_nn(int lane) { return tile_off<D>(lane & 15, lane >> 4); }

// s[16 rows x 16] = A (16 x D) times the 16 rows at `chunk`, transposed; chunk = tile address + row *
// 2 D + lane_off_nt (the tile 128-byte aligned)
template <int D>
__device__ __forceinline__ void product_nt(const uint32_t (&a)[D / 16][4], uint32_t chunk, float (&s)[2][4]) {
#pragma unroll
  for (int k = 0; k < D / 16; ++k) {
    uint32_t b[4];
    ldsm4(chunk ^ (32 * k), b);
    if (k == 0) {
      mma16816_0(s[0], a[0], b[0], b[1]);
      mma16816_0(s[1], a[0], b[2], b[3]);
    } else {
      mma16816(s[0], a[k], b[0], b[1]);
      mma16816(s[1], a[k], b[2], b[3]);
    }
  }
}
// the same added to s
template <int D>
__device__ __forceinline__ void product_nt_add(const uint32_t (&a)[D / 16][4], uint32_t chunk, float (&s)[2][4]) {
#pragma unroll
  for (int k = 0; k < D / 16; ++k) {
    uint32_t b[4];
    ldsm4(chunk ^ (32 * k), b);
    mma16816(s[0], a[k], b[0], b[1]);
    mma16816(s[1], a[k], b[2], b[3]);
  }
}
// the same with every 16 columns' product formed from zero and then added (fewer roundings in a row)
template <int D>
__device__ __forceinline__ void product_nt_steps(const uint32_t (&a)[D / 16][4], uint32_t chunk, float (&s)[2][4]) {
#pragma unroll
  for (int k = 0; k < D / 16; ++k) {
    uint32_t b[4];
    float x[2][4];
    ldsm4(chunk ^ (32 * k), b);
    mma16816_0(x[0], a[k], b[0], b[1]);
    mma16816_0(x[1], a[k], b[2], b[3]);
#pragma unroll
    for (int nt = 0; nt < 2; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) s[nt][e] += x[nt][e];
  }
}
// acc[16 rows x D] += A (16 x 16) times the 16 rows at `chunk` (tile address + row * 2 D + lane_off_nn)
template <int D>
__device__ __forceinline__ void product_nn(const uint32_t (&a)[4], uint32_t chunk, float (&acc)[D / 8][4]) {
#pragma unroll
  for (int n2 = 0; n2 < D / 16; ++n2) {
    uint32_t b[4];
    ldsm4t(chunk ^ (32 * n2), b);
    mma16816(acc[2 * n2], a, b[0], b[1]);
    mma16816(acc[2 * n2 + 1], a, b[2], b[3]);
  }
}
// Probabilities (accumulator layout, 16 x 16) -> first operand of the next product.
__device__ __forceinline__ void to_a(const float (&p)[2][4], uint32_t (&a)[4]) {
  a[0] = pack2(p[0][0], p[0][1]);
  a[1] = pack2(p[0][2], p[0][3]);
  a[2] = pack2(p[1][0], p[1][1]);
  a[3] = pack2(p[1][2], p[1][3]);
}

// Rows t0 .. t0 + 15 of a bf16 tensor from accumulators scaled per row (f0: rows lane / 4, f1: rows
// lane / 4 + 8), through a 16-row staging tile of this warp: whole 16-byte pieces per lane instead
// of 4-byte ones.  Rows outside [0, hi) are not written.
template <int D>
__device__ __forceinline__ void store_rows(__nv_bfloat16 *base, int64_t sl, int t0, int hi, const float (&acc)[D / 8][4],
                                           float f0, float f1, uint8_t *stage, int lane) {
  const uint32_t st = smem_addr(stage);
  const int m = lane >> 3, rr = (lane & 7) + (m & 1) * 8;
  __syncwarp();
#pragma unroll
  for (int nt = 0; nt < D / 8; nt += 2)
    stsm4(st + tile_off<D>(rr, nt + (m >> 1)), pack2(acc[nt][0] * f0, acc[nt][1] * f0), pack2(acc[nt][2] * f1, acc[nt][3] * f1),
          pack2(acc[nt + 1][0] * f0, acc[nt + 1][1] * f0), pack2(acc[nt + 1][2] * f1, acc[nt + 1][3] * f1));
  __syncwarp();
#pragma unroll
  for (int i = 0; i < D / 16; ++i) {
    const int e = i * 32 + lane, r = e / (D / 8), ch = e % (D / 8);
    const uint4 v = *reinterpret_cast<const uint4 *>(stage + tile_off<D>(r, ch));
    if (t0 + r < hi) *reinterpret_cast<uint4 *>(base + (int64_t)(t0 + r) * sl + ch * 8) = v;
  }
}

// Copies rows [lo, hi) (multiples of 16 apart from the ends, which are zero-filled outside [vlo, vhi))
// of a [.][D] tensor into a tile whose row 0 is row lo.
template <int D>
__device__ __forceinline__ void stage_rows(uint8_t *tile, const __nv_bfloat16 *base, int64_t sl, int lo, int hi, int vlo,
                                           int vhi, int tid, int nthreads) {
  // (a thread keeps its 16-byte column; its rows are a multiple of 8 apart, so the swizzle stays the same)
  const int step = nthreads / (D / 8), r = tid / (D / 8), ch = tid % (D / 8);
  uint32_t dst = smem_addr(tile) + tile_off<D>(r, ch);
  const __nv_bfloat16 *src = base + (int64_t)(lo + r) * sl + ch * 8;
#pragma unroll 2
  for (int p = lo + r; p < hi; p += step) {
    if (p >= vlo && p < vhi) cp_async16(dst, src);
    else asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(dst), "r"(0u) : "memory");
    dst += step * 2 * D;
    src += step * sl;
  }
}

__device__ __forceinline__ uint32_t bits_range(int lo, int hi) {  // bits lo .. hi - 1 of 32
  const uint32_t up = hi >= 32 ? ~0u : ((1u << hi) - 1u);
  return lo >= 32 ? 0u : up & ~((1u << lo) - 1u);
}
// a 64-bit set of 16-position chunks from a test evaluated per lane for chunks lane and lane + 32
__device__ __forceinline__ uint64_t ballot64(bool lo, bool hi) {
  return (uint64_t)__ballot_sync(0xffffffffu, lo) | ((uint64_t)__ballot_sync(0xffffffffu, hi) << 32);
}
// ---- 16-column masks (bit c = column c) ----
__device__ __forceinline__ uint32_t cols16(int lo, int hi) {  // columns lo .. hi, clipped to 0 .. 15
  lo = max(lo, 0);
  hi = min(hi, 15);
  return lo > hi ? 0u : (0xffffu >> (15 - hi)) & (0xffffu << lo);
}
__device__ __forceinline__ int pow2_ge(int x) { return x <= 1 ? 1 : 1 << (32 - __clz(x - 1)); }
__device__ __forceinline__ int mask_block_of(const Shape &s, int t) { return s.stis_blk == 1 ? t : t / s.stis_blk; }
// Eq. 15 for query t over the keys p0 ... p0 + 15, without causality and padding (the caller ANDs them).
template <bool PLAIN>
__device__ __forceinline__ uint32_t st_keys16(const Shape &s, int t, int p0, bool causal) {
  if (PLAIN) return cols16(t - s.window + 1 - p0, 15);
  uint32_t m = cols16(t - s.window + 1 - p0, causal ? 15 : t + s.window - 1 - p0);
  if (s.stis_mode) {
    const int blk = s.stis_blk;
    m |= cols16(s.L - blk - p0, 15);
    if (blk == 1 && causal) {
      // single keys at power-of-two distances: column c is at distance d0 - c.  Up to distance 31 the
      // pattern is a shifted constant (bits 1, 2, 4, 8, 16 mirrored), beyond it a chunk holds at most one.
      const int d0 = t - p0;
      if (d0 <= 31) return d0 < 0 ? m : (m | (__brev(0x00010116u) >> (31 - d0))) & 0xffffu;
      const int pw = 1 << (31 - __clz(d0));
      return d0 - pw <= 15 ? m | (1u << (d0 - pw)) : m;
    }
    const int bq = mask_block_of(s, t);
    for (int d = pow2_ge(bq - mask_block_of(s, p0 + 15)); d <= bq; d <<= 1) {  // key block bq - d
      const int a = (bq - d) * blk - p0;
      if (a + blk - 1 < 0) break;
      m |= cols16(a, a + blk - 1);
    }
    if (!causal)
      for (int d = pow2_ge(mask_block_of(s, p0) - bq);; d <<= 1) {  // and key block bq + d
        const int a = (bq + d) * blk - p0;
        if (a > 15 || a + p0 >= s.L) break;
        m |= cols16(a, a + blk - 1);
      }
  }
  return m;
}
// The same mask seen from key p over the queries t0 ... t0 + 15.
template <bool PLAIN>
__device__ __forceinline__ uint32_t st_queries16(const Shape &s, int p, int t0, bool causal) {
  if (PLAIN) return cols16(0, p + s.window - 1 - t0);
  uint32_t m = cols16(causal ? 0 : p - s.window + 1 - t0, p + s.window - 1 - t0);
  if (s.stis_mode) {
    const int blk = s.stis_blk;
    if (p >= s.L - blk) return 0xffffu;
    if (blk == 1 && causal) {  // column c is at distance d0 + c
      const int d0 = t0 - p;
      if (d0 <= 16) return (m | (d0 >= 0 ? 0x00010116u >> d0 : d0 > -16 ? 0x00010116u << -d0 : 0u)) & 0xffffu;
      const int pw = pow2_ge(d0);
      return pw - d0 <= 15 ? m | (1u << (pw - d0)) : m;
    }
    const int bk = mask_block_of(s, p);
    for (int d = pow2_ge(mask_block_of(s, t0) - bk);; d <<= 1) {  // query block bk + d
      const int a = (bk + d) * blk - t0;
      if (a > 15 || a + t0 >= s.L) break;
      m |= cols16(a, a + blk - 1);
    }
    if (!causal)
      for (int d = pow2_ge(bk - mask_block_of(s, t0 + 15)); d <= bk; d <<= 1) {  // and query block bk - d
        const int a = (bk - d) * blk - t0;
        if (a + blk - 1 < 0) break;
        m |= cols16(a, a + blk - 1);
      }
  }
  return m;
}
__device__ __forceinline__ float quad_sum(float x) {
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x + __shfl_xor_sync(0xffffffffu, x, 2);
}
__device__ __forceinline__ float quad_max(float x) {
  x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 1));
  return fmaxf(x, __shfl_xor_sync(0xffffffffu, x, 2));
}
__device__ __forceinline__ float head_alpha(const float *gate, int h) {
  return 1.f / (1.f + __expf(-(gate[h * 2 + 0] - gate[h * 2 + 1])));
}

}  // namespace sh
}  // namespace blossom
