// Rotary position embedding of q and k inside the library (paper: "RoPE is applied to Q and K to
// encode relative positional information" before both branches).
//
// With rope_theta > 0 every entry point first writes rotated copies of q and k into the workspace
// (same strides as the originals) and runs on those; the backward afterwards turns the gradients
// of the rotated tensors back (the rotation is orthogonal: its transpose).  Pairs are the
// interleaved ones of the original formulation, (x[2i], x[2i+1]), rotated by the angle
// t * theta^(-2i / D) at array position t.  The rotation is evaluated in double precision and
// rounded once to the storage type, so that it is the storage-type rounding of the exact rotation.
#include "common.cuh"

namespace blossom {
namespace {

// Eight consecutive elements (four pairs), rotated in double precision, rounded once.
template <typename T>
struct Vec8;
template <>
struct Vec8<float> {
  float4 a, b;
  __device__ __forceinline__ void load(const float *p) {
    a = reinterpret_cast<const float4 *>(p)[0];
    b = reinterpret_cast<const float4 *>(p)[1];
  }
  __device__ __forceinline__ static void turn(float &x, float &y, double2 cs) {
    const double u = x, v = y;
    x = (float)(u * cs.x - v * cs.y);
    y = (float)(u * cs.y + v * cs.x);
  }
  __device__ __forceinline__ void rotate_store(const double2 (&cs)[4], float *p) {
    turn(a.x, a.y, cs[0]); turn(a.z, a.w, cs[1]); turn(b.x, b.y, cs[2]); turn(b.z, b.w, cs[3]);
    reinterpret_cast<float4 *>(p)[0] = a;
    reinterpret_cast<float4 *>(p)[1] = b;
  }
};
template <>
struct Vec8<__nv_bfloat16> {
  uint4 r;
  __device__ __forceinline__ void load(const __nv_bfloat16 *p) { r = *reinterpret_cast<const uint4 *>(p); }
  __device__ __forceinline__ static uint32_t turn(uint32_t w, double2 cs) {
    const double u = __uint_as_float(w << 16), v = __uint_as_float(w & 0xffff0000u);
    __nv_bfloat162 h;
    h.x = __double2bfloat16(u * cs.x - v * cs.y);
    h.y = __double2bfloat16(u * cs.y + v * cs.x);
    return *reinterpret_cast<uint32_t *>(&h);
  }
  __device__ __forceinline__ void rotate_store(const double2 (&cs)[4], __nv_bfloat16 *p) {
    *reinterpret_cast<uint4 *>(p) = make_uint4(turn(r.x, cs[0]), turn(r.y, cs[1]), turn(r.z, cs[2]), turn(r.w, cs[3]));
  }
};

// cos and sin of every (position, pair), once per call: [L][D / 2].
__global__ void __launch_bounds__(128) rope_table_kernel(int L, int D, double theta, double2 *__restrict__ table) {
  grid_chain_enter();
  const int half = D / 2;
  const int e = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (e >= L * half) return;
  const int i = e % half, t = e / half;
  double sn, cs;
  sincos((double)t * pow(theta, -2.0 * (double)i / (double)D), &sn, &cs);
  table[e] = make_double2(cs, sn);
}

// One or two tensors ([B][heads][L][D] with strides) rotated by the table's angles (dir = +1) or their
// negatives (-1).  A thread owns four consecutive pairs of a position and walks a slice of the (batch,
// head) rows of both tensors with them, four rows in flight: the table is read once per slice.  Double
// precision per pair and one rounding; what bounds it then is memory (q and k of B 16, H 4, L 900, D 64:
// 15 MB in and as much out).  Evaluating the angles in every slice of the rows instead took 16 us a tensor
// at that size (900 x 32 angles, eleven times), four launches a training step.
struct RopeTensor {
  const void *src;  // may equal dst
  void *dst;
  int rows, heads;  // rows = B * heads
  int64_t sb, sh, sl;
};
template <typename T>
__global__ void __launch_bounds__(256) rope_kernel(int L, int D, int dir, const double2 *__restrict__ table, RopeTensor x,
                                                   RopeTensor y) {
  grid_chain_enter();
  const int quads = D / 8;
  const int e = (int)(blockIdx.x * blockDim.x + threadIdx.x);
  if (e >= L * quads) return;
  const int t = e / quads, c = (e % quads) * 8;
  double2 cs[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    cs[j] = table[t * (D / 2) + c / 2 + j];
    if (dir < 0) cs[j].y = -cs[j].y;
  }
  const int rows = x.rows + y.rows;
  for (int r0 = (int)blockIdx.y * 4; r0 < rows; r0 += (int)gridDim.y * 4) {
    Vec8<T> v[4];
    T *out[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + j;
      if (r < rows) {
        const RopeTensor &z = r < x.rows ? x : y;
        const int k = r < x.rows ? r : r - x.rows;
        const int64_t off = (int64_t)(k / z.heads) * z.sb + (int64_t)(k % z.heads) * z.sh + (int64_t)t * z.sl + c;
        v[j].load(static_cast<const T *>(z.src) + off);
        out[j] = static_cast<T *>(z.dst) + off;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (r0 + j < rows) v[j].rotate_store(cs, out[j]);
  }
}

}  // namespace

// Rotates q-shaped `qs` into `qd` and k-shaped `ks` into `kd` (dir = +1) or back (-1).  table: [L][D / 2]
// double2 in the workspace, filled first unless `have_table`.
int launch_rope(const Shape &s, int dtype, int dir, const void *qs, void *qd, const void *ks, void *kd, void *table,
                bool have_table, cudaStream_t st) {
  double2 *tab = static_cast<double2 *>(table);
  if (!have_table) {
    LaunchScope ls(K_ROPE, st);
    launch_chained(rope_table_kernel, dim3((unsigned)((s.L * (s.D / 2) + 127) / 128)), dim3(128), 0, st, s.L, s.D,
                   s.rope_theta, tab);
  }
  const RopeTensor x = {qs, qd, s.B * s.H, s.H, s.sb, s.sh, s.sl}, y = {ks, kd, s.B * s.Hkv, s.Hkv, s.ksb, s.ksh, s.ksl};
  const unsigned gx = (unsigned)((s.L * (s.D / 8) + 255) / 256);
  // enough slices of the rows to fill the GPU about eight CTAs deep, each of at least four rows
  const int64_t want = (148 * 8 + gx - 1) / gx, most = ((int64_t)x.rows + y.rows + 3) / 4;
  int64_t gy = want < 1 ? 1 : (want > most ? most : want);
  if (gy > 65535) gy = 65535;
  LaunchScope ls(K_ROPE, st);
  auto kern = dtype == BLOSSOM_DTYPE_FP32 ? rope_kernel<float> : rope_kernel<__nv_bfloat16>;
  launch_chained(kern, dim3(gx, (unsigned)gy), dim3(256), 0, st, s.L, s.D, dir, (const double2 *)tab, x, y);
  return cudaGetLastError() == cudaSuccess ? BLOSSOM_OK : BLOSSOM_ERR_CUDA;
}

}  // namespace blossom
