// Rows of one layout into another: an upstream gradient that arrives as the transposed view a projection hands
// back, inputs that are slices of a packed projection.
//
// Bound: memory, every byte once in and once out.  A thread moves 16 bytes of four rows, all four loads before the
// first store; lanes run along a row and then along the positions, so that either side is touched in whole rows
// (64 bytes and more: whole sectors) whatever the order of its dimensions.  PyTorch's strided copy moves one
// element a time and divides for each.  B 128, H 2, L 1024, D 32 from [B, L, H, D] (34 MB in and out): forward + backward
// 311.9 -> 293.8 us, of which PyTorch's copy was 24.
#include "common.cuh"

namespace blossom {
namespace {

constexpr int kCopyThreads = 256, kCopyRows = 4;

struct RowStrides {  // in bytes
  int64_t b, h, l;
};

__global__ void __launch_bounds__(kCopyThreads) copy_rows_kernel(int H, int L, unsigned rows, int chunk_bits,
                                                                 const uint8_t *__restrict__ src, RowStrides ss,
                                                                 uint8_t *__restrict__ dst, RowStrides ds) {
  grid_chain_enter();
  const unsigned step = kCopyThreads >> chunk_bits;  // rows a CTA takes at a time
  const int c = ((int)threadIdx.x & ((1 << chunk_bits) - 1)) * 16;
  const unsigned row0 = blockIdx.x * (step * kCopyRows) + (threadIdx.x >> chunk_bits);
  unsigned bh = row0 / (unsigned)L, l = row0 - bh * (unsigned)L, b = bh / (unsigned)H, h = bh - b * (unsigned)H;
  uint4 v[kCopyRows];
  uint8_t *to[kCopyRows];
#pragma unroll
  for (int j = 0; j < kCopyRows; ++j) {
    if (row0 + j * step < rows) {
      v[j] = *reinterpret_cast<const uint4 *>(src + b * ss.b + h * ss.h + l * ss.l + c);
      to[j] = dst + b * ds.b + h * ds.h + l * ds.l + c;
    }
    l += step;
    if (l >= (unsigned)L) {
      const unsigned over = l / (unsigned)L;
      l -= over * (unsigned)L;
      h += over;
      if (h >= (unsigned)H) {
        const unsigned more = h / (unsigned)H;
        h -= more * (unsigned)H;
        b += more;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < kCopyRows; ++j)
    if (row0 + j * step < rows) *reinterpret_cast<uint4 *>(to[j]) = v[j];
}

}  // namespace
}  // namespace blossom

extern "C" int blossom_copy_rows(int32_t B, int32_t H, int32_t L, int32_t row_bytes, const void *src, const int64_t *src_strides,
                                 void *dst, const int64_t *dst_strides, blossom_stream_t stream) {
  using namespace blossom;
  if (B < 1 || H < 1 || L < 1 || !src || !dst || !src_strides || !dst_strides) return BLOSSOM_ERR_INVALID_ARG;
  // 16-byte pieces: a row of 2^n of them, and every row of either side on a 16-byte boundary
  const int chunks = row_bytes / 16;
  if (row_bytes < 16 || row_bytes > 16 * kCopyThreads || row_bytes != chunks * 16 || (chunks & (chunks - 1)))
    return BLOSSOM_ERR_UNSUPPORTED;
  if ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15) return BLOSSOM_ERR_UNSUPPORTED;
  for (int i = 0; i < 3; ++i)
    if (src_strides[i] < 0 || dst_strides[i] < 0 || ((src_strides[i] | dst_strides[i]) & 15)) return BLOSSOM_ERR_UNSUPPORTED;
  const int64_t most = (int64_t)1 << 30, units = (int64_t)B * H, rows = units * L;  // (row numbers in 32 bits, the last CTA's too)
  if (units > most || rows > most) return BLOSSOM_ERR_UNSUPPORTED;  // (units first: their product with L may not fit 64 bits)
  int bits = 0;
  while (1 << bits < chunks) ++bits;
  const int64_t per_cta = (int64_t)(kCopyThreads >> bits) * kCopyRows;
  const RowStrides ss = {src_strides[0], src_strides[1], src_strides[2]}, ds = {dst_strides[0], dst_strides[1], dst_strides[2]};
  const cudaStream_t st = (cudaStream_t)stream;
  LaunchScope ls(K_COPY_ROWS, st);
  launch_chained(copy_rows_kernel, dim3((unsigned)((rows + per_cta - 1) / per_cta)), dim3(kCopyThreads), 0, st, H, L,
                 (unsigned)rows, bits, static_cast<const uint8_t *>(src), ss, static_cast<uint8_t *>(dst), ds);
  return cudaGetLastError() == cudaSuccess ? BLOSSOM_OK : BLOSSOM_ERR_CUDA;
}
