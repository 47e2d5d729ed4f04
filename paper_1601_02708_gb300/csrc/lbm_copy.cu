// One launch for a list of copies on the device.
#include <cstring>

#include "lbm_ctx.h"

namespace {

constexpr int kCopyThreads = 256;
constexpr int kCopyChunk = kCopyThreads * 4 * 16;  // bytes a block moves

struct CopyArgs {
  CopyItem item[kCopyMax];
  int first[kCopyMax + 1];  // first block of each item
  int n;
  int head_bytes;
  unsigned char* head_dst;
  unsigned char head[kCopyHead];
};
static_assert(sizeof(CopyArgs) <= 4000, "kernel parameters");

template <typename V>
__device__ __forceinline__ void move_as(char* dst, const char* src, size_t len) {
  const size_t n = len / sizeof(V);
  V* d = (V*)dst;
  const V* s = (const V*)src;
  size_t i = threadIdx.x;
  for (; i + 3 * kCopyThreads < n; i += 4 * kCopyThreads) {
    V v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = s[i + k * kCopyThreads];
#pragma unroll
    for (int k = 0; k < 4; ++k) d[i + k * kCopyThreads] = v[k];
  }
  for (; i < n; i += kCopyThreads) d[i] = s[i];
  for (size_t b = n * sizeof(V) + threadIdx.x; b < len; b += kCopyThreads) dst[b] = src[b];
}

// A block moves one chunk of one item, by the widest words that both addresses
// allow; a null source stores zeros.  Such lists are a saved state's dozen
// arrays and the edge data of a call: megabytes at most on a small lattice,
// whose separate copies took about 5 us each (2 of work, 3 between two of
// them).  Ten substeps of a 256 x 64 channel with restore and trace went from 139
// to 119 us, 50 of a dissolving 512 x 512 block from 653 to 552, 25 of 24 lattices
// together, with 72 pieces of edge data, from 2.58 to 2.21 ms.  Large states
// gain too: saved and restored, 1024 x 1024 nodes with mineral (73 MB) took 98
// and 103 us as separate copies, 28 and 43 this way; 4096 x 4096 (1.15 GB)
// 435 and 427, now 343 and 388.
__global__ void __launch_bounds__(kCopyThreads) k_copy_list(const __grid_constant__ CopyArgs a) {
  if (blockIdx.x == 0 && (int)threadIdx.x < a.head_bytes) a.head_dst[threadIdx.x] = a.head[threadIdx.x];
  if (a.n == 0) return;  // the head alone
  int i = 0;
  while (i + 1 < a.n && (int)blockIdx.x >= a.first[i + 1]) ++i;
  const CopyItem it = a.item[i];
  const size_t off = (size_t)((int)blockIdx.x - a.first[i]) * kCopyChunk;
  const size_t len = it.bytes - off < (size_t)kCopyChunk ? it.bytes - off : (size_t)kCopyChunk;
  char* dst = (char*)it.dst + off;
  const char* src = (const char*)it.src + off;
  if (!it.src) {
    size_t n = ((size_t)dst & 15) ? 0 : len / 16;
    for (size_t k = threadIdx.x; k < n; k += kCopyThreads) ((uint4*)dst)[k] = make_uint4(0, 0, 0, 0);
    for (size_t k = n * 16 + threadIdx.x; k < len; k += kCopyThreads) dst[k] = 0;
    return;
  }
  const size_t both = (size_t)dst | (size_t)src;
  if ((both & 15) == 0) move_as<uint4>(dst, src, len);
  else if ((both & 7) == 0) move_as<uint2>(dst, src, len);
  else if ((both & 3) == 0) move_as<unsigned>(dst, src, len);
  else move_as<unsigned char>(dst, src, len);
}

}  // namespace

cudaError_t ctx_copy_list(const CopyItem* items, int n, cudaStream_t stream, const void* head,
                          void* head_dst, int head_bytes) {
  int k = 0;
  bool headed = head_bytes == 0;
  while (k < n || !headed) {
    CopyArgs a;
    a.n = 0;
    a.head_bytes = headed ? 0 : head_bytes;
    a.head_dst = (unsigned char*)head_dst;
    if (a.head_bytes) memcpy(a.head, head, (size_t)head_bytes);
    long long blocks = 0;
    for (; k < n && a.n < kCopyMax; ++k) {
      const long long need = (long long)((items[k].bytes + kCopyChunk - 1) / kCopyChunk);
      if (need == 0) continue;
      if (blocks + need > 0x7FFFFFFFll) break;  // (one item is below 2^35 bytes)
      a.item[a.n] = items[k];
      a.first[a.n++] = (int)blocks;
      blocks += need;
    }
    if (a.n == 0 && k < n) return cudaErrorInvalidValue;
    if (a.n == 0 && headed) break;
    headed = true;
    a.first[a.n] = (int)blocks;
    k_copy_list<<<(unsigned)(blocks > 0 ? blocks : 1), kCopyThreads, 0, stream>>>(a);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

bool ctx_on_this_device(const void* p, int device) {
  cudaPointerAttributes at;
  if (!p || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice && at.device == device;
}

bool ctx_in_reach(const void* p, int device) {
  cudaPointerAttributes at;
  if (!p || cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == device);
}
