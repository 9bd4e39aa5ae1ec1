// Kernels without a texel class (table upload, vertex setup, raster) and the
// host-side launchers, which dispatch the shading kernels to the
// translation unit of the batch's texel class.

#include "vs_kernels.cuh"

namespace vsd {

template <int BYTES>
__device__ __forceinline__ void write_chunk(char* ws, const Upload<BYTES>& c) {
  uint4* dst = reinterpret_cast<uint4*>(ws + c.dst_off);
  for (uint32_t i = threadIdx.x; i < c.nbytes / 16; i += blockDim.x) dst[i] = c.data[i];
  if (c.reset && threadIdx.x == 0) {
    WsHeader* h = reinterpret_cast<WsHeader*>(ws);
    h->next_unit = 0;
    h->abort = 0;
    h->launches += (unsigned long long)c.launches;
    h->kernel_class = c.kernel_class;
  }
}

template <int BYTES>
__global__ void __launch_bounds__(kThreads) k_upload(char* ws, const __grid_constant__ Upload<BYTES> c) {
  write_chunk(ws, c);
}

// Plain per-phase kernels, with the same arithmetic as the persistent kernel.
// Setup: each warp runs one unit (8 per block) on the table it got as a kernel
// parameter, which block 0 writes to the workspace for the kernels behind: a
// launch (3 us on the GPU, and the host's share of a small frame) less than
// with an upload before it.  Shading: block b runs unit b, its warp w runs
// round w of it.
__global__ void __launch_bounds__(kThreads) k_setup(char* ws, const __grid_constant__ SmallUpload t,
                                                    uint32_t shells_off) {
  if (blockIdx.x == 0) {
    write_chunk(ws, t);
    return;
  }
  const char* table = reinterpret_cast<const char*>(t.data);
  const DItem& it = *reinterpret_cast<const DItem*>(table);
  const int u = (blockIdx.x - 1) * kWarps + (threadIdx.x >> 5);
  if (u < it.units[PH_SETUP]) unit_setup(it, reinterpret_cast<const DShell*>(table + shells_off) + it.shell0, u);
}

// Raster: resident blocks only, every warp strides over the item's units (of
// 32 triangles, or fewer where the mesh is too small to give every warp
// one: see vs_units.h).  What bounds it: latency of the dependent index and
// vertex loads and of the walk.  A block adds its counts to the workspace
// header once: additions by each warp of 256 triangles are 87 k atomics on one
// cache line for an 800^2 view of 7 x 200 k triangles, and they are then the
// kernel's time.
template <bool FULL>
__global__ void __launch_bounds__(kThreads, kRasterBlocks) k_raster(TableRef tb, int item) {
  __shared__ unsigned s_count[7];
  const DItem& it = tb.items[item];
  const DShell* sh = tb.shells + it.shell0;
  const int w = threadIdx.x >> 5;
  if (threadIdx.x < 7) s_count[threadIdx.x] = 0;
  __syncthreads();
  RasterCounts rc = {0, 0, 0, 0};
  for (int u = blockIdx.x * kWarps + w; u < it.units[PH_RASTER]; u += gridDim.x * kWarps)
    unit_raster<FULL>(it, sh, u, vs_smem + w * kRasterWarpBytes, rc);
  const unsigned c[7] = {rc.fb & 0xFFFFu, rc.fb >> 16, rc.ng & 0xFFFFu, rc.ng >> 16, rc.lc & 0xFFFFu, rc.lc >> 16,
                         rc.bad};
#pragma unroll
  for (int q = 0; q < 7; ++q) {
    const unsigned v = __reduce_add_sync(0xffffffffu, c[q]);
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_count[q], v);
  }
  __syncthreads();
  if (threadIdx.x < 6 && s_count[threadIdx.x]) {
    WsHeader* h = tb.hdr;
    unsigned long long* dst[6] = {&h->front, &h->back, &h->nearc, &h->guard, &h->large, &h->clipped};
    atomicAdd(dst[threadIdx.x], (unsigned long long)s_count[threadIdx.x]);
  }
  if (threadIdx.x == 6 && s_count[6]) record_error(tb.hdr, VS_ERR_INVALID_ARG);
}

}  // namespace vsd

// ----------------------------------------------------------------------------
// host-side launchers (C++ linkage, used by vs_api.cu)
// ----------------------------------------------------------------------------
namespace vsk {

const TcOps& tc_ops(int tc) {
  switch (tc) {
    case vsd::TC_RGBA: return kTcRgba;
    case vsd::TC_SH0: return kTcSh0;
    case vsd::TC_SH0 + 1: return kTcSh1;
    case vsd::TC_SH0 + 2: return kTcSh2;
    case vsd::TC_SH0 + 3: return kTcSh3;
    case vsd::TC_U80: return kTcU80;
    case vsd::TC_U80 + 1: return kTcU81;
    case vsd::TC_U80 + 2: return kTcU82;
    case vsd::TC_U80 + 3: return kTcU83;
    default: return kTcAny;
  }
}

cudaError_t upload(char* ws, const UploadChunk& c, cudaStream_t st) {
  vsd::k_upload<<<1, vsd::kThreads, 0, st>>>(ws, c);
  return cudaGetLastError();
}
cudaError_t upload(char* ws, const SmallUpload& c, cudaStream_t st) {
  vsd::k_upload<<<1, vsd::kThreads, 0, st>>>(ws, c);
  return cudaGetLastError();
}

static void launch_setup(char* ws, const SmallUpload& t, uint32_t shells_off, int units, cudaStream_t st) {
  const int W = vsd::kWarps;
  vsd::k_setup<<<1 + (units + W - 1) / W, vsd::kThreads, 0, st>>>(ws, t, shells_off);
}

int plain_forward_launches(const int units[4]) { return 1 + (units[1] > 0) + (units[2] > 0); }
int plain_backward_launches(const int units[4]) { return 1 + (units[2] > 0); }

cudaError_t plain_forward(const TableRef& tb, char* ws, const SmallUpload& t, uint32_t shells_off, const int units[4],
                          int tc, bool full, int sms, cudaStream_t st) {
  const int W = vsd::kWarps;
  launch_setup(ws, t, shells_off, units[0], st);
  if (units[1]) {
    const int grid = std::min((units[1] + W - 1) / W, sms * vsd::kRasterBlocks);
    if (full) vsd::k_raster<true><<<grid, vsd::kThreads, vsd::kRasterWarpBytes * W, st>>>(tb, 0);
    else vsd::k_raster<false><<<grid, vsd::kThreads, vsd::kRasterWarpBytes * W, st>>>(tb, 0);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !units[2]) return e;
  return tc_ops(tc).shade(tb, false, full, units[2], vsd::block_smem_bytes(tb.kmax, false, tc), st);
}

cudaError_t plain_backward(const TableRef& tb, char* ws, const SmallUpload& t, uint32_t shells_off, const int units[4],
                           int tc, bool full, cudaStream_t st) {
  launch_setup(ws, t, shells_off, units[0], st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !units[2]) return e;
  return tc_ops(tc).shade(tb, true, full, units[2], vsd::block_smem_bytes(tb.kmax, true, tc), st);
}

cudaError_t persistent(const TableRef& tb, bool bwd, int tc, bool full, int grid, long long spin_limit,
                       cudaStream_t st) {
  return tc_ops(tc).persistent(tb, bwd, full, grid, spin_limit, vsd::pers_smem_bytes(tb.kmax, bwd, tc), st);
}

cudaError_t persistent_occupancy(bool bwd, int tc, bool full, int kmax, int* blocks_per_sm) {
  return tc_ops(tc).occupancy(bwd, full, vsd::pers_smem_bytes(kmax, bwd, tc), blocks_per_sm);
}

cudaError_t configure_kernels() {
  for (int tc = 0; tc < vsd::kNumTc; ++tc) {
    const int most_f = (int)std::max(vsd::block_smem_bytes(vsd::kMaxShells, false, tc),
                                     vsd::pers_smem_bytes(vsd::kMaxShells, false, tc));
    const int most_b = (int)std::max(vsd::block_smem_bytes(vsd::kMaxShells, true, tc),
                                     vsd::pers_smem_bytes(vsd::kMaxShells, true, tc));
    cudaError_t e = tc_ops(tc).configure(most_f, most_b);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace vsk
