// Pocket packing kernel and the dispatch from (bucket, grid dtype) to kernel instantiations.
#include <cuda_fp16.h>
#include <math_constants.h>

#include "dock_internal.h"

namespace dockgpu {

// One instantiation per (grid type, warps per item, pose tile), from dock_kernels_inst.cu; the
// tile of 2 exists for 1 and 2 warps per item (larger groups already hold many angles in flight).
#define DOCK_DECLARE_INST(f, g, t)                                                                          \
  cudaError_t launch_bucket_f##f##_##g##_##t(int bucket, const PocketDev& pk, const BatchDev& b, const ParamsDev& p, \
                                             const uint32_t* items, int n_items, const LaunchCfg& cfg,            \
                                             cudaStream_t s, bool set_attributes);
#define DOCK_DECLARE_GT(f) \
  DOCK_DECLARE_INST(f, 1, 1) DOCK_DECLARE_INST(f, 2, 1) DOCK_DECLARE_INST(f, 4, 1) DOCK_DECLARE_INST(f, 8, 1) \
  DOCK_DECLARE_INST(f, 1, 2) DOCK_DECLARE_INST(f, 2, 2)
DOCK_DECLARE_GT(0)
DOCK_DECLARE_GT(1)
DOCK_DECLARE_GT(2)

// The latency form, one instantiation per grid type, from dock_latency_inst.cu.
#define DOCK_DECLARE_LAT(f)                                                                                \
  cudaError_t launch_latency_f##f(int bucket, const PocketDev& pk, const BatchDev& b, const ParamsDev& p, int l, \
                                  const LatScratch& sc, cudaStream_t s, int* launches);
DOCK_DECLARE_LAT(0)
DOCK_DECLARE_LAT(1)
DOCK_DECLARE_LAT(2)

// Cell c = (k*(ny-1) + j)*(nx-1) + i gathers the 8 corner voxels of the grid cell whose lower
// corner is voxel (i, j, k); the extra last cell is all zeros (positions outside the grid).
__global__ void pack_pocket_kernel(const float* __restrict__ v, void* cells, int nx, int ny, int nz, int f16) {
  const long long nc = (long long)(nx - 1) * (ny - 1) * (nz - 1);
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c <= nc; c += (long long)gridDim.x * blockDim.x) {
    float q[8];
    if (c == nc) {
#pragma unroll
      for (int t = 0; t < 8; ++t) q[t] = 0.f;
    } else {
      const long long i = c % (nx - 1), j = (c / (nx - 1)) % (ny - 1), k = c / ((long long)(nx - 1) * (ny - 1));
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        const long long di = t & 1, dj = (t >> 1) & 1, dk = (t >> 2) & 1;
        q[t] = v[((k + dk) * ny + (j + dj)) * nx + (i + di)];
      }
    }
    if (f16) {
      __half2 h[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) h[t] = __halves2half2(__float2half_rn(q[2 * t]), __float2half_rn(q[2 * t + 1]));
      reinterpret_cast<uint4*>(cells)[c] = *reinterpret_cast<const uint4*>(h);
    } else {
      float4* o = reinterpret_cast<float4*>(cells) + 2 * c;
      o[0] = make_float4(q[0], q[1], q[2], q[3]);
      o[1] = make_float4(q[4], q[5], q[6], q[7]);
    }
  }
}

cudaError_t launch_pack_pocket(const float* values, void* cells, int nx, int ny, int nz, int f16, cudaStream_t s) {
  const long long nc = (long long)(nx - 1) * (ny - 1) * (nz - 1) + 1;
  const int threads = 256;
  const long long want = (nc + threads - 1) / threads;
  const int blocks = (int)(want < 65536 ? want : 65536);
  pack_pocket_kernel<<<blocks, threads, 0, s>>>(values, cells, nx, ny, nz, f16);
  return cudaGetLastError();
}

// The voxel (x, y, z) of the field a screening cell is built from: outside the grid 0, or the nearest
// voxel where only poses inside the grid are screened.
__device__ __forceinline__ float screen_voxel(const float* v, int x, int y, int z, int nx, int ny, int nz, int f16,
                                              bool outside) {
  const int cx = min(max(x, 0), nx - 1), cy = min(max(y, 0), ny - 1), cz = min(max(z, 0), nz - 1);
  if (outside && (cx != x || cy != y || cz != z)) return 0.f;
  const float a = v[((long long)cz * ny + cy) * nx + cx];
  return f16 ? __half2float(__float2half_rn(a)) : a;
}

__global__ void screen_range_kernel(const float* __restrict__ v, int nx, int ny, int nz, int f16, bool outside, int* r) {
  const long long cx = nx + 1, cy = ny + 1, nc = cx * cy * (nz + 1);  // cells -1 .. n - 1 of each axis
  float m[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < nc; c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % cx) - 1, j = (int)((c / cx) % cy) - 1, k = (int)(c / (cx * cy)) - 1;
    float q[8], lo = CUDART_INF_F, hi = -CUDART_INF_F;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      q[t] = screen_voxel(v, i + (t & 1), j + ((t >> 1) & 1), k + (t >> 2), nx, ny, nz, f16, outside);
      lo = fminf(lo, q[t]);
      hi = fmaxf(hi, q[t]);
    }
    m[0] = fmaxf(m[0], hi);
    m[1] = fmaxf(m[1], -lo);
    m[2] = fmaxf(m[2], hi - lo);
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      m[3] = fmaxf(m[3], fabsf(q[2 * t + 1] - q[2 * t]));
      m[4] = fmaxf(m[4], fabsf(q[(t & 1) + 4 * (t >> 1) + 2] - q[(t & 1) + 4 * (t >> 1)]));
      m[5] = fmaxf(m[5], fabsf(q[t + 4] - q[t]));
    }
  }
#pragma unroll
  for (int t = 0; t < 6; ++t) {
    for (int o = 16; o; o >>= 1) m[t] = fmaxf(m[t], __shfl_xor_sync(0xffffffffu, m[t], o));
    if ((threadIdx.x & 31) == 0) atomicMax(r + t, __float_as_int(m[t]));  // non-negative floats order as their bits
  }
}

// Screening cell (i, j, k), padded coordinates: the 8 corner voxels as integers Q = rint((V - vmin) / step),
// each stored as Q - mult * base in 7 bits; base (4 bits, common to the corners) sits in the top bits of the
// z = 0 corners' bytes.  Byte order (x, y) = (0,0), (1,0), (0,1), (1,1); the z = 1 corners follow.
__global__ void pack_screen_kernel(const float* __restrict__ v, uint2* out, ScreenDev sc, int nx, int ny, int nz, int cz,
                                   int f16, float inv_step) {
  const long long nc = (long long)sc.cx * sc.cy * cz;
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < nc; c += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(c % sc.cx) - kScreenPad, j = (int)((c / sc.cx) % sc.cy) - kScreenPad,
              k = (int)(c / ((long long)sc.cx * sc.cy)) - kScreenPad;
    int q[8], lo = 0x7fffffff;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      const float a = screen_voxel(v, i + (t & 1), j + ((t >> 1) & 1), k + (t >> 2), nx, ny, nz, f16, !sc.inside);
      q[t] = max(__float2int_rn((a - sc.vmin) * inv_step), 0);
      lo = min(lo, q[t]);
    }
    const int base = min(lo / (int)sc.mult, 15);
    unsigned w[2] = {0u, 0u};
#pragma unroll
    for (int t = 0; t < 8; ++t) w[t >> 2] |= (unsigned)min(q[t] - base * (int)sc.mult, 127) << (8 * (t & 3));
#pragma unroll
    for (int t = 0; t < 4; ++t) w[0] |= (unsigned)((base >> t) & 1) << (8 * t + 7);
    out[c] = make_uint2(w[0], w[1]);
  }
}

cudaError_t launch_screen_range(const float* values, int nx, int ny, int nz, int f16, int outside, int* r, cudaStream_t s) {
  const long long want = ((long long)(nx + 1) * (ny + 1) * (nz + 1) + 255) / 256;
  screen_range_kernel<<<(int)(want < 1216 ? want : 1216), 256, 0, s>>>(values, nx, ny, nz, f16, outside != 0, r);
  return cudaGetLastError();
}

cudaError_t launch_pack_screen(const float* values, void* cells, const ScreenDev& sc, int nx, int ny, int nz, int f16,
                               float inv_step, cudaStream_t s) {
  const int cz = nz - 1 + 2 * kScreenPad;
  const long long want = ((long long)sc.cx * sc.cy * cz + 255) / 256;
  pack_screen_kernel<<<(int)(want < 4864 ? want : 4864), 256, 0, s>>>(values, reinterpret_cast<uint2*>(cells), sc, nx, ny, nz,
                                                                     cz, f16, inv_step);
  return cudaGetLastError();
}

cudaError_t launch_dock_bucket(int bucket, const PocketDev& pk, const BatchDev& b, const ParamsDev& p,
                               const uint32_t* items, int n_items, const LaunchCfg& cfg, cudaStream_t s,
                               bool set_attributes) {
  if (n_items <= 0 && !set_attributes) return cudaSuccess;
  const int key = cfg.warps_per_item * 10 + (cfg.tile == 2 ? 2 : 1);
#define DOCK_DISPATCH_GT(f)                                                                        \
  switch (key) {                                                                                   \
    case 11: return launch_bucket_f##f##_1_1(bucket, pk, b, p, items, n_items, cfg, s, set_attributes); \
    case 21: return launch_bucket_f##f##_2_1(bucket, pk, b, p, items, n_items, cfg, s, set_attributes); \
    case 41: return launch_bucket_f##f##_4_1(bucket, pk, b, p, items, n_items, cfg, s, set_attributes); \
    case 81: return launch_bucket_f##f##_8_1(bucket, pk, b, p, items, n_items, cfg, s, set_attributes); \
    case 12: return launch_bucket_f##f##_1_2(bucket, pk, b, p, items, n_items, cfg, s, set_attributes); \
    case 22: return launch_bucket_f##f##_2_2(bucket, pk, b, p, items, n_items, cfg, s, set_attributes); \
  }
  if (pk.dtype == 2) {
    DOCK_DISPATCH_GT(2)
  } else if (pk.dtype == 1) {
    DOCK_DISPATCH_GT(1)
  } else {
    DOCK_DISPATCH_GT(0)
  }
#undef DOCK_DISPATCH_GT
  return cudaErrorInvalidValue;
}

cudaError_t launch_latency_ligand(int bucket, const PocketDev& pk, const BatchDev& b, const ParamsDev& p, int l,
                                  const LatScratch& sc, cudaStream_t s, int* launches) {
  switch (pk.dtype) {
    case 0: return launch_latency_f0(bucket, pk, b, p, l, sc, s, launches);
    case 1: return launch_latency_f1(bucket, pk, b, p, l, sc, s, launches);
    case 2: return launch_latency_f2(bucket, pk, b, p, l, sc, s, launches);
  }
  return cudaErrorInvalidValue;
}

}  // namespace dockgpu
