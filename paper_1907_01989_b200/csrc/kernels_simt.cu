// CUDA-core kernels: layout conversion, depthwise 3x3, direct convolution, element-wise, channel
// concatenation, global average pool, bilinear resize.  All work on the channel-sliced layout
//   element (b,h,w,c) -> ((c/4 * B + b) * P + h*W + w) * 4 + c%4,   P = H*W rounded up to even,
// and move one pixel-slice (4 channels: 8 bytes fp16, 16 bytes fp32) per vector access, so a
// warp touches 32 consecutive pixels of one plane = one contiguous 256 / 512-byte run.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "kernels.h"
#include "pdl.cuh"

namespace gi {
namespace {

template <typename T>
struct Px;  // one pixel-slice in storage type T

template <>
struct Px<__half> {
  static __device__ __forceinline__ float4 load(const __half* p) {
    const uint2 u = *reinterpret_cast<const uint2*>(p);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
    return make_float4(a.x, a.y, b.x, b.y);
  }
  static __device__ __forceinline__ void store(__half* p, float4 v) {
    const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
    uint2 u;
    u.x = *reinterpret_cast<const unsigned*>(&a);
    u.y = *reinterpret_cast<const unsigned*>(&b);
    *reinterpret_cast<uint2*>(p) = u;
  }
  static __device__ __forceinline__ float get(const __half* p) { return __half2float(*p); }
  static __device__ __forceinline__ void put(__half* p, float v) { *p = __float2half_rn(v); }
};

template <>
struct Px<float> {
  static __device__ __forceinline__ float4 load(const float* p) { return *reinterpret_cast<const float4*>(p); }
  static __device__ __forceinline__ void store(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
  static __device__ __forceinline__ float get(const float* p) { return *p; }
  static __device__ __forceinline__ void put(float* p, float v) { *p = v; }
};

__device__ __forceinline__ float act1(float v, int kind) {
  if (kind == GI_ACT_RELU) return fmaxf(v, 0.0f);
  if (kind == GI_ACT_RELU6) return fminf(fmaxf(v, 0.0f), 6.0f);
  return v;
}
__device__ __forceinline__ float4 act4(float4 v, int kind) {
  return make_float4(act1(v.x, kind), act1(v.y, kind), act1(v.z, kind), act1(v.w, kind));
}

// bias is already in v: activation, residual add, activation, in graph order
template <typename T>
__device__ __forceinline__ float4 epilogue(float4 v, const Epilogue& ep, const T* res, size_t idx) {
  v = act4(v, ep.act_pre);
  if (ep.has_res) {
    const float4 r = Px<T>::load(res + idx);
    v.x += r.x;
    v.y += r.y;
    v.z += r.z;
    v.w += r.w;
  }
  return act4(v, ep.act_post);
}

// ------------------------------------------------------------------ layout conversion
// grid: x over the pixels of a plane (padding pixel included), y strides over planes (slice * B + image; a grid
// dimension holds at most 65535, deep tensors at large batch have more planes than that)
template <typename T>
__global__ void pack_kernel(const T* __restrict__ nhwc, T* __restrict__ out, int B, int HW, int C, int P, int S) {
  pdl_launch_dependents();
  pdl_wait();
  const int pix = blockIdx.x * blockDim.x + threadIdx.x;
  if (pix >= P) return;
  for (int plane = blockIdx.y; plane < S * B; plane += gridDim.y) {
    const int s = plane / B, b = plane - s * B;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pix < HW) {
      const T* src = nhwc + (static_cast<size_t>(b) * HW + pix) * C + s * 4;
      const int n = min(4, C - s * 4);
      float t[4] = {0.f, 0.f, 0.f, 0.f};
      for (int j = 0; j < n; ++j) t[j] = Px<T>::get(src + j);
      v = make_float4(t[0], t[1], t[2], t[3]);
    }
    Px<T>::store(out + (static_cast<size_t>(plane) * P + pix) * 4, v);
  }
}

// fp16 images with 3 channels (the usual network input) whose pixel count is a multiple of 4:
// a thread turns 4 pixels (24 contiguous bytes, three 8-byte loads) into 4 pixel-slices (two
// 16-byte stores).  grid: x over quads of an image, y over images.
__global__ void pack3_f16_kernel(const uint2* __restrict__ nhwc, uint4* __restrict__ out, int quads) {
  pdl_launch_dependents();
  pdl_wait();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= quads) return;
  const size_t at = static_cast<size_t>(blockIdx.y) * quads + q;
  const uint2 a = __ldg(nhwc + at * 3), c = __ldg(nhwc + at * 3 + 1), d = __ldg(nhwc + at * 3 + 2);
  // halves h0..h11 = a.x, a.y, c.x, c.y, d.x, d.y (two per word); pixel i takes h[3i .. 3i+2] and a zero
  uint4 lo, hi;
  lo.x = a.x;
  lo.y = a.y & 0xffffu;
  lo.z = (a.y >> 16) | (c.x << 16);
  lo.w = c.x >> 16;
  hi.x = c.y;
  hi.y = d.x & 0xffffu;
  hi.z = (d.x >> 16) | (d.y << 16);
  hi.w = d.y >> 16;
  out[at * 2] = lo;
  out[at * 2 + 1] = hi;
}

template <typename T>
__global__ void unpack_kernel(const T* __restrict__ in, T* __restrict__ nhwc, int B, int HW, int C, int P, int S) {
  pdl_launch_dependents();
  pdl_wait();
  const size_t idx = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  const size_t total = static_cast<size_t>(B) * HW * S;
  if (idx >= total) return;
  const int s = static_cast<int>(idx % S);
  const int pix = static_cast<int>((idx / S) % HW);
  const int b = static_cast<int>(idx / (static_cast<size_t>(S) * HW));
  const float4 v = Px<T>::load(in + ((static_cast<size_t>(s) * B + b) * P + pix) * 4);
  const float t[4] = {v.x, v.y, v.z, v.w};
  T* dst = nhwc + (static_cast<size_t>(b) * HW + pix) * C + s * 4;
  const int n = min(4, C - s * 4);
  for (int j = 0; j < n; ++j) Px<T>::put(dst + j, t[j]);
}

// fp16, any channel count: a block turns 128 consecutive pixels of one image into one contiguous
// run of 128 * C halves.  The pixel-slices are read coalesced (8 bytes per lane and slice) into
// shared memory in NHWC order; the run is then written with 4-byte stores (plus a 2-byte store at
// a misaligned head / tail) instead of one 2-byte store per element.  grid: x over 128-pixel
// chunks of an image, y over images; dynamic shared memory: 128 * C halves.
__global__ void __launch_bounds__(128) unpack_f16_kernel(const __half* __restrict__ in, __half* __restrict__ nhwc, int B, int HW, int C,
                                                         int P, int S) {
  extern __shared__ __align__(16) unsigned char unpack_smem[];
  unsigned short* tile = reinterpret_cast<unsigned short*>(unpack_smem);
  pdl_launch_dependents();
  pdl_wait();
  const int pix0 = blockIdx.x * 128, b = blockIdx.y;
  const int npx = min(128, HW - pix0);
  const int t = threadIdx.x;
  if (t < npx) {
    const uint2* src = reinterpret_cast<const uint2*>(in) + static_cast<size_t>(b) * P + pix0 + t;
    const size_t step = static_cast<size_t>(B) * P;
    unsigned short* dst = tile + t * C;
    for (int s = 0; s < S; ++s, src += step) {
      const uint2 u = __ldg(src);
      const unsigned short h[4] = {static_cast<unsigned short>(u.x & 0xffffu), static_cast<unsigned short>(u.x >> 16),
                                   static_cast<unsigned short>(u.y & 0xffffu), static_cast<unsigned short>(u.y >> 16)};
      const int n = min(4, C - s * 4);
      for (int j = 0; j < n; ++j) dst[s * 4 + j] = h[j];
    }
  }
  __syncthreads();
  const size_t first = (static_cast<size_t>(b) * HW + pix0) * C;  // in halves
  const int total = npx * C;
  unsigned short* out = reinterpret_cast<unsigned short*>(nhwc) + first;
  const int head = static_cast<int>(first & 1);  // halves before the first 4-byte boundary
  if (t == 0 && head) out[0] = tile[0];
  const int words = (total - head) / 2;
  unsigned* out32 = reinterpret_cast<unsigned*>(out + head);
  for (int w = t; w < words; w += 128) {
    const int i = head + 2 * w;
    out32[w] = static_cast<unsigned>(tile[i]) | (static_cast<unsigned>(tile[i + 1]) << 16);
  }
  if (t == 0 && ((total - head) & 1)) out[total - 1] = tile[total - 1];
}

// ------------------------------------------------------------------ direct convolution
struct ConvGeom {
  int B, H, W, Sin, Pin, Ho, Wo, Sout, Pout;
  int kh, kw, sh, sw, dh, dw, pt, pl;
};

// Direct convolution on the CUDA cores: fp32 storage, and the shapes no tensor-core kernel runs in fp16 storage.
//
// A warp owns 32 output pixels x 32 output channels of the batch's flattened pixel axis, a lane 4 pixels x 8 channels.  The sum
// runs over units of (tap, 4 input channels); a unit is 32 pixel-slices + 512 bytes of weights, one 16-byte cp.async of each per
// lane into a ring of kConvStages units that belongs to the warp alone, so nothing waits for another warp.  Even and odd input
// channels are summed in the two halves of packed fp32 pairs (fma.rn.f32x2: pixel-slice and weights are pairs as they lie).
// The sum is split over `kw` warps of a CTA until the launch fills the chip - a layer of the last stage at batch 2 has 20 such
// tiles of 240 units each - and the partial sums are added in warp order through shared memory, so results do not depend on
// timing.  What bounds it: at small batch the chain of a launch (about 4 us), at large batch the shared-memory reads
// (12 16-byte reads per 64 packed multiply-adds).  The kernel before it gave one pixel and up to 32 channels to a thread
// that walked the whole sum by itself: 7x7 960 -> 160 at batch 2 took 225 us with one block per 32 channels (16 us now, each
// with an event pair around it); MobileNetV2-224 in fp32 storage at batch 2 3849 -> 352 us.
constexpr int kConvStages = 6;
constexpr int kConvStageBytes = 1024;  // 32 pixel-slices (512 bytes in fp32 storage) and 32 channels x 4 weights
constexpr int kConvWarpBytes = kConvStages * kConvStageBytes;
constexpr int kConvMaxSplit = 16;

__device__ __forceinline__ void cp_async_px(unsigned dst, const float* src, bool valid) {
  const unsigned n = valid ? 16u : 0u;  // 0: nothing is read, zeros are written
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_px(unsigned dst, const __half* src, bool valid) {
  const unsigned n = valid ? 8u : 0u;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void fma2(unsigned long long& acc, float a0, float a1, float b0, float b1) {
  unsigned long long a, b;
  asm("mov.b64 %0, {%1, %2};" : "=l"(a) : "f"(a0), "f"(a1));
  asm("mov.b64 %0, {%1, %2};" : "=l"(b) : "f"(b0), "f"(b1));
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

template <typename T>
__global__ void __launch_bounds__(32 * kConvMaxSplit) conv_simt_kernel(const T* __restrict__ in, const float4* __restrict__ w,
                                                                       const float* __restrict__ bias, const T* __restrict__ res,
                                                                       T* __restrict__ out, ConvGeom g, Epilogue ep, int kw) {
  extern __shared__ __align__(128) unsigned char conv_smem[];
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int part = warp % kw, tpc = (blockDim.x >> 5) / kw;
  const long long m_total = static_cast<long long>(g.B) * g.Pout;
  const long long m0 = (static_cast<long long>(blockIdx.x) * tpc + warp / kw) * 32;
  const int grp = blockIdx.y, taps = g.kh * g.kw, units = taps * g.Sin;
  const int u0 = static_cast<int>(static_cast<long long>(units) * part / kw), u1 = static_cast<int>(static_cast<long long>(units) * (part + 1) / kw);
  unsigned char* ring = conv_smem + warp * kConvWarpBytes;
  const unsigned ring_s = static_cast<unsigned>(__cvta_generic_to_shared(ring));

  // this lane copies one pixel: m0 + lane
  const long long m = m0 + lane;
  const int b = m < m_total ? static_cast<int>(m / g.Pout) : 0;
  const int rem = m < m_total ? static_cast<int>(m - static_cast<long long>(b) * g.Pout) : g.Pout;
  const int oy = rem / g.Wo, ox = rem - oy * g.Wo;
  const bool real = rem < g.Ho * g.Wo;
  const int y0 = oy * g.sh - g.pt, x0 = ox * g.sw - g.pl;
  const size_t slice_step = static_cast<size_t>(g.B) * g.Pin * 4;
  const float4* wsrc = w + (static_cast<size_t>(grp) * units + u0) * 32 + lane;
  int tap = u0 / g.Sin, s = u0 - tap * g.Sin;
  bool ok = false;
  const T* src = in;
  auto at_tap = [&]() {
    const int ky = tap / g.kw, kx = tap - ky * g.kw;
    const int iy = y0 + ky * g.dh, ix = x0 + kx * g.dw;
    ok = real && iy >= 0 && iy < g.H && ix >= 0 && ix < g.W;
    src = in + (ok ? (static_cast<size_t>(b) * g.Pin + static_cast<size_t>(iy) * g.W + ix) * 4 : 0) + s * slice_step;
  };
  at_tap();
  auto issue = [&](int u) {
    if (u < u1) {
      const unsigned dst = ring_s + ((u - u0) % kConvStages) * kConvStageBytes;
      cp_async_px(dst + lane * 4 * static_cast<unsigned>(sizeof(T)), src, ok);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 512 + lane * 16), "l"(wsrc) : "memory");
      wsrc += 32;
      src += slice_step;
      if (++s == g.Sin) {
        s = 0;
        ++tap;
        at_tap();
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  pdl_wait();
  for (int i = 0; i < kConvStages - 1; ++i) issue(u0 + i);
  const int pl = lane & 7, cl = lane >> 3;  // pixels pl + 8 i, channels cl + 4 j: lane cl holds component cl of every output slice
  unsigned long long acc[4][8];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0ull;
  for (int u = u0; u < u1; ++u) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kConvStages - 2) : "memory");
    __syncwarp();
    const unsigned char* st = ring + ((u - u0) % kConvStages) * kConvStageBytes;
    float4 x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = Px<T>::load(reinterpret_cast<const T*>(st) + (pl + 8 * i) * 4);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 wv = *reinterpret_cast<const float4*>(st + 512 + (cl + 4 * j) * 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        fma2(acc[i][j], x[i].x, x[i].y, wv.x, wv.y);
        fma2(acc[i][j], x[i].z, x[i].w, wv.z, wv.w);
      }
    }
    __syncwarp();
    issue(u + kConvStages - 1);
  }

  // partial sums: [output slice][pixel] float4 in the warp's own ring, then summed over the parts in order
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();
  float* part_sum = reinterpret_cast<float*>(ring);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float lo, hi;
      asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[i][j]));
      part_sum[(j * 32 + pl + 8 * i) * 4 + cl] = lo + hi;
    }
  __syncthreads();
  const float4* first = reinterpret_cast<const float4*>(conv_smem + (warp - part) * kConvWarpBytes);
  for (int i = part * 32 + lane; i < 256; i += kw * 32) {
    const int so = grp * 8 + (i >> 5);
    const long long mo = m0 + (i & 31);
    if (so >= g.Sout || mo >= m_total) continue;
    const size_t idx = (static_cast<size_t>(so) * m_total + mo) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (static_cast<int>(mo % g.Pout) < g.Ho * g.Wo) {  // the padding pixel of an odd plane holds zeros
      v = *reinterpret_cast<const float4*>(bias + so * 4);
      for (int k = 0; k < kw; ++k) {
        const float4 q = first[k * (kConvWarpBytes / 16) + i];
        v.x += q.x;
        v.y += q.y;
        v.z += q.z;
        v.w += q.w;
      }
      v = epilogue<T>(v, ep, res, idx);
    }
    Px<T>::store(out + idx, v);
  }
}

// ------------------------------------------------------------------ depthwise 3x3
template <typename T>
__global__ void __launch_bounds__(128) depthwise_kernel(const T* __restrict__ in, const float* __restrict__ w,
                                                        const float* __restrict__ bias, const T* __restrict__ res,
                                                        T* __restrict__ out, ConvGeom g, Epilogue ep) {
  pdl_launch_dependents();
  pdl_wait();
  const int pix = blockIdx.x * 128 + threadIdx.x;
  const int s = blockIdx.y, b = blockIdx.z;
  if (pix >= g.Pout) return;
  const size_t idx = ((static_cast<size_t>(s) * g.B + b) * g.Pout + pix) * 4;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (pix < g.Ho * g.Wo) {
    const int oy = pix / g.Wo, ox = pix - oy * g.Wo;
    const int C4 = g.Sin * 4;
    v = *reinterpret_cast<const float4*>(bias + s * 4);
    const T* plane = in + (static_cast<size_t>(s) * g.B + b) * g.Pin * 4;
#pragma unroll
    for (int ky = 0; ky < 3; ++ky) {
      const int iy = oy * g.sh - g.pt + ky * g.dh;
      if (iy < 0 || iy >= g.H) continue;
#pragma unroll
      for (int kx = 0; kx < 3; ++kx) {
        const int ix = ox * g.sw - g.pl + kx * g.dw;
        if (ix < 0 || ix >= g.W) continue;
        const float4 x = Px<T>::load(plane + (static_cast<size_t>(iy) * g.W + ix) * 4);
        const float4 wv = __ldg(reinterpret_cast<const float4*>(w + (ky * 3 + kx) * C4 + s * 4));
        v.x = fmaf(x.x, wv.x, v.x);
        v.y = fmaf(x.y, wv.y, v.y);
        v.z = fmaf(x.z, wv.z, v.z);
        v.w = fmaf(x.w, wv.w, v.w);
      }
    }
    v = epilogue<T>(v, ep, res, idx);
  }
  Px<T>::store(out + idx, v);
}

// ------------------------------------------------------------------ element-wise
template <typename T>
__global__ void eltwise_kernel(const T* __restrict__ a, const T* __restrict__ b, T* __restrict__ out, size_t n_px,
                               Epilogue ep) {
  pdl_launch_dependents();
  pdl_wait();
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (i >= n_px) return;
  const float4 v = epilogue<T>(Px<T>::load(a + i * 4), ep, b, i * 4);
  Px<T>::store(out + i * 4, v);
}

// ------------------------------------------------------------------ channel concatenation
// grid: x over the pixels of all planes of one output slice (B * P), y over output slices.  Output channel c
// is channel c of `a` for c < Ca and channel c - Ca of `b` after that; lanes beyond Ca + Cb and the padding
// pixel of a plane are written as zeros.  With Ca a multiple of 4 every output slice is one whole input
// slice (one vector load); otherwise each lane is fetched from the slice that holds it.
template <typename T>
__global__ void concat_kernel(const T* __restrict__ a, const T* __restrict__ b, T* __restrict__ out, size_t n_px, int P, int HW,
                              int Ca, int Cb) {
  pdl_launch_dependents();
  pdl_wait();
  const size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x;
  if (i >= n_px) return;
  const int so = blockIdx.y, c0 = so * 4;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (static_cast<int>(i % P) < HW) {
    if ((Ca & 3) == 0) {
      const bool from_a = c0 < Ca;
      const T* src = from_a ? a + (static_cast<size_t>(so) * n_px + i) * 4 : b + (static_cast<size_t>(so - Ca / 4) * n_px + i) * 4;
      v = Px<T>::load(src);
      const int valid = (from_a ? Ca : Ca + Cb) - c0;  // channels of this slice that exist
      if (valid < 4) v.w = 0.f;
      if (valid < 3) v.z = 0.f;
      if (valid < 2) v.y = 0.f;
    } else {
      float lane[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = c0 + j;
        lane[j] = 0.f;
        if (c < Ca) lane[j] = Px<T>::get(a + (static_cast<size_t>(c >> 2) * n_px + i) * 4 + (c & 3));
        else if (c < Ca + Cb) lane[j] = Px<T>::get(b + (static_cast<size_t>((c - Ca) >> 2) * n_px + i) * 4 + ((c - Ca) & 3));
      }
      v = make_float4(lane[0], lane[1], lane[2], lane[3]);
    }
  }
  Px<T>::store(out + (static_cast<size_t>(so) * n_px + i) * 4, v);
}

// ------------------------------------------------------------------ global average pool
// eight lanes (or a whole warp, launch_pool) per (slice, image): a lane strides over the pixels with all its
// loads independent (many small planes are latency-bound otherwise), then a shuffle reduction over
// the lanes in a fixed order
template <typename T, int L>
__global__ void pool_kernel(const T* __restrict__ in, T* __restrict__ out, int planes, int HW, int Pin, int Pout) {
  pdl_launch_dependents();
  pdl_wait();
  const int sub = threadIdx.x % L, plane_id = (blockIdx.x * blockDim.x + threadIdx.x) / L;
  const bool live = plane_id < planes;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (live) {
    const T* plane = in + static_cast<size_t>(plane_id) * Pin * 4;
    int p = sub;
    for (; p + 3 * L < HW; p += 4 * L) {  // four loads in flight
      const float4 x0 = Px<T>::load(plane + static_cast<size_t>(p) * 4), x1 = Px<T>::load(plane + static_cast<size_t>(p + L) * 4);
      const float4 x2 = Px<T>::load(plane + static_cast<size_t>(p + 2 * L) * 4), x3 = Px<T>::load(plane + static_cast<size_t>(p + 3 * L) * 4);
      s.x += (x0.x + x1.x) + (x2.x + x3.x);
      s.y += (x0.y + x1.y) + (x2.y + x3.y);
      s.z += (x0.z + x1.z) + (x2.z + x3.z);
      s.w += (x0.w + x1.w) + (x2.w + x3.w);
    }
    for (; p < HW; p += L) {
      const float4 x = Px<T>::load(plane + static_cast<size_t>(p) * 4);
      s.x += x.x;
      s.y += x.y;
      s.z += x.z;
      s.w += x.w;
    }
  }
  for (int d = L / 2; d > 0; d >>= 1) {
    s.x += __shfl_down_sync(0xffffffffu, s.x, d, L);
    s.y += __shfl_down_sync(0xffffffffu, s.y, d, L);
    s.z += __shfl_down_sync(0xffffffffu, s.z, d, L);
    s.w += __shfl_down_sync(0xffffffffu, s.w, d, L);
  }
  if (live && sub < Pout) {
    const float inv = 1.0f / static_cast<float>(HW);
    const float4 v = sub == 0 ? make_float4(s.x * inv, s.y * inv, s.z * inv, s.w * inv) : make_float4(0.f, 0.f, 0.f, 0.f);
    Px<T>::store(out + (static_cast<size_t>(plane_id) * Pout + sub) * 4, v);
  }
}

// ------------------------------------------------------------------ bilinear resize
// source coordinate as an exact fraction num/den so that floor() never depends on rounding.
// grid: x over the columns of a row, y = SOURCE row y0, z = image.  All output rows whose upper
// source row is y0 share the four source pixels of a column, so a thread interpolates along x once
// per slice (top, bottom - top) and then emits every such output row with one FMA per channel;
// the row weights are block-uniform and live in shared memory.  I is the integer type of the
// coordinate products (32 bits whenever OH*ny and OW*nx fit: 64-bit divisions are emulated).
constexpr int kResizeRows = 32;
template <typename T, typename I>
__global__ void __launch_bounds__(128) resize_kernel(const T* __restrict__ in, T* __restrict__ out, int B, int S, int H, int W,
                                                     int Pin, int OH, int OW, int Pout, int ny, int dy, int nx, int dx) {
  __shared__ float wy_s[kResizeRows];
  pdl_launch_dependents();
  pdl_wait();
  const int ox = blockIdx.x * 128 + threadIdx.x, y0 = blockIdx.y;
  const bool active = ox < OW;
  // output rows oy with floor(oy * ny / dy) == y0
  int oy_lo, oy_hi;
  if (ny == 0) {
    oy_lo = 0;
    oy_hi = y0 == 0 ? OH : 0;
  } else {
    oy_lo = static_cast<int>((static_cast<I>(y0) * static_cast<I>(dy) + static_cast<I>(ny - 1)) / static_cast<I>(ny));
    const I hi = (static_cast<I>(y0 + 1) * static_cast<I>(dy) + static_cast<I>(ny - 1)) / static_cast<I>(ny);
    oy_hi = hi > static_cast<I>(OH) ? OH : static_cast<int>(hi);
  }
  const int y1 = min(y0 + 1, H - 1);
  // column: source pixel pair and weight
  int x0 = 0, x1 = 0;
  float wx = 0.f;
  if (active) {
    const I qx = static_cast<I>(ox) * static_cast<I>(nx);
    x0 = static_cast<int>(qx / static_cast<I>(dx));
    wx = static_cast<float>(qx - static_cast<I>(x0) * static_cast<I>(dx)) / static_cast<float>(dx);
    if (x0 > W - 1) {
      x0 = W - 1;
      wx = 0.f;
    }
    x1 = min(x0 + 1, W - 1);
  }
  const int o00 = (y0 * W + x0) * 4, o01 = (y0 * W + x1) * 4, o10 = (y1 * W + x0) * 4, o11 = (y1 * W + x1) * 4;
  const size_t in_step = static_cast<size_t>(B) * Pin * 4, out_step = static_cast<size_t>(B) * Pout * 4;
  const bool pad_col = ox == OW - 1 && Pout > OH * OW;  // an odd plane carries one extra pixel: keep it zero
  for (int base = oy_lo; base < oy_hi; base += kResizeRows) {
    const int cnt = min(kResizeRows, oy_hi - base);
    __syncthreads();  // the previous chunk's weights are no longer needed
    if (static_cast<int>(threadIdx.x) < cnt) {
      const I py = static_cast<I>(base + threadIdx.x) * static_cast<I>(ny);
      wy_s[threadIdx.x] = static_cast<float>(py - static_cast<I>(y0) * static_cast<I>(dy)) / static_cast<float>(dy);
    }
    __syncthreads();
    if (!active) continue;
    const T* plane = in + static_cast<size_t>(blockIdx.z) * Pin * 4;
    T* orow = out + static_cast<size_t>(blockIdx.z) * Pout * 4 + (static_cast<size_t>(base) * OW + ox) * 4;
    for (int s = 0; s < S; ++s, plane += in_step, orow += out_step) {
      const float4 a = Px<T>::load(plane + o00), c = Px<T>::load(plane + o01), d = Px<T>::load(plane + o10), e = Px<T>::load(plane + o11);
      const float4 top = make_float4(fmaf(c.x - a.x, wx, a.x), fmaf(c.y - a.y, wx, a.y), fmaf(c.z - a.z, wx, a.z), fmaf(c.w - a.w, wx, a.w));
      const float4 bot = make_float4(fmaf(e.x - d.x, wx, d.x), fmaf(e.y - d.y, wx, d.y), fmaf(e.z - d.z, wx, d.z), fmaf(e.w - d.w, wx, d.w));
      const float4 dif = make_float4(bot.x - top.x, bot.y - top.y, bot.z - top.z, bot.w - top.w);
      T* o = orow;
      for (int r = 0; r < cnt; ++r, o += static_cast<size_t>(OW) * 4) {
        const float wy = wy_s[r];
        Px<T>::store(o, make_float4(fmaf(dif.x, wy, top.x), fmaf(dif.y, wy, top.y), fmaf(dif.z, wy, top.z), fmaf(dif.w, wy, top.w)));
      }
      if (pad_col && base + cnt == OH) Px<T>::store(o - static_cast<size_t>(OW) * 4 + 4, make_float4(0.f, 0.f, 0.f, 0.f));
    }
  }
}

// The same straight into the caller's NHWC tensor (fp16).  A warp owns 28 neighbouring groups of four values of an output row
// (group k: values 4k .. 4k + 3 of the row's OW * C), walks down the source rows [y_lo, y_hi), interpolates its groups along x
// once per source row and stores them in every output row of that interval, 8 bytes per lane.  Rows start on any half, so the
// groups stored start `s` values later, on a 32-byte boundary, with values of up to four lanes further on (hence 28): a warp
// then writes whole sectors only.  513x513x21 x 16 images (177 MB): 49 + 88 us as two kernels, 67 us so (46 M warp
// instructions, issue slots 60 % busy: bound by issue; 82 us with stores of two values on 4-byte boundaries and one source
// row per warp).  Values are those of the two kernels one after the other.
template <typename I>
__global__ void __launch_bounds__(128) resize_nhwc_kernel(const __half* __restrict__ in, __half* __restrict__ out, int B, int C, int H, int W,
                                                          int Pin, int OH, int OW, int ny, int dy, int nx, int dx, int y_step) {
  pdl_launch_dependents();
  pdl_wait();
  const int b = blockIdx.z, lane = threadIdx.x & 31;
  const int n = OW * C;                                                       // values of an output row
  const int k = (blockIdx.x * 4 + (static_cast<int>(threadIdx.x) >> 5)) * 28 + lane;  // this lane's group
  const int y_lo = blockIdx.y * y_step, y_hi = min(H, y_lo + y_step);
  const bool inner = k - lane >= 4 && 4 * (k - lane + 32) + 16 <= n;  // no group of the warp meets an end of the row
  const __half* p0[4];  // the group's source values in row 0: left neighbour, and how far the right one is
  int right[4];
  float wx[4];
  int ox = 4 * k / C, c = 4 * k - ox * C;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const bool in_row = 4 * k + e < n;
    const I qx = static_cast<I>(in_row ? ox : 0) * static_cast<I>(nx);
    int x0 = static_cast<int>(qx / static_cast<I>(dx));
    wx[e] = static_cast<float>(qx - static_cast<I>(x0) * static_cast<I>(dx)) / static_cast<float>(dx);
    if (x0 > W - 1) {
      x0 = W - 1;
      wx[e] = 0.f;
    }
    right[e] = x0 + 1 < W ? 4 : 0;
    const int ch = in_row ? c : 0;
    p0[e] = in + (static_cast<size_t>(ch >> 2) * B + b) * Pin * 4 + (ch & 3) + x0 * 4;
    if (++c == C) {
      c = 0;
      ++ox;
    }
  }
  __half raw[4][2];  // of the row below the current one
  float bot[4];
  auto fetch = [&](int y) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const __half* p = p0[e] + static_cast<size_t>(y) * W * 4;
      raw[e][0] = __ldg(p);
      raw[e][1] = __ldg(p + right[e]);
    }
  };
  auto along_x = [&]() {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float l = __half2float(raw[e][0]), r = __half2float(raw[e][1]);
      bot[e] = fmaf(r - l, wx[e], l);
    }
  };
  fetch(y_lo);
  along_x();
  fetch(min(y_lo + 1, H - 1));
  for (int y0 = y_lo; y0 < y_hi; ++y0) {
    const float top[4] = {bot[0], bot[1], bot[2], bot[3]};
    along_x();
    const float dif[4] = {bot[0] - top[0], bot[1] - top[1], bot[2] - top[2], bot[3] - top[3]};
    if (y0 + 1 < y_hi) fetch(min(y0 + 2, H - 1));
    // output rows oy with floor(oy * ny / dy) == y0
    int oy_lo = 0, oy_hi = y0 == 0 ? OH : 0;
    if (ny != 0) {
      oy_lo = static_cast<int>((static_cast<I>(y0) * static_cast<I>(dy) + static_cast<I>(ny - 1)) / static_cast<I>(ny));
      const I hi = (static_cast<I>(y0 + 1) * static_cast<I>(dy) + static_cast<I>(ny - 1)) / static_cast<I>(ny);
      oy_hi = hi > static_cast<I>(OH) ? OH : static_cast<int>(hi);
    }
    for (int base = oy_lo; base < oy_hi; base += 32) {
      const int cnt = min(32, oy_hi - base);
      const I py = static_cast<I>(base + lane) * static_cast<I>(ny);
      const float wy_lane = static_cast<float>(py - static_cast<I>(y0) * static_cast<I>(dy)) / static_cast<float>(dy);
      const size_t first = (static_cast<size_t>(b) * OH + base) * n;  // the row's first value
      __half* row = out + first + 4 * k;
      unsigned s = static_cast<unsigned>(-static_cast<long long>(first)) & 15u;  // values before the row's first 32-byte boundary
      auto rows = [&](auto edge) {
#pragma unroll 2
        for (int r = 0; r < cnt; ++r, row += n, s = (s - static_cast<unsigned>(n)) & 15u) {
          const float wy = __shfl_sync(0xffffffffu, wy_lane, r);
          const __half2 h0 = __floats2half2_rn(fmaf(dif[0], wy, top[0]), fmaf(dif[1], wy, top[1]));
          const __half2 h1 = __floats2half2_rn(fmaf(dif[2], wy, top[2]), fmaf(dif[3], wy, top[3]));
          const unsigned o0 = *reinterpret_cast<const unsigned*>(&h0), o1 = *reinterpret_cast<const unsigned*>(&h1);
          const unsigned d = s >> 2;
          const unsigned q0 = __shfl_down_sync(0xffffffffu, o0, d), q1 = __shfl_down_sync(0xffffffffu, o1, d);
          const unsigned n0 = __shfl_down_sync(0xffffffffu, o0, d + 1), n1 = __shfl_down_sync(0xffffffffu, o1, d + 1);
          const unsigned a0 = s & 2 ? q1 : q0, a1 = s & 2 ? n0 : q1, a2 = s & 2 ? n1 : n0, sh = (s & 1) * 16;
          const unsigned w0 = __funnelshift_r(a0, a1, sh), w1 = __funnelshift_r(a1, a2, sh);
          if (lane >= 28) continue;
          unsigned short* at = reinterpret_cast<unsigned short*>(row + s);
          const int left = decltype(edge)::value ? n - 4 * k - static_cast<int>(s) : 4;  // values of the row from this group on
          if (left >= 4) {
            *reinterpret_cast<uint2*>(at) = make_uint2(w0, w1);
          } else if (left > 0) {
            at[0] = static_cast<unsigned short>(w0);
            if (left > 1) at[1] = static_cast<unsigned short>(w0 >> 16);
            if (left > 2) at[2] = static_cast<unsigned short>(w1);
          }
          if (decltype(edge)::value && 4 * k < static_cast<int>(s)) {  // values before the first boundary
            unsigned short* f = reinterpret_cast<unsigned short*>(row);
            const int head = min(static_cast<int>(s), n) - 4 * k;
            if (head > 0) f[0] = static_cast<unsigned short>(o0);
            if (head > 1) f[1] = static_cast<unsigned short>(o0 >> 16);
            if (head > 2) f[2] = static_cast<unsigned short>(o1);
            if (head > 3) f[3] = static_cast<unsigned short>(o1 >> 16);
          }
        }
      };
      if (inner) rows(std::false_type{});
      else rows(std::true_type{});
    }
  }
}

ConvGeom geom(const LaunchRec& r) {
  ConvGeom g;
  g.B = r.B;
  g.H = r.H;
  g.W = r.W;
  g.Sin = slices(r.C);
  g.Pin = plane_pixels(r.H, r.W);
  g.Ho = r.Ho;
  g.Wo = r.Wo;
  g.Sout = slices(r.Co);
  g.Pout = plane_pixels(r.Ho, r.Wo);
  g.kh = r.kh;
  g.kw = r.kw;
  g.sh = r.sh;
  g.sw = r.sw;
  g.dh = r.dh;
  g.dw = r.dw;
  g.pt = r.pt;
  g.pl = r.pl;
  return g;
}

inline unsigned blocks_for(size_t n, unsigned per) { return static_cast<unsigned>((n + per - 1) / per); }

}  // namespace

#define GI_BY_STORAGE(call_h, call_f) \
  do {                                \
    if (storage == GI_F16) {          \
      call_h;                         \
    } else {                          \
      call_f;                         \
    }                                 \
  } while (0)

int launch_pack(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int S = slices(r.C), P = plane_pixels(r.H, r.W), HW = r.H * r.W;
  if (storage == GI_F16 && r.C == 3 && HW % 4 == 0 && r.B <= 65535) {
    // P == HW here (no padding pixel), one slice: the planes of the images are back to back
    const int quads = HW / 4;
    launch_pdl(pack3_f16_kernel, dim3(blocks_for(quads, 256), r.B), 256, 0, st, static_cast<const uint2*>(p.in0),
               static_cast<uint4*>(p.out), quads);
    return static_cast<int>(cudaGetLastError());
  }
  const long long planes = static_cast<long long>(S) * r.B;
  if (planes > 2147483647LL) return static_cast<int>(cudaErrorInvalidConfiguration);
  const dim3 grid(blocks_for(P, 256), static_cast<unsigned>(planes < 65535 ? planes : 65535));
  GI_BY_STORAGE((launch_pdl(pack_kernel<__half>, grid, 256, 0, st, static_cast<const __half*>(p.in0), static_cast<__half*>(p.out),
                            r.B, HW, r.C, P, S)),
                (launch_pdl(pack_kernel<float>, grid, 256, 0, st, static_cast<const float*>(p.in0), static_cast<float*>(p.out), r.B,
                            HW, r.C, P, S)));
  return static_cast<int>(cudaGetLastError());
}

int launch_unpack(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int S = slices(r.C), P = plane_pixels(r.H, r.W), HW = r.H * r.W;
  const size_t total = static_cast<size_t>(S) * r.B * HW;
  if (storage == GI_F16 && r.B <= 65535 && static_cast<size_t>(r.C) * 256 <= 48 * 1024) {
    launch_pdl(unpack_f16_kernel, dim3(blocks_for(HW, 128), r.B), 128, static_cast<size_t>(r.C) * 256, st,
               static_cast<const __half*>(p.in0), static_cast<__half*>(p.out), r.B, HW, r.C, P, S);
    return static_cast<int>(cudaGetLastError());
  }
  GI_BY_STORAGE((launch_pdl(unpack_kernel<__half>, blocks_for(total, 256), 256, 0, st, static_cast<const __half*>(p.in0),
                                                                               static_cast<__half*>(p.out), r.B, HW, r.C, P, S)),
                (launch_pdl(unpack_kernel<float>, blocks_for(total, 256), 256, 0, st, static_cast<const float*>(p.in0),
                                                                              static_cast<float*>(p.out), r.B, HW, r.C, P, S)));
  return static_cast<int>(cudaGetLastError());
}

template <typename T>
static int conv_dispatch(const LaunchRec& r, const Ptrs& p, cudaStream_t st) {
  const ConvGeom g = geom(r);
  const long long tiles = (static_cast<long long>(g.B) * g.Pout + 31) / 32;
  const int groups = (g.Sout + 7) / 8, units = g.kh * g.kw * g.Sin;
  // split the sum until there are 16 warps per SM or a warp has 4 units left: 7x7 960 -> 160 at batch 2, 225 -> 16 us (event pair around one launch)
  int kw = 1;
  while (kw < kConvMaxSplit && tiles * groups * kw < 148 * 16 && units >= kw * 8) kw *= 2;
  const int warps = kw > 8 ? kw : 8, tpc = warps / kw;
  const size_t smem = static_cast<size_t>(warps) * kConvWarpBytes;
  static bool attr_done_dev[kMaxDevices] = {};
  bool& attr_done = attr_done_dev[current_device_slot()];
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(conv_simt_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kConvMaxSplit * kConvWarpBytes);
    if (e != cudaSuccess) return static_cast<int>(e);
    attr_done = true;
  }
  const long long blocks = (tiles + tpc - 1) / tpc;
  if (blocks > 2147483647LL || groups > 65535) return static_cast<int>(cudaErrorInvalidConfiguration);
  return static_cast<int>(launch_pdl(conv_simt_kernel<T>, dim3(static_cast<unsigned>(blocks), groups), 32 * warps, smem, st,
                                     static_cast<const T*>(p.in0), static_cast<const float4*>(p.wts), static_cast<const float*>(p.bias),
                                     static_cast<const T*>(p.res), static_cast<T*>(p.out), g, r.ep, kw));
}

int launch_conv_simt(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return storage == GI_F16 ? conv_dispatch<__half>(r, p, st) : conv_dispatch<float>(r, p, st);
}

int launch_depthwise(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (r.dw_staged) return launch_depthwise_f16(r, p, stream);
  if (r.B > 65535) return static_cast<int>(cudaErrorInvalidConfiguration);
  const ConvGeom g = geom(r);
  const dim3 grid(blocks_for(g.Pout, 128), g.Sout, r.B);
  GI_BY_STORAGE((launch_pdl(depthwise_kernel<__half>, grid, 128, 0, st, static_cast<const __half*>(p.in0), static_cast<const float*>(p.wts),
                                                               static_cast<const float*>(p.bias), static_cast<const __half*>(p.res),
                                                               static_cast<__half*>(p.out), g, r.ep)),
                (launch_pdl(depthwise_kernel<float>, grid, 128, 0, st, static_cast<const float*>(p.in0), static_cast<const float*>(p.wts),
                                                              static_cast<const float*>(p.bias), static_cast<const float*>(p.res),
                                                              static_cast<float*>(p.out), g, r.ep)));
  return static_cast<int>(cudaGetLastError());
}

int launch_eltwise(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t n_px = static_cast<size_t>(slices(r.Co)) * r.B * plane_pixels(r.Ho, r.Wo);
  GI_BY_STORAGE((launch_pdl(eltwise_kernel<__half>, blocks_for(n_px, 256), 256, 0, st, static_cast<const __half*>(p.in0),
                                                                               static_cast<const __half*>(p.in1),
                                                                               static_cast<__half*>(p.out), n_px, r.ep)),
                (launch_pdl(eltwise_kernel<float>, blocks_for(n_px, 256), 256, 0, st, static_cast<const float*>(p.in0),
                                                                              static_cast<const float*>(p.in1),
                                                                              static_cast<float*>(p.out), n_px, r.ep)));
  return static_cast<int>(cudaGetLastError());
}

int launch_concat(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int P = plane_pixels(r.Ho, r.Wo), sout = slices(r.Co);
  const size_t n_px = static_cast<size_t>(r.B) * P;
  if (sout > 65535) return static_cast<int>(cudaErrorInvalidConfiguration);
  const dim3 grid(blocks_for(n_px, 256), sout);
  const int Ca = r.C, Cb = r.Co - r.C;
  GI_BY_STORAGE((launch_pdl(concat_kernel<__half>, grid, 256, 0, st, static_cast<const __half*>(p.in0), static_cast<const __half*>(p.in1),
                            static_cast<__half*>(p.out), n_px, P, r.Ho * r.Wo, Ca, Cb)),
                (launch_pdl(concat_kernel<float>, grid, 256, 0, st, static_cast<const float*>(p.in0), static_cast<const float*>(p.in1),
                            static_cast<float*>(p.out), n_px, P, r.Ho * r.Wo, Ca, Cb)));
  return static_cast<int>(cudaGetLastError());
}

int launch_pool(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int planes = slices(r.C) * r.B, HW = r.H * r.W, Pin = plane_pixels(r.H, r.W), Pout = plane_pixels(1, 1);
  // a whole warp for a plane of 128 pixels and more while eight lanes each would leave SMs without work (64 images of 16x16x64,
  // 32 CTAs: 10.2 us between events, 128 CTAs: 7.0)
  const bool warp = HW >= 128 && planes <= 148 * 32;
  const unsigned blocks = blocks_for(static_cast<size_t>(planes) * (warp ? 32 : 8), 256);
#define GI_POOL(T, L) (launch_pdl(pool_kernel<T, L>, blocks, 256, 0, st, static_cast<const T*>(p.in0), static_cast<T*>(p.out), planes, HW, Pin, Pout))
  if (warp) {
    GI_BY_STORAGE(GI_POOL(__half, 32), GI_POOL(float, 32));
  } else {
    GI_BY_STORAGE(GI_POOL(__half, 8), GI_POOL(float, 8));
  }
#undef GI_POOL
  return static_cast<int>(cudaGetLastError());
}

int launch_resize(const LaunchRec& r, const Ptrs& p, int storage, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int ny, dy, nx, dx;
  if (r.align_corners) {
    ny = r.Ho > 1 ? r.H - 1 : 0;
    dy = r.Ho > 1 ? r.Ho - 1 : 1;
    nx = r.Wo > 1 ? r.W - 1 : 0;
    dx = r.Wo > 1 ? r.Wo - 1 : 1;
  } else {
    ny = r.H;
    dy = r.Ho;
    nx = r.W;
    dx = r.Wo;
  }
  const int Pout = plane_pixels(r.Ho, r.Wo), Pin = plane_pixels(r.H, r.W);
  if (r.H > 65535 || r.B > 65535) return static_cast<int>(cudaErrorInvalidConfiguration);
  const bool narrow = (static_cast<long long>(r.Ho) + 1) * ny + static_cast<long long>(r.H + 1) * dy < (1LL << 31) &&
                      static_cast<long long>(r.Wo) * nx < (1LL << 31);
  if (r.nhwc_out) {
    const unsigned gx = blocks_for((static_cast<size_t>(r.Wo) * r.C + 3) / 4, 4 * 28);
    // source rows per warp: as many as leave three waves of the eight CTAs an SM holds (1200 CTAs, one wave and a bit: 104 us)
    const int y_step = static_cast<int>(std::max<long long>(1, std::min<long long>(8, static_cast<long long>(gx) * r.H * r.B / (148 * 24))));
    const dim3 grid(gx, blocks_for(r.H, y_step), r.B);
    const __half* in = static_cast<const __half*>(p.in0);
    __half* out = static_cast<__half*>(p.out);
    launch_pdl(narrow ? resize_nhwc_kernel<unsigned> : resize_nhwc_kernel<unsigned long long>, grid, 128, 0, st, in, out, r.B, r.C, r.H, r.W, Pin,
               r.Ho, r.Wo, ny, dy, nx, dx, y_step);
    return static_cast<int>(cudaGetLastError());
  }
  const dim3 grid(blocks_for(r.Wo, 128), r.H, r.B);
#define GI_RESIZE(T, I)                                                                                                       \
  launch_pdl(resize_kernel<T, I>, grid, 128, 0, st, static_cast<const T*>(p.in0), static_cast<T*>(p.out), r.B, slices(r.C), r.H, r.W, \
             Pin, r.Ho, r.Wo, Pout, ny, dy, nx, dx)
  if (narrow) {
    GI_BY_STORAGE(GI_RESIZE(__half, unsigned), GI_RESIZE(float, unsigned));
  } else {
    GI_BY_STORAGE(GI_RESIZE(__half, unsigned long long), GI_RESIZE(float, unsigned long long));
  }
#undef GI_RESIZE
  return static_cast<int>(cudaGetLastError());
}

}  // namespace gi
