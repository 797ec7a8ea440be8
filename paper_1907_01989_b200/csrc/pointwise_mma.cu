// Pointwise (1x1) convolution for launches that are bound by latency, not by a pipe: those whose tiles of 32 pixels x 32
// channels fit on the chip at once - the late layers of a network at batch 1 to 32, its classifier, a segmentation head.
//
// The tcgen05 kernel for such layers (pointwise_ts.cu) pays for tensor memory and a transfer step per chunk, and walks all
// input channels of 128 pixels in one chain.  Here the pixel-slices go from shared memory straight into the operand registers
// of mma.sync.m16n8k16 (a slice of 4 channels is 8 bytes: lane t of a quad takes slice t of 16 channels, the weights are
// permuted to match when they are packed), and eight warps split the input channels of ONE tile, so that a warp's chain is an
// eighth of the sum; their partial sums meet in shared memory and are added in a fixed order.  One thread requests a stage
// with one bulk copy (weights, before the previous kernel has finished) and one tiled copy (pixels; 36 instead of 32 of them,
// which spreads the slices over the banks).  (Copies of a slice or of 16 bytes each, by 32 lanes or 256 threads, took 1 us a
// stage.)  The results leave the registers as whole pixel-slices, or - at the end of a graph - as the caller's NHWC rows, which
// saves the layout conversion's launch.
//
// Measured inside chains of launches against pointwise_ts.cu: 7x7 960 -> 320 at batch 1 2.1 us less, 320 -> 1280 1.4, 33x33
// 960 -> 160 2.1, 1280 -> 1001 at batch 8 1.8 (and the 3 us of the layout conversion).  Larger tiles lose to the tcgen05
// kernels wherever these 32 x 32 ones do not fit (14x14 512 -> 512 at batch 64: 128 x 128 tiles 32 us, pointwise_mm.cu 12).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

#include "kernels.h"
#include "mma_frag.cuh"
#include "pdl.cuh"
#include "sm100_ptx.cuh"
#include "tma_host.h"

namespace gi {
namespace {

using namespace ptx;
using namespace frag;

constexpr int kThreads = 256;  // threads that compute; one more warp issues the copies
constexpr int kMaxStages = 12;
constexpr int kBarBytes = 2 * kMaxStages * 8 + 16;
constexpr unsigned kWaitNs = 1000000000u;
// Shared memory for stages: two CTAs on an SM, or (0.5 % of a whole MobileNetV2 at batch 1 and 8) up to all twelve where no
// SM gets a second one.
constexpr int kSmemTwo = 109 * 1024, kSmemOne = 220 * 1024;
constexpr int kTile = 32;             // pixels, and output channels, of a tile
constexpr int kSplit = 8;             // warps that share a tile's sum, one 16-channel step of a stage each
constexpr int kTilePx = kTile + 4;    // pixels copied per slice: 32 bytes modulo 128 between slices, so that the four slices x
                                      // four pixels half a warp reads lie in different banks
constexpr int kSlicePitch = kTilePx * 8;
constexpr int kABytes = kSplit * 4 * kSlicePitch, kWBytes = kTile / 16 * kSplit * 512, kStage = kABytes + kWBytes;
constexpr int kSumBytes = kSplit * 4096;

struct Params {
  const __half* res;
  __half* out;
  const unsigned char* wts;  // [tile][stage][16 output channels][16 input channels][lane][16 bytes]
  const float* bias;
  long long out_sl;         // elements between slices
  int rows;                 // pixels (stored ones, both of a padded pair included)
  int k16, sout;
  int n_tiles, stages;
  int act_pre, has_res, act_post;
  int nhwc, C, P, HW;       // caller's layout: channels, stored and real pixels per image
  unsigned mul_p;           // ceil(2^32 / P)
};

__device__ unsigned g_pm_error = 0;

// One pixel-slice of the result: bias, activation, residual, activation, fp16; stored as a slice or into the caller's tensor.
__device__ __forceinline__ void finish(const Params& p, int row, int slice, const float4& bias, float v0, float v1, float v2, float v3) {
  if (row >= p.rows || slice >= p.sout) return;
  v0 = act_f(v0 + bias.x, p.act_pre);
  v1 = act_f(v1 + bias.y, p.act_pre);
  v2 = act_f(v2 + bias.z, p.act_pre);
  v3 = act_f(v3 + bias.w, p.act_pre);
  const long long at = slice * p.out_sl + static_cast<long long>(row) * 4;
  if (p.has_res) {
    const uint2 r = *reinterpret_cast<const uint2*>(p.res + at);
    const float2 r01 = __half22float2(*reinterpret_cast<const __half2*>(&r.x));
    const float2 r23 = __half22float2(*reinterpret_cast<const __half2*>(&r.y));
    v0 = act_f(v0 + r01.x, p.act_post);
    v1 = act_f(v1 + r01.y, p.act_post);
    v2 = act_f(v2 + r23.x, p.act_post);
    v3 = act_f(v3 + r23.y, p.act_post);
  }
  const unsigned lo = pack_f16x2<false>(v0, v1), hi = pack_f16x2<false>(v2, v3);
  if (!p.nhwc) {
    *reinterpret_cast<uint2*>(p.out + at) = make_uint2(lo, hi);
    return;
  }
  long long px = row;
  if (p.P != p.HW) {  // skip the second pixel of an odd plane's last pair
    const int img = static_cast<int>(__umulhi(static_cast<unsigned>(row), p.mul_p));
    const int in = row - img * p.P;
    if (in >= p.HW) return;
    px = static_cast<long long>(img) * p.HW + in;
  }
  unsigned short* dst = reinterpret_cast<unsigned short*>(p.out) + px * p.C + slice * 4;
  const int n = p.C - slice * 4;
  if (p.C % 4 == 0) {
    *reinterpret_cast<uint2*>(dst) = make_uint2(lo, hi);
  } else {
    dst[0] = static_cast<unsigned short>(lo);
    if (n > 1) dst[1] = static_cast<unsigned short>(lo >> 16);
    if (n > 2) dst[2] = static_cast<unsigned short>(hi);
    if (n > 3) dst[3] = static_cast<unsigned short>(hi >> 16);
  }
}

__global__ void __launch_bounds__(kThreads + 32, 2) pointwise_mma_kernel(const __grid_constant__ CUtensorMap map, const Params p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const unsigned smem = smem_u32(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int tm = blockIdx.x / p.n_tiles, tn = blockIdx.x - tm * p.n_tiles;
  const int row0 = tm * kTile, n_st = (p.k16 + kSplit - 1) / kSplit;
  const unsigned full = smem + p.stages * kStage, empty = full + kMaxStages * 8;
  volatile unsigned* abort_flag = reinterpret_cast<volatile unsigned*>(smem_raw + p.stages * kStage + 2 * kMaxStages * 8);

  pdl_launch_dependents();
  if (tid == 0) {
    prefetch_tensormap(&map);
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(full + i * 8, 1);
      mbar_init(empty + i * 8, kSplit);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  float acc[2][2][2][4];  // [16 pixels][16 channels]: two fragments
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i / 16][i / 8 % 2][i / 4 % 2][i % 4] = 0.0f;

  int asked = 0;  // stages the copying thread has requested
  if (warp == kSplit) {
    if (lane == 0) {
      auto load_w = [&](int st, int slot) {
        mbar_expect_tx(full + slot * 8, kStage);
        bulk_load(smem + slot * kStage + kABytes, p.wts + (static_cast<size_t>(tn) * n_st + st) * kWBytes, kWBytes, full + slot * 8);
      };
      auto load_a = [&](int st, int slot) { tma_load_2d(smem + slot * kStage, &map, row0, st * kSplit * 4, full + slot * 8); };
      const int ahead = min(p.stages, n_st);
      for (int st = 0; st < ahead; ++st) load_w(st, st);
      pdl_wait();
      for (int st = 0; st < ahead; ++st) load_a(st, st);
      asked = ahead;
      for (int slot = 0, round = 0; asked < n_st; ++asked) {
        if (!mbar_wait(empty + slot * 8, round & 1, abort_flag, kWaitNs, &g_pm_error, 1u)) break;
        load_w(asked, slot);
        load_a(asked, slot);
        if (++slot == p.stages) slot = 0, ++round;
      }
    }
  } else {
    pdl_wait();
#pragma unroll 1
    for (int st = 0, slot = 0, round = 0; st < n_st; ++st) {
      if (!mbar_wait_warp(full + slot * 8, round & 1, abort_flag, kWaitNs, &g_pm_error, 2u)) break;
      if (st * kSplit + warp < p.k16) {
        const unsigned a_at = smem + slot * kStage + (warp * 4 + t) * kSlicePitch + g * 8, b_at = smem + slot * kStage + kABytes + warp * 512 + lane * 16;
        unsigned a[2][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint2 v = lds64(a_at + i * 64);
          a[i >> 1][i & 1] = v.x;
          a[i >> 1][2 + (i & 1)] = v.y;
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint4 b = lds128(b_at + j * kSplit * 512);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            mma16816(acc[i][j][0], a[i], b.x, b.y);
            mma16816(acc[i][j][1], a[i], b.z, b.w);
          }
        }
      }
      __syncwarp();
      if (lane == 0 && st + p.stages < n_st) mbar_arrive(empty + slot * 8);
      if (++slot == p.stages) slot = 0, ++round;
    }
  }
  // a wait that ran out: the copies in flight land before the CTA leaves (bounded as well), nothing is stored
  if (__syncthreads_or(static_cast<int>(*abort_flag))) {
    for (int st = max(0, asked - p.stages); st < asked; ++st) {
      unsigned none = 0;
      mbar_wait(full + st % p.stages * 8, (st / p.stages) & 1, &none, kWaitNs, &g_pm_error, 4u);
    }
    return;
  }
  if (warp == kSplit) return;

  // the partial sums take the stages' place: [warp][granule of 16 pixels x 16 channels][fragment][lane].  Two warps add up a
  // granule, a row of 8 pixels each.
  const unsigned mine = smem + warp * 4096 + lane * 16;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int f = 0; f < 2; ++f) {
        const float(&v)[4] = acc[i][j][f];
        sts128(mine + (i * 2 + j) * 1024 + f * 512, __float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]), __float_as_uint(v[3]));
      }
  asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");  // the warps that compute
  const int gr = warp >> 1, half = warp & 1;
  const unsigned at = smem + gr * 1024 + lane * 16 + half * 8;
  float2 s0 = make_float2(0.0f, 0.0f), s1 = s0;
#pragma unroll
  for (int k = 0; k < kSplit; ++k) {
    const uint2 v0 = lds64(at + k * 4096), v1 = lds64(at + k * 4096 + 512);
    s0.x += __uint_as_float(v0.x);
    s0.y += __uint_as_float(v0.y);
    s1.x += __uint_as_float(v1.x);
    s1.y += __uint_as_float(v1.y);
  }
  const int slice = (tn * 2 + (gr & 1)) * 4 + t;
  const float4 b = reinterpret_cast<const float4*>(p.bias)[slice];
  finish(p, row0 + (gr >> 1) * 16 + half * 8 + g, slice, b, s0.x, s0.y, s1.x, s1.y);
}

// rows of the operand: stored pixels
long long rows_of(const LaunchRec& r) { return static_cast<long long>(r.B) * plane_pixels(r.H, r.W); }
long long tiles_of(const LaunchRec& r) { return ((rows_of(r) + kTile - 1) / kTile) * ((r.Co + kTile - 1) / kTile); }

}  // namespace

// Two CTAs share an SM: with more tiles than that the kernel loses (21 images of 7x7: 960 -> 160, 165 tiles, 2.1 us faster than
// pointwise_ts.cu, 960 -> 320, 330 tiles, 2.2 us slower; 33x33 320 -> 256, 280 tiles, 0.5 us faster).
bool pointwise_mma_wanted(const LaunchRec& r) { return tiles_of(r) <= 2 * 148; }

// w: [cout][cin]; the weights of a tile's stage are one run of bytes
void pointwise_mma_pack(const float* w, const float* bias, int cin, int cout, std::vector<uint8_t>* blob, LaunchRec* r) {
  const int nb = kTile / 16, n_tiles = (cout + kTile - 1) / kTile, n_st = (cin + 16 * kSplit - 1) / (16 * kSplit);
  const uint64_t woff = round_up_u64(blob->size(), 256), wbytes = static_cast<uint64_t>(n_tiles) * n_st * kWBytes;
  const uint64_t boff = round_up_u64(woff + wbytes, 256);
  blob->resize(boff + static_cast<size_t>(n_tiles) * nb * 16 * sizeof(float), 0);
  uint16_t* q = reinterpret_cast<uint16_t*>(blob->data() + woff);
  for (int tile = 0; tile < n_tiles; ++tile)
    for (int st = 0; st < n_st; ++st)
      for (int j = tile * nb; j < (tile + 1) * nb; ++j)
        for (int kk = st * kSplit; kk < (st + 1) * kSplit; ++kk)
          for (int lane = 0; lane < 32; ++lane)
            for (int e = 0; e < 8; ++e, ++q) {  // {fragment 0: b0, b1; fragment 1: b0, b1}
              const int f = e >> 2, hi8 = (e >> 1) & 1, lo = e & 1, n = lane >> 2, t = lane & 3;
              const int co = channel_of(j, f, n), ci = 16 * kk + 4 * t + 2 * hi8 + lo;
              if (co < cout && ci < cin) *q = f32_to_f16_rne(w[static_cast<size_t>(co) * cin + ci]);
            }
  std::memcpy(blob->data() + boff, bias, static_cast<size_t>(cout) * sizeof(float));
  r->wts = Loc{W_WEIGHTS, 0, woff};
  r->bias = Loc{W_WEIGHTS, 0, boff};
  r->wts_bytes = wbytes;
}

unsigned int pointwise_mma_error_word(int* cuda_err) {
  unsigned int v = 0;
  const cudaError_t e = cudaMemcpyFromSymbol(&v, g_pm_error, sizeof v);
  if (cuda_err) *cuda_err = static_cast<int>(e);
  return v;
}

int launch_pointwise_mma(const LaunchRec& r, const Ptrs& ptr, void** state, int launch_index, void* stream) {
  const int P = plane_pixels(r.H, r.W);
  Params p{};
  p.res = static_cast<const __half*>(ptr.res);
  p.out = static_cast<__half*>(ptr.out);
  p.wts = static_cast<const unsigned char*>(ptr.wts);
  p.bias = static_cast<const float*>(ptr.bias);
  p.out_sl = static_cast<long long>(r.B) * P * 4;
  p.rows = static_cast<int>(rows_of(r));
  p.k16 = (r.C + 15) / 16;
  p.sout = slices(r.Co);
  p.act_pre = r.ep.act_pre;
  p.has_res = r.ep.has_res;
  p.act_post = r.ep.act_post;
  p.nhwc = r.nhwc_out;
  p.C = r.Co;
  p.P = P;
  p.HW = r.H * r.W;
  p.mul_p = static_cast<unsigned>((0x100000000ull + P - 1) / P);  // exact: at most 296 tiles of 32 rows
  p.n_tiles = (r.Co + kTile - 1) / kTile;
  const int n_st = (p.k16 + kSplit - 1) / kSplit;
  p.stages = std::min({kMaxStages, n_st, (tiles_of(r) <= 148 ? kSmemOne : kSmemTwo) / kStage});
  while (p.stages * kStage < kSumBytes) ++p.stages;
  CUtensorMap map;
  const int err = map_cache_lookup(state, launch_index, ptr.in0, &map, [&](CUtensorMap* m) {
    return encode_plane_map(m, ptr.in0, static_cast<unsigned long long>(p.rows), slices(r.C), kTilePx, kSplit * 4);
  });
  if (err != 0) return err;
  static bool attr_done_dev[kMaxDevices] = {};
  bool& attr_done = attr_done_dev[current_device_slot()];
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(pointwise_mma_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemOne + kBarBytes);
    if (e != cudaSuccess) return static_cast<int>(e);
    attr_done = true;
  }
  return static_cast<int>(launch_pdl(pointwise_mma_kernel, dim3(static_cast<unsigned>(tiles_of(r))), dim3(kThreads + 32),
                                     p.stages * kStage + kBarBytes, static_cast<cudaStream_t>(stream), map, p));
}

}  // namespace gi
