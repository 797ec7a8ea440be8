// k x k convolution (k = 1 .. 3) with few channels, alone or as a whole fire module, as ONE kernel (fp16 storage):
//   k x k                                             input in slices, or the caller's NHWC image of at most 4 channels
//   1x1 squeeze -> { 1x1 expand, k x k expand } -> concatenation (-> + residual)
// A fire module's two expansions read the same squeezed tensor: they are one convolution whose output channels are both
// parts', the 1x1 part with zero weights outside the window's middle, so that the concatenation is where the results are stored
// and costs nothing, at any channel count.  The squeezed tensor never leaves the SM (rounded to fp16 where a kernel of its own
// would have stored it; beyond the range of fp16 it is the largest finite value, not infinity, so that the zero weights around a
// 1x1's middle stay zeros).
//
// A unit is a tile of output pixels of one image.  Its input is staged as [pixel][channels] rows of 16-byte units of 8
// channels; all sums are mma.sync.m16n8k16.  The K axis is (window position, 8 channels) taken in pairs: the two halves of an
// ldmatrix row set are two such units with offsets of their own (a small table), so that 8 squeezed channels fill a step with
// two window positions instead of half a step with one, and stride, dilation and window cost addresses only.  A warp takes 16
// or 32 output pixels x all output channels (at most 64).
//
// What bounds it: at batch 1 the chain of one tile, 3 to 4 us (conv_tc.cu, which gathers 8-byte slices per window position and
// waits for three roles to hand over: 4.4 to 6.9).  At batch 64 the instructions of staging and squeezing: a module on 48x48
// 32 -> 8 -> 32 takes 11.6 us, where its four launches took 29; 48x48 32 -> 48, stride 3, 6.5 against 8.8.  With a large output
// plane behind few inputs (batch 256, 96x96 3 -> 24) or a long sum at a large batch conv_tc.cu is the faster one.
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>

#include "kernels.h"
#include "mma_frag.cuh"
#include "pdl.cuh"
#include "sm100_ptx.cuh"

namespace gi {
namespace {

using namespace ptx;
using namespace frag;

constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kSmemTwo = 110 * 1024;  // a CTA's share of an SM's shared memory when two fit
constexpr unsigned kWaitNs = 1000000000u;

__device__ unsigned g_cm_error = 0;

struct Params {
  const __half* in;
  const __half* res;
  __half* out;
  const unsigned char* wts;
  int H, W, Ho, Wo, C;
  int kw, stride, dil, pad_t, pad_l;
  int tw, th, tiles_x, tiles_y, units;
  int cols, n_in, mt;       // staged pixels per row, of a tile, in groups of 16
  int n_out;                // output pixels of a tile
  int sin;                  // input slices
  int u_in, x_pitch;        // 16-byte units of an input pixel, bytes between pixels
  int u_z, z_pitch;         // the same of the tensor the window walks over (the input or the squeezed one)
  int n_units, steps, sq_steps;
  long long in_sl, out_sl;  // elements between slices
  int in_img, out_img;      // ... between images
  int nhwc;                 // the input is the caller's NHWC image
  int sout, wts_bytes;
  unsigned off_conv, off_bias, off_sqb, off_tab, off_x, off_z, off_bar;
  unsigned mul_cols, mul_tw, mul_per, mul_tx;
  int act_sq, act_pre, has_res, act_post;
  int pad_px;               // an odd plane holds one more pixel: zero it
};

__device__ __forceinline__ float round_f16(float v) { return __half2float(__float2half_rn(v)); }

// SQ: the 1x1 squeeze in front.  NB: 16-channel output blocks.  MG: groups of 16 output pixels a warp takes at a time.
template <int NB, int MG, bool SQ>
__global__ void __launch_bounds__(kThreads, NB * MG > 4 ? 2 : 3) conv_mma_kernel(const Params p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const unsigned smem = smem_u32(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const unsigned bar = smem + p.off_bar, xs = smem + p.off_x, zs = SQ ? smem + p.off_z : xs;
  volatile unsigned* abort_flag = reinterpret_cast<volatile unsigned*>(smem_raw + p.off_bar + 8);

  pdl_launch_dependents();
  if (tid == 0) {
    mbar_init(bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(bar, p.wts_bytes);
    bulk_load(smem, p.wts, p.wts_bytes, bar);
  }
  // where the K units lie relative to a window's first pixel
  for (int i = tid; i < 2 * p.steps; i += kThreads) {
    const int tap = i / p.u_z, ky = tap / p.kw;
    sts32(smem + p.off_tab + i * 4, i < p.n_units ? ((ky * p.cols + tap - ky * p.kw) * p.dil * p.z_pitch + (i - tap * p.u_z) * 16) : 0);
  }
  // bytes behind the last pixel that a half of a step without weights reads
  if (tid < 4) sts32(xs + p.mt * 16 * p.x_pitch + tid * 4, 0u);
  __syncthreads();
  pdl_wait();
  // a wait that ran out: nothing is stored, and the weights' copy lands before the CTA leaves (bounded as well)
  if (!__syncthreads_and(mbar_wait(bar, 0u, abort_flag, kWaitNs, &g_cm_error, 1u))) {
    unsigned none = 0;
    if (tid == 0) mbar_wait(bar, 0u, &none, kWaitNs, &g_cm_error, 4u);
    return;
  }

  const int per = p.tiles_x * p.tiles_y;
  for (int unit = blockIdx.x; unit < p.units; unit += gridDim.x) {
    const int img = per == 1 ? unit : div_by(unit, p.mul_per);
    const int rest = unit - img * per, ty = p.tiles_x == 1 ? rest : div_by(rest, p.mul_tx);
    const int y0 = ty * p.th, x0 = (rest - ty * p.tiles_x) * p.tw;
    const int iy0 = y0 * p.stride - p.pad_t, ix0 = x0 * p.stride - p.pad_l;
    if (unit != static_cast<int>(blockIdx.x)) __syncthreads();  // the tiles are free

    // ---- stage the input tile
    for (int i = tid; i < p.mt * 16; i += kThreads) {
      const int r = div_by(i, p.mul_cols), c = i - r * p.cols, y = iy0 + r, x = ix0 + c;
      const bool in = i < p.n_in && static_cast<unsigned>(y) < static_cast<unsigned>(p.H) && static_cast<unsigned>(x) < static_cast<unsigned>(p.W);
      const unsigned dst = xs + i * p.x_pitch;
      if (p.nhwc) {
        const unsigned short* src = reinterpret_cast<const unsigned short*>(p.in) + (static_cast<long long>(img) * p.in_img + (y * p.W + x) * p.C);
        unsigned v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = in && k < p.C ? __ldg(src + k) : 0u;
        sts128(dst, v[0] | v[1] << 16, v[2] | v[3] << 16, 0u, 0u);
      } else {
        const uint2* src = reinterpret_cast<const uint2*>(p.in + static_cast<long long>(img) * p.in_img + (y * p.W + x) * 4);
        for (int s = 0; s < 2 * p.u_in; s += 4) {
          uint2 v[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            v[k] = make_uint2(0u, 0u);
            if (in && s + k < p.sin) v[k] = *(src + (s + k) * (p.in_sl / 4));
          }
#pragma unroll
          for (int k = 0; k < 4; k += 2)
            if (s + k < 2 * p.u_in) sts128(dst + (s + k) * 8, v[k].x, v[k].y, v[k + 1].x, v[k + 1].y);
        }
      }
    }
    __syncthreads();

    // ---- squeeze: every pixel of the tile, zero outside the image (the window's padding)
    if (SQ) {
      const uint4 bq = lds128(smem + p.off_sqb + t * 16);
      for (int m = warp; m < p.mt; m += kWarps) {
        float c[2][4] = {{__uint_as_float(bq.x), __uint_as_float(bq.y), __uint_as_float(bq.x), __uint_as_float(bq.y)},
                         {__uint_as_float(bq.z), __uint_as_float(bq.w), __uint_as_float(bq.z), __uint_as_float(bq.w)}};
        unsigned at = xs + (m * 16 + (lane & 15)) * p.x_pitch + (lane >> 4) * 16, wt = smem + lane * 16;
#pragma unroll 2
        for (int s = 0; s < p.sq_steps; ++s, at += 32, wt += 512) {
          unsigned a[4];
          ldsm4(at, a);
          const uint4 b = lds128(wt);
          mma16816(c[0], a, b.x, b.y);
          mma16816(c[1], a, b.z, b.w);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = m * 16 + g + h * 8, r = div_by(i, p.mul_cols), x = ix0 + i - r * p.cols;
          const bool in = static_cast<unsigned>(iy0 + r) < static_cast<unsigned>(p.H) && static_cast<unsigned>(x) < static_cast<unsigned>(p.W);
          // finite: the 1x1 part meets its neighbours with zero weights
          const unsigned lo = finite_f16x2(pack_f16x2<false>(act_f(c[0][h * 2], p.act_sq), act_f(c[0][h * 2 + 1], p.act_sq)));
          const unsigned hi = finite_f16x2(pack_f16x2<false>(act_f(c[1][h * 2], p.act_sq), act_f(c[1][h * 2 + 1], p.act_sq)));
          if (t < 2 * p.u_z) sts64(zs + i * p.z_pitch + t * 8, in ? lo : 0u, in ? hi : 0u);
        }
      }
      __syncthreads();
    }

    // ---- the window
    for (int m0 = warp * MG; m0 * 16 < p.n_out; m0 += kWarps * MG) {
      unsigned base[MG];
#pragma unroll
      for (int k = 0; k < MG; ++k) {
        const int i = min((m0 + k) * 16 + (lane & 15), p.n_out - 1), y = div_by(i, p.mul_tw), x = i - y * p.tw;
        base[k] = zs + (y * p.cols + x) * p.stride * p.z_pitch;
      }
      float acc[MG][NB][2][4];
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        const uint4 q = lds128(smem + p.off_bias + (4 * j + t) * 16);
#pragma unroll
        for (int k = 0; k < MG; ++k)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            acc[k][j][0][h * 2] = __uint_as_float(q.x);
            acc[k][j][0][h * 2 + 1] = __uint_as_float(q.y);
            acc[k][j][1][h * 2] = __uint_as_float(q.z);
            acc[k][j][1][h * 2 + 1] = __uint_as_float(q.w);
          }
      }
      unsigned tab = smem + p.off_tab + (lane >> 4) * 4, wt = smem + p.off_conv + lane * 16;
#pragma unroll 2
      for (int s = 0; s < p.steps; ++s, tab += 8, wt += NB * 512) {
        const unsigned off = lds32(tab);
        unsigned a[MG][4];
#pragma unroll
        for (int k = 0; k < MG; ++k) ldsm4(base[k] + off, a[k]);
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const uint4 b = lds128(wt + j * 512);
#pragma unroll
          for (int k = 0; k < MG; ++k) {
            mma16816(acc[k][j][0], a[k], b.x, b.y);
            mma16816(acc[k][j][1], a[k], b.z, b.w);
          }
        }
      }
#pragma unroll
      for (int k = 0; k < MG; ++k)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int i = (m0 + k) * 16 + g + h * 8, yy = div_by(i, p.mul_tw), y = y0 + yy, x = x0 + i - yy * p.tw;
          if (i >= p.n_out || y >= p.Ho || x >= p.Wo) continue;
          const long long px = static_cast<long long>(img) * p.out_img + static_cast<long long>(y * p.Wo + x) * 4;
#pragma unroll
          for (int j = 0; j < NB; ++j) {
            const int slice = 4 * j + t;
            if (slice >= p.sout) continue;
            float v[4] = {act_f(acc[k][j][0][h * 2], p.act_pre), act_f(acc[k][j][0][h * 2 + 1], p.act_pre), act_f(acc[k][j][1][h * 2], p.act_pre),
                          act_f(acc[k][j][1][h * 2 + 1], p.act_pre)};
            __half* dst = p.out + slice * p.out_sl + px;
            if (p.has_res) {
              const uint2 rr = *reinterpret_cast<const uint2*>(p.res + slice * p.out_sl + px);
              const float2 r01 = __half22float2(*reinterpret_cast<const __half2*>(&rr.x)), r23 = __half22float2(*reinterpret_cast<const __half2*>(&rr.y));
              // behind a concatenation the sum is an operator of its own: its input is the rounded tensor
              const float r[4] = {r01.x, r01.y, r23.x, r23.y};
#pragma unroll
              for (int q = 0; q < 4; ++q) v[q] = act_f((SQ ? round_f16(v[q]) : v[q]) + r[q], p.act_post);
            }
            *reinterpret_cast<uint2*>(dst) = make_uint2(pack_f16x2<false>(v[0], v[1]), pack_f16x2<false>(v[2], v[3]));
            if (p.pad_px && y == p.Ho - 1 && x == p.Wo - 1) *reinterpret_cast<uint2*>(dst + 4) = make_uint2(0u, 0u);
          }
        }
    }
  }
}

// ---------------------------------------------------------------- host side
int units_of(int c) { return (c + 7) / 8; }
int nb_of(int cout) { return (cout + 15) / 16; }

struct Sizes {  // of the packed weights
  int u_in, u_z, n_units, steps, sq_steps, off_conv, off_bias, off_sqb, bytes;
};
Sizes sizes_of(int cin, int csq, int cout, int k) {
  Sizes z;
  z.u_in = units_of(cin);
  z.u_z = csq ? units_of(csq) : z.u_in;
  z.n_units = k * k * z.u_z;
  z.steps = (z.n_units + 1) / 2;
  z.sq_steps = csq ? (z.u_in + 1) / 2 : 0;
  z.off_conv = z.sq_steps * 512;
  z.off_bias = z.off_conv + z.steps * nb_of(cout) * 512;
  z.off_sqb = z.off_bias + nb_of(cout) * 64;
  z.bytes = z.off_sqb + (csq ? 64 : 0);
  return z;
}

// Everything that follows from the record and the tile.
bool layout_of(const LaunchRec& r, int tw, int th, Params* p, unsigned* smem) {
  const Sizes z = sizes_of(r.C, r.Cmid, r.Co, r.kh);
  p->tw = tw;
  p->th = th;
  p->kw = r.kw;
  p->stride = r.sh;
  p->dil = r.dh;
  p->tiles_x = (r.Wo + tw - 1) / tw;
  p->tiles_y = (r.Ho + th - 1) / th;
  const long long units = static_cast<long long>(r.B) * p->tiles_x * p->tiles_y;
  if (units * p->tiles_x * p->tiles_y >= (1LL << 32) || units >= (1LL << 30)) return false;
  p->units = static_cast<int>(units);
  p->cols = (tw - 1) * r.sh + (r.kw - 1) * r.dh + 1;
  p->n_in = p->cols * ((th - 1) * r.sh + (r.kh - 1) * r.dh + 1);
  p->mt = (p->n_in + 15) / 16;
  p->n_out = tw * th;
  p->u_in = z.u_in;
  p->u_z = z.u_z;
  p->x_pitch = (z.u_in | 1) * 16;  // an odd number of units is free of conflicts
  p->z_pitch = (z.u_z | 1) * 16;
  p->n_units = z.n_units;
  p->steps = z.steps;
  p->sq_steps = z.sq_steps;
  p->off_conv = z.off_conv;
  p->off_bias = z.off_bias;
  p->off_sqb = z.off_sqb;
  p->wts_bytes = z.bytes;
  p->off_tab = static_cast<unsigned>(round_up_u64(z.bytes, 128));
  p->off_x = static_cast<unsigned>(round_up_u64(p->off_tab + z.steps * 8, 128));
  p->off_z = static_cast<unsigned>(round_up_u64(p->off_x + p->mt * 16 * p->x_pitch + 16, 128));
  p->off_bar = static_cast<unsigned>(round_up_u64(p->off_z + (r.Cmid ? p->mt * 16 * p->z_pitch + 16 : 0), 128));
  *smem = p->off_bar + 16;
  return p->n_in < 4096 && *smem <= static_cast<unsigned>(kSmemTwo);
}

// groups of 16 pixels a warp takes at a time
int mg_of(const Params& p) { return p.n_out >= 2 * 16 * kWarps ? 2 : 1; }
int ctas_of(unsigned smem, int nb, int mg) { return std::min(nb * mg > 4 ? 2 : 3, static_cast<int>(227 * 1024 / (smem + 1024))); }

// Estimated time: the chain of one CTA's units and what an SM's pipes need for the units of its CTAs.  Least-squares fit to 2100
// measured launches (26 shapes at batch 1 to 256; rms error 9 %, the tile it picks takes 1.04 times the best one's time).
double cost_us(const LaunchRec& r, const Params& p, unsigned smem) {
  const int nb = nb_of(r.Co), mg = mg_of(p), occ = ctas_of(smem, nb, mg), groups = (p.n_out + 15) / 16;
  const long long ctas = std::min<long long>(p.units, 148LL * occ), upc = (p.units + ctas - 1) / ctas, per_sm = (ctas + 147) / 148;
  const int rounds = (p.mt * 16 + kThreads - 1) / kThreads;
  double lat = rounds * (307.0 * p.u_in + (r.nhwc_in ? 402 : 0)), thr = 386 + p.mt * (2.1 + 5.9 * p.u_in);
  lat += (groups + kWarps * mg - 1) / (kWarps * mg) * (p.steps * (56.5 + 29 * nb * mg) + 332.0 * nb * mg);
  thr += groups * (0.81 * p.steps * (6 + 5 * nb) + 36.5 * nb);
  if (r.Cmid) {
    lat += (p.mt + kWarps - 1) / kWarps * 1221;
    thr += p.mt * 46.9;
  }
  const double a = upc * lat, b = upc * per_sm * thr;
  return 1.75 + std::cbrt(a * a * a + b * b * b) / 1900.0;
}

}  // namespace

// r: C input channels, Cmid squeezed ones (0: no squeeze), Co outputs, window, stride, pads; chooses the tile.
bool conv_mma_choose(const LaunchRec& r, BlockCfg* cfg, double* us) {
  if (r.kh != r.kw || r.kh < 1 || r.kh > 3 || r.sh != r.sw || r.sh < 1 || r.sh > 3 || r.dh != r.dw || r.dh > 2) return false;
  if (r.Co > 64 || r.C > 64 || r.Cmid > 16 || r.pt < 0 || r.pl < 0 || r.Ho < 1 || r.Wo < 2) return false;
  if (r.nhwc_in && (r.C > 4 || r.Cmid)) return false;
  if (r.Cmid && (r.sh != 1 || r.kh % 2 == 0)) return false;
  if (static_cast<int64_t>(plane_pixels(r.H, r.W)) * 4 >= (1LL << 30) || static_cast<int64_t>(plane_pixels(r.Ho, r.Wo)) * 4 >= (1LL << 30)) return false;
  double best = 0.0;
  for (int th = 1; th <= 32 && th <= r.Ho; ++th)
    for (int tw = 4; tw <= 64 && tw < r.Wo + 4; tw += 4) {
      const int w = std::min(tw, r.Wo);
      if (w * th > 1024) break;
      Params p{};
      unsigned smem = 0;
      if (!layout_of(r, w, th, &p, &smem)) continue;
      const double c = cost_us(r, p, smem);
      if (best != 0.0 && c >= best) continue;
      best = c;
      cfg->tw = w;
      cfg->nb = th;
    }
  if (us) *us = best;
  return best != 0.0;
}

// w [cout][k][k][c]: rows [0, c1) of the output channels from `wa` (k = `ka`), the others from `wb`; sq [csq][cin].
void conv_mma_pack(const float* sq, const float* sqb, const float* wa, const float* ba, int ka, int c1, const float* wb, const float* bb, int kb,
                   int cin, int csq, int cout, int k, std::vector<uint8_t>* blob, LaunchRec* r) {
  const Sizes z = sizes_of(cin, csq, cout, k);
  const int nb = nb_of(cout), cz = csq ? csq : cin;
  const uint64_t woff = round_up_u64(blob->size(), 256);
  blob->resize(woff + z.bytes, 0);
  uint8_t* base = blob->data() + woff;
  auto pair = [](int w, int lane, int* n, int* ch) {  // half w of a lane's {fragment 0: b0, b1; fragment 1: b0, b1}
    *n = lane >> 2;
    *ch = 2 * (lane & 3) + (w & 1);  // channel within the unit of 8
    return (w >> 1) & 1;             // which of the step's two units
  };
  for (int s = 0; s < z.sq_steps; ++s)
    for (int lane = 0; lane < 32; ++lane)
      for (int w = 0; w < 8; ++w) {
        int n, ch;
        const int u = 2 * s + pair(w, lane, &n, &ch), c = u * 8 + ch, co = channel_of(0, w >> 2, n);
        if (co < csq && c < cin) reinterpret_cast<uint16_t*>(base)[(s * 32 + lane) * 8 + w] = f32_to_f16_rne(sq[static_cast<size_t>(co) * cin + c]);
      }
  uint16_t* q = reinterpret_cast<uint16_t*>(base + z.off_conv);
  for (int s = 0; s < z.steps; ++s)
    for (int j = 0; j < nb; ++j)
      for (int lane = 0; lane < 32; ++lane)
        for (int w = 0; w < 8; ++w, ++q) {
          int n, ch;
          const int unit = 2 * s + pair(w, lane, &n, &ch), co = channel_of(j, w >> 2, n);
          const int tap = unit / z.u_z, c = unit % z.u_z * 8 + ch;
          if (unit >= z.n_units || c >= cz || co >= cout) continue;
          const bool first = co < c1;
          const int kk = first ? ka : kb;
          const float* src = first ? wa : wb;
          const int row = first ? co : co - c1;
          if (kk == k) *q = f32_to_f16_rne(src[(static_cast<size_t>(row) * k * k + tap) * cz + c]);
          else if (tap == k * k / 2) *q = f32_to_f16_rne(src[static_cast<size_t>(row) * cz + c]);  // a 1x1 in the window's middle
        }
  float* b = reinterpret_cast<float*>(base + z.off_bias);
  for (int co = 0; co < cout; ++co) b[co] = co < c1 ? ba[co] : bb[co - c1];
  if (csq) std::memcpy(base + z.off_sqb, sqb, static_cast<size_t>(csq) * sizeof(float));
  r->wts = Loc{W_WEIGHTS, 0, woff};
  r->wts_bytes = z.bytes;
}

unsigned int conv_mma_error_word(int* cuda_err) {
  unsigned int v = 0;
  const cudaError_t e = cudaMemcpyFromSymbol(&v, g_cm_error, sizeof v);
  if (cuda_err) *cuda_err = static_cast<int>(e);
  return v;
}

namespace {
template <int NB, int MG, bool SQ>
int launch_t(const Params& p, unsigned smem, cudaStream_t stream) {
  auto kern = conv_mma_kernel<NB, MG, SQ>;
  static bool attr_done_dev[kMaxDevices] = {};
  bool& attr_done = attr_done_dev[current_device_slot()];
  if (!attr_done) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemTwo);
    if (e != cudaSuccess) return static_cast<int>(e);
    attr_done = true;
  }
  const long long slots = static_cast<long long>(device_sm_count()) * ctas_of(smem, NB, MG);
  return static_cast<int>(launch_pdl(kern, dim3(static_cast<unsigned>(std::min<long long>(p.units, slots))), dim3(kThreads), smem, stream, p));
}
template <int MG, bool SQ>
int launch_nb(int nb, const Params& p, unsigned smem, cudaStream_t st) {
  switch (nb) {
    case 1: return launch_t<1, MG, SQ>(p, smem, st);
    case 2: return launch_t<2, MG, SQ>(p, smem, st);
    case 3: return launch_t<3, MG, SQ>(p, smem, st);
    default: return launch_t<4, MG, SQ>(p, smem, st);
  }
}
}  // namespace

int launch_conv_mma(const LaunchRec& r, const Ptrs& ptr, void* stream) {
  Params p{};
  unsigned smem = 0;
  if (!layout_of(r, r.block.tw, r.block.nb, &p, &smem)) return static_cast<int>(cudaErrorInvalidConfiguration);
  const int P = plane_pixels(r.H, r.W), Po = plane_pixels(r.Ho, r.Wo);
  p.in = static_cast<const __half*>(ptr.in0);
  p.res = static_cast<const __half*>(ptr.res);
  p.out = static_cast<__half*>(ptr.out);
  p.wts = static_cast<const unsigned char*>(ptr.wts);
  p.H = r.H;
  p.W = r.W;
  p.Ho = r.Ho;
  p.Wo = r.Wo;
  p.C = r.C;
  p.pad_t = r.pt;
  p.pad_l = r.pl;
  p.sin = slices(r.C);
  p.sout = slices(r.Co);
  p.nhwc = r.nhwc_in;
  p.in_sl = static_cast<long long>(r.B) * P * 4;
  p.in_img = r.nhwc_in ? r.H * r.W * r.C : P * 4;
  p.out_sl = static_cast<long long>(r.B) * Po * 4;
  p.out_img = Po * 4;
  p.mul_cols = magic(p.cols);
  p.mul_tw = magic(p.tw);
  p.mul_per = magic(static_cast<uint64_t>(p.tiles_x) * p.tiles_y);
  p.mul_tx = magic(p.tiles_x);
  p.pad_px = r.Ho * r.Wo % 2;
  p.act_sq = r.ep.act_pre;
  p.act_pre = r.ep2.act_pre;
  p.has_res = r.ep2.has_res;
  p.act_post = r.ep2.act_post;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int nb = nb_of(r.Co);
  if (mg_of(p) == 2) return r.Cmid ? launch_nb<2, true>(nb, p, smem, st) : launch_nb<2, false>(nb, p, smem, st);
  return r.Cmid ? launch_nb<1, true>(nb, p, smem, st) : launch_nb<1, false>(nb, p, smem, st);
}

}  // namespace gi
