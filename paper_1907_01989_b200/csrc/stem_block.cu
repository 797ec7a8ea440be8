// The first layers of the MobileNets as ONE kernel, for any image size (fp16 storage):
//   3x3 stride-2 convolution of a 3-channel NHWC image to at most 32 channels -> depthwise 3x3 -> 1x1
// The two tensors between the operators, at 112 x 112 x 32 the largest of the network, never reach memory; they are rounded to
// fp16 exactly where separate kernels would have stored them.
//
// A unit is a tile of output pixels.  Its image rows arrive by bulk copies (a warp of its own issues them, one row a lane, for
// the next unit while this one is computed).  All arithmetic is mma.sync.m16n8k16 with fp32 sums:
//   stem       16 pixels x 32 channels: lane t of a quad takes words t of the three window rows - values 2 t, 2 t + 1 of the 9 -
//              and the ninth value of row t, straight from the staged rows: 27 values are the 32 of two steps, nothing is
//              rearranged.  Results go to the hidden tile as pixel-slices, zero outside the image.
//   depthwise  as in block_mma.cu: an output pair (x, x + 1) of a slice is a row of the banded 16 x 8 product, a warp takes 16
//              pairs and two output rows, so that a fragment of a hidden row serves both.
//   1x1        the depthwise results of all 32 channels are its A operand in the registers they were computed in; its output
//              blocks are computed and stored one after the other, so their number costs no registers.
//
// A group of 16 pixels of the hidden tile lies in one of its rows, so that what depends on the row - where its image rows start,
// which need not be on a 16-byte boundary, not even on a word - is worked out once for the warp.
//
// What bounds it: at 112x112 3 -> 32 -> 16, batch 256, 350 instructions per 16 output pixels (half of them the depthwise
// operator's), the shared-memory pipe busy 56 % of the time, the matrix pipe 24 %, with 14 warps on an SM.  Measured on one B200
// against separate kernels: 132 against 213 us there, 176 against 272 with 64 output channels; 16 images of 513 pixels 50
// against 83 (the same chain with rearranged window values and 4-byte copies).
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

constexpr int kWarps = 7;  // that compute; one more copies.  Two CTAs of 8 warps leave 128 registers a thread.
constexpr int kTR = 2;     // output rows a warp walks down
constexpr int kMaxPx = 39 * 16;                  // pixels of a hidden tile
constexpr int kSliceBytes = kMaxPx * 8 + 32;     // 32 modulo 128: the stores of half a warp meet 32 different banks
constexpr int kHidBytes = 8 * kSliceBytes;
constexpr int kSub = 2 * 512 + kBiasBytes + kTableBytes + kDwBiasBytes;  // packed weights of 16 hidden channels without the 1x1's
constexpr unsigned kWaitNs = 1000000000u;
constexpr int kSmemPerSm = 227 * 1024;

__device__ unsigned g_stem_error = 0;

struct Params {
  const __half* in;
  __half* out;
  const unsigned char* wts;
  int H, W, Ho, Wo, Hi, Wi;  // hidden plane, output plane, image
  int spt, spl, pad_t, pad_l;
  int tw, th, tiles_x, tiles_y, units;
  int rows, pitch, gpr, mt;     // hidden tile: rows, pixels per row and groups of 16 pixels per row, groups
  int pw, ncols, ngroups;       // pairs per band of kTR rows; pairs and groups of 16 of them
  int raw_rows, raw_pitch, raw_bytes;  // staged image rows (two tiles' worth), bytes between them and of a tile
  int np, wts_bytes;
  long long total_bytes;        // of the image tensor
  long long o_sl, o_img;
  int o_px, sout;
  unsigned off_raw, off_hid, off_bar;
  unsigned mul_gpr, mul_per, mul_tx;
  unsigned hi_s, hi_d, hi_p;  // upper clamps behind the three operators, two halves (6; hi_s: or the largest finite value, the others: or infinity)
  int wide, pad_px;     // a pair of pixels is one aligned 16-byte store; an odd plane holds one more pixel: zero it
};

struct Pos {
  int img, y0, x0;
};
__device__ __forceinline__ Pos unit_pos(const Params& p, int unit) {
  Pos u;
  const int per = p.tiles_x * p.tiles_y;
  u.img = per == 1 ? unit : div_by(unit, p.mul_per);
  const int r = unit - u.img * per, ty = p.tiles_x == 1 ? r : div_by(r, p.mul_tx);
  u.y0 = ty * p.th;
  u.x0 = (r - ty * p.tiles_x) * p.tw;
  return u;
}

__device__ __forceinline__ void sync_compute() { asm volatile("bar.sync 1, %0;" ::"n"(kWarps * 32) : "memory"); }

// The copying warp's part of a unit.
__device__ __forceinline__ void load_rows(const Params& p, const Pos& u, unsigned raw, unsigned bar, int lane) {
  const int iy0 = 2 * (u.y0 - p.pad_t) - p.spt, ix0 = 2 * (u.x0 - p.pad_l) - p.spl;
  const long long full16 = p.total_bytes & ~15LL;
  const char* base = reinterpret_cast<const char*>(p.in);
  auto span = [&](int r, long long& from, int& skip, int& bytes) {  // what a bulk copy brings of row r
    const long long b0 = ((static_cast<long long>(u.img) * p.Hi + iy0 + r) * p.Wi + ix0) * 6;
    const long long a0 = b0 & ~15LL, a1 = min((b0 + (2 * p.tw + 5) * 6 + 15) & ~15LL, full16);
    skip = a0 < 0 ? static_cast<int>(-a0) : 0;
    from = a0 + skip;
    bytes = static_cast<unsigned>(iy0 + r) < static_cast<unsigned>(p.Hi) ? max(0, static_cast<int>(a1 - from)) : 0;
  };
  int total = 0;
  for (int r = lane; r < p.raw_rows; r += 32) {
    long long from;
    int skip, bytes;
    span(r, from, skip, bytes);
    total += bytes;
    const unsigned dst = raw + r * p.raw_pitch;
    if (static_cast<unsigned>(iy0 + r) >= static_cast<unsigned>(p.Hi)) {
      for (int i = 0; i < p.raw_pitch; i += 16) sts128(dst + i, 0u, 0u, 0u, 0u);
    } else if (from + bytes >= full16) {  // the tensor's last bytes, less than a copy's 16
      for (long long b = full16; b < p.total_bytes; b += 2) {
        const int at = static_cast<int>(b - from) + skip;
        if (at >= 0 && at + 2 <= p.raw_pitch)
          asm volatile("st.shared.u16 [%0], %1;" ::"r"(dst + at), "h"(*reinterpret_cast<const unsigned short*>(base + b)) : "memory");
      }
    }
  }
  total = __reduce_add_sync(0xffffffffu, total);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  __syncwarp();
  if (lane == 0) mbar_expect_tx(bar, total);
  __syncwarp();
  for (int r = lane; r < p.raw_rows; r += 32) {
    long long from;
    int skip, bytes;
    span(r, from, skip, bytes);
    if (bytes > 0) bulk_load(raw + r * p.raw_pitch + skip, base + from, bytes, bar);
  }
}

// ODD: rows of the image may start on an odd half.
template <bool ODD, bool RELU>
__global__ void __launch_bounds__(kWarps * 32 + 32, 2) stem_block_kernel(const Params p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const unsigned smem = smem_u32(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const unsigned bar_w = smem + p.off_bar, bar_full = bar_w + 8, bar_empty = bar_w + 24;  // full and empty: two each
  volatile unsigned* abort_flag = reinterpret_cast<volatile unsigned*>(smem_raw + p.off_bar + 40);
  const int my_units = (p.units - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x);

  pdl_launch_dependents();
  if (tid == 0) {
    mbar_init(bar_w, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_full + i * 8, 1);
      mbar_init(bar_empty + i * 8, kWarps);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp == kWarps) {
    if (lane == 0) {
      mbar_expect_tx(bar_w, p.wts_bytes);
      bulk_load(smem, p.wts, p.wts_bytes, bar_w);
    }
    pdl_wait();
    int k = 0;  // units whose rows have been requested
    for (; k < my_units; ++k) {
      if (k > 1 && !mbar_wait_warp(bar_empty + (k & 1) * 8, (k / 2 - 1) & 1, abort_flag, kWaitNs, &g_stem_error, 1u)) break;
      load_rows(p, unit_pos(p, blockIdx.x + k * gridDim.x), smem + p.off_raw + (k & 1) * p.raw_bytes, bar_full + (k & 1) * 8, lane);
    }
    // the warps that compute stop waiting once a wait has run out: the copies in flight land before this warp leaves (bounded as well)
    if (lane == 0) {
      unsigned none = 0;
      mbar_wait(bar_w, 0u, &none, kWaitNs, &g_stem_error, 4u);
      for (int i = max(0, k - 2); i < k; ++i) mbar_wait(bar_full + (i & 1) * 8, (i / 2) & 1, &none, kWaitNs, &g_stem_error, 4u);
    }
    return;
  }

  pdl_wait();
  const unsigned hid = smem + p.off_hid;
  const int subb = kSub + p.np * 512;
  // this lane's rows of the depthwise A operand, its two output pairs, and which half of a banded weight word it takes
  unsigned dw_base, col[2];
  {
    int c = warp * 16 + (lane & 15);
    if (c >= p.ncols) c = 0;
    const int band = c / p.pw;
    dw_base = static_cast<unsigned>(band * kTR * p.pitch) * 8u + (c - band * p.pw) * 16u + (lane >> 4) * 16u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = warp * 16 + g + h * 8, b = q / p.pw;
      col[h] = q < p.ncols ? static_cast<unsigned>(b * kTR) << 16 | static_cast<unsigned>(2 * (q - b * p.pw)) : 0xffffffffu;
    }
  }
  const bool band_lane = (g >> 2) == (t & 1);
  const unsigned sel_a = !band_lane ? 0x4444u : ((g >> 1) & 1) ? 0x1044u : 0x4410u;
  const unsigned sel_b = !band_lane ? 0x4444u : ((g >> 1) & 1) ? 0x3244u : 0x4432u;
  const unsigned dw_entry = ((t >> 1) * 8 + g) * 16;
  const int wi3 = 3 * p.Wi;
  const unsigned lane_g = 12 * g, lane_gt = 12 * g + 4 * t, ninth = t < 3 ? 0xffffu : 0u;

  bool ok = mbar_wait_warp(bar_w, 0u, abort_flag, kWaitNs, &g_stem_error, 2u);
#pragma unroll 1
  for (int k = 0; k < my_units; ++k) {
    const Pos u = unit_pos(p, blockIdx.x + k * gridDim.x);
    const unsigned raw = smem + p.off_raw + (k & 1) * p.raw_bytes;
    ok = mbar_wait_warp(bar_full + (k & 1) * 8, (k / 2) & 1, abort_flag, kWaitNs, &g_stem_error, 2u) && ok;
    sync_compute();  // the hidden tile is free

    // ---- stem: groups of 16 pixels of the hidden tile
    {
      const int iy0 = 2 * (u.y0 - p.pad_t) - p.spt, ix0 = 2 * (u.x0 - p.pad_l) - p.spl;
      // halves between the 16-byte boundary a staged row starts at and the row's first value, modulo 8
      const int f0 = static_cast<int>((((static_cast<long long>(u.img) * p.Hi + iy0) * p.Wi + ix0) * 3) & 7);
      uint4 wf[2][2], be[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        wf[h][0] = lds128(smem + h * subb + lane * 16);
        wf[h][1] = lds128(smem + h * subb + 512 + lane * 16);
        be[h] = lds128(smem + h * subb + 1024 + t * 16);
      }
#pragma unroll 1
      for (int m = warp; m < p.mt; m += kWarps) {  // a group lies in one row: everything but the column is the warp's
        const int r = p.gpr == 1 ? m : div_by(m, p.mul_gpr), cg = (m - r * p.gpr) * 16;
        const bool row_in = static_cast<unsigned>(u.y0 - p.pad_t + r) < static_cast<unsigned>(p.H);
        const int x = u.x0 - p.pad_l + cg + g, ix = ix0 + 2 * (cg + g);
        const bool in[2] = {row_in && static_cast<unsigned>(x) < static_cast<unsigned>(p.W), row_in && static_cast<unsigned>(x + 8) < static_cast<unsigned>(p.W)};
        unsigned at[3];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) at[ky] = raw + (2 * r + ky) * p.raw_pitch + ((f0 + (2 * r + ky) * wi3) & 7) * 2 + cg * 12;
        const unsigned at3 = (t == 0 ? at[0] : t == 1 ? at[1] : at[2]) + lane_g + 16;
        unsigned v[2][4];
#pragma unroll
        for (int ky = 0; ky < 3; ++ky) {
          if (!ODD || !(at[ky] & 2u)) {
            v[0][ky] = lds32(at[ky] + lane_gt);
            v[1][ky] = lds32(at[ky] + lane_gt + 96);
          } else {
            const unsigned w = at[ky] - 2 + lane_gt;
            v[0][ky] = __funnelshift_r(lds32(w), lds32(w + 4), 16);
            v[1][ky] = __funnelshift_r(lds32(w + 96), lds32(w + 100), 16);
          }
        }
        const unsigned sh3 = ODD ? (at3 & 2u) * 8u : 0u, w3 = ODD ? at3 & ~3u : at3;
        v[0][3] = (lds32(w3) >> sh3) & ninth;
        v[1][3] = (lds32(w3 + 96) >> sh3) & ninth;
        if (ix0 + 2 * cg < 0 || ix0 + 2 * cg + 32 >= p.Wi) {  // columns outside the image hold neighbours' values
#pragma unroll
          for (int h = 0; h < 2; ++h) {
#pragma unroll
            for (int q = 0; q < 2; ++q)
              if (static_cast<unsigned>(ix + 16 * h + (2 * t + q) / 3) >= static_cast<unsigned>(p.Wi))
#pragma unroll
                for (int ky = 0; ky < 3; ++ky) v[h][ky] &= q ? 0x0000ffffu : 0xffff0000u;
            if (static_cast<unsigned>(ix + 16 * h + 2) >= static_cast<unsigned>(p.Wi)) v[h][3] = 0u;
          }
        }
        const unsigned a0[4] = {v[0][0], v[1][0], v[0][1], v[1][1]}, a1[4] = {v[0][2], v[1][2], v[0][3], v[1][3]};
        const unsigned hi[2] = {in[0] ? p.hi_s : 0u, in[1] ? p.hi_s : 0u};
        float c[2][2][4];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const float b0 = __uint_as_float(be[s].x), b1 = __uint_as_float(be[s].y), b2 = __uint_as_float(be[s].z), b3 = __uint_as_float(be[s].w);
          mma16816c(c[s][0], a0, wf[s][0].x, wf[s][0].y, b0, b1, b0, b1);
          mma16816c(c[s][1], a0, wf[s][0].z, wf[s][0].w, b2, b3, b2, b3);
        }
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          mma16816(c[s][0], a1, wf[s][1].x, wf[s][1].y);
          mma16816(c[s][1], a1, wf[s][1].z, wf[s][1].w);
        }
        const unsigned to = hid + t * kSliceBytes + (m * 16 + g) * 8;
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            sts64(to + s * 4 * kSliceBytes + h * 64, min_f16x2(pack_f16x2<true>(c[s][0][h * 2], c[s][0][h * 2 + 1]), hi[h]),
                  min_f16x2(pack_f16x2<true>(c[s][1][h * 2], c[s][1][h * 2 + 1]), hi[h]));
      }
    }
    sync_compute();  // the hidden tile is complete, the staged rows are free
    if (lane == 0 && k + 2 < my_units) mbar_arrive(bar_empty + (k & 1) * 8);
    if (warp >= p.ngroups) continue;

    // ---- depthwise: the results of 32 channels stay in registers as the 1x1's A operand
    unsigned af[2][kTR][2][4];
    const unsigned hb = hid + dw_base, row_b = p.pitch * 8;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned wd = smem + h * subb + 1024 + kBiasBytes;
#pragma unroll
      for (int sp = 0; sp < 2; ++sp) {
        float d[2][kTR][4];
#pragma unroll
        for (int s2 = 0; s2 < 2; ++s2) {
          const int sl = sp * 2 + s2;
          const uint4 w = lds128(wd + sl * 256 + dw_entry);
          const uint4 bq = lds128(wd + kTableBytes + sl * 64 + t * 16);
          const unsigned b0[3] = {prmt(w.x, sel_a), prmt(w.y, sel_a), prmt(w.z, sel_a)};
          const unsigned b1[3] = {prmt(w.x, sel_b), prmt(w.y, sel_b), prmt(w.z, sel_b)};
#pragma unroll
          for (int rr = 0; rr < kTR + 2; ++rr) {
            unsigned a[4];
            ldsm4(hb + rr * row_b + (h * 4 + sl) * kSliceBytes, a);
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
              const int v = rr - ky;
              if (v < 0 || v >= kTR) continue;
              if (ky == 0)
                mma16816c(d[s2][v], a, b0[ky], b1[ky], __uint_as_float(bq.x), __uint_as_float(bq.y), __uint_as_float(bq.z), __uint_as_float(bq.w));
              else
                mma16816(d[s2][v], a, b0[ky], b1[ky]);
            }
          }
        }
#pragma unroll
        for (int v = 0; v < kTR; ++v)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            af[h][v][q][sp * 2] = min_f16x2(pack_f16x2<true>(d[0][v][q], d[1][v][q]), p.hi_d);
            af[h][v][q][sp * 2 + 1] = min_f16x2(pack_f16x2<true>(d[0][v][2 + q], d[1][v][2 + q]), p.hi_d);
          }
      }
    }

    // ---- 1x1, one block of 16 output channels at a time
#pragma unroll 1
    for (int j = 0; j < p.np; ++j) {
      float acc[kTR][2][2][4];
      const uint4 b = lds128(smem + 2 * subb + (j * 4 + t) * 16);
      const uint4 w0 = lds128(smem + kSub + j * 512 + lane * 16), w1 = lds128(smem + subb + kSub + j * 512 + lane * 16);
      const float f0 = __uint_as_float(b.x), f1 = __uint_as_float(b.y), f2 = __uint_as_float(b.z), f3 = __uint_as_float(b.w);
#pragma unroll
      for (int v = 0; v < kTR; ++v)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          mma16816c(acc[v][q][0], af[0][v][q], w0.x, w0.y, f0, f1, f0, f1);
          mma16816c(acc[v][q][1], af[0][v][q], w0.z, w0.w, f2, f3, f2, f3);
        }
#pragma unroll
      for (int v = 0; v < kTR; ++v)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          mma16816(acc[v][q][0], af[1][v][q], w1.x, w1.y);
          mma16816(acc[v][q][1], af[1][v][q], w1.z, w1.w);
        }
      const int slice = 4 * j + t;
      if (slice >= p.sout || !ok) continue;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int x = u.x0 + static_cast<int>(col[h] & 0xffffu), y0 = u.y0 + static_cast<int>(col[h] >> 16);
        if (col[h] == 0xffffffffu || x >= p.Wo) continue;
        const bool two = x + 1 < p.Wo;
        __half* dst = p.out + slice * p.o_sl + u.img * p.o_img + static_cast<long long>(y0 * p.Wo + x) * p.o_px;
#pragma unroll
        for (int v = 0; v < kTR; ++v, dst += p.Wo * p.o_px) {
          if (y0 + v >= p.Ho) break;
          uint2 o[2];
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            o[q] = make_uint2(pack_f16x2<RELU>(acc[v][q][0][h * 2], acc[v][q][0][h * 2 + 1]), pack_f16x2<RELU>(acc[v][q][1][h * 2], acc[v][q][1][h * 2 + 1]));
            if (RELU) o[q] = make_uint2(min_f16x2(o[q].x, p.hi_p), min_f16x2(o[q].y, p.hi_p));
          }
          if (p.wide) {
            *reinterpret_cast<uint4*>(dst) = make_uint4(o[0].x, o[0].y, o[1].x, o[1].y);
          } else {
            *reinterpret_cast<uint2*>(dst) = o[0];
            if (two) *reinterpret_cast<uint2*>(dst + p.o_px) = o[1];
            if (p.pad_px && y0 + v == p.Ho - 1 && x + (two ? 1 : 0) == p.Wo - 1) *reinterpret_cast<uint2*>(dst + (two ? 8 : 4)) = make_uint2(0, 0);
          }
        }
      }
    }
  }
}

// ---------------------------------------------------------------- host side
int wts_bytes(int np) { return 2 * (kSub + np * 512) + np * 64; }

bool layout_of(const LaunchRec& r, const BlockCfg& c, Params* p) {
  p->th = c.nb * kTR;
  p->tw = c.tw;
  p->rows = p->th + 2;
  p->gpr = (c.tw + 2 + 15) / 16;
  p->pitch = p->gpr * 16;
  p->mt = p->rows * p->gpr;
  p->pw = c.tw / 2;
  p->ncols = c.nb * p->pw;
  p->ngroups = (p->ncols + 15) / 16;
  if (p->mt * 16 > kMaxPx || p->ngroups > kWarps) return false;
  p->raw_rows = 2 * p->rows + 1;
  p->raw_pitch = static_cast<int>(round_up_u64((2 * p->pitch + 1) * 6 + 14 + 32, 16));  // a group's tail may read past the last column
  p->raw_bytes = static_cast<int>(round_up_u64(p->raw_rows * p->raw_pitch, 128));
  p->np = c.np;
  p->wts_bytes = wts_bytes(c.np);
  p->off_raw = static_cast<unsigned>(round_up_u64(p->wts_bytes, 128));
  p->off_hid = static_cast<unsigned>(round_up_u64(p->off_raw + 2 * p->raw_bytes, 128));
  p->off_bar = p->off_hid + kHidBytes;
  return p->off_bar + 64 <= (kSmemPerSm - 4096) / 2;
}

// Estimated time: the chain of one CTA's units, and what an SM's pipes need for the units of both CTAs.  Least-squares fit to 1200
// measured launches (batch 1 to 256, images of 160 to 513 pixels, 16 and 64 output channels; rms error 7 %).
double cost_us(const Params& p, long long units) {
  const long long ctas = std::min<long long>(units, 2 * 148), upc = (units + ctas - 1) / ctas, per_sm = ctas > 148 ? 2 : 1;
  const double a = upc * (414.5 * ((p.mt + kWarps - 1) / kWarps) + 580.6 * p.np + 71.2 * p.raw_rows);
  const double b = upc * per_sm * (361.1 + 32 * p.mt + p.ngroups * (399.4 + 62.9 * p.np));
  return 3.3 + std::cbrt(a * a * a + b * b * b) / 1900.0;
}

}  // namespace

bool stem_block_choose(const LaunchRec& r, BlockCfg* best, double* us) {
  if (r.kh != 3 || r.kw != 3 || r.sh != 1 || r.sw != 1 || r.dh != 1 || r.dw != 1 || r.C != 3 || r.Cmid > 32 || r.ep2.has_res) return false;
  if (r.pt < 0 || r.pt > 2 || r.pl < 0 || r.pl > 2 || r.W < 2 || r.Ho < 1 || r.Co2 > 512 || r.Wo >= 32768) return false;
  if (static_cast<int64_t>(r.Ho) * r.Wo * std::max(4, r.Co2) >= (1LL << 31)) return false;
  BlockCfg c;
  c.stem = 1;
  c.np = (r.Co2 + 15) / 16;
  double best_cost = 0.0;
  const int wo_even = (r.Wo + 1) / 2 * 2;
  for (int tx = (wo_even + 63) / 64; tx <= 64 && tx <= wo_even / 2; ++tx) {
    c.tw = ((wo_even + tx - 1) / tx + 1) / 2 * 2;
    c.tiles_x = (r.Wo + c.tw - 1) / c.tw;
    for (c.nb = 1; c.nb <= 28 && (c.nb - 1) * kTR < r.Ho; ++c.nb) {
      c.tiles_y = (r.Ho + c.nb * kTR - 1) / (c.nb * kTR);
      const long long units = static_cast<long long>(r.B) * c.tiles_x * c.tiles_y;
      if (units * c.tiles_x * c.tiles_y >= (1LL << 32) || units > (1 << 28)) continue;
      Params p{};
      if (!layout_of(r, c, &p)) continue;
      c.units = static_cast<int>(units);
      const double cost = cost_us(p, units);
      if (best_cost != 0.0 && cost >= best_cost) continue;
      best_cost = cost;
      *best = c;
    }
  }
  if (us) *us = best_cost;
  return best_cost != 0.0;
}

// One run of bytes: two blocks of 16 hidden channels (stem fragments and bias, banded depthwise operands and bias, 1x1
// fragments), then the 1x1's bias.  ws [chid][3][3][3], wd [9][chid], wp [cout][chid].
void stem_block_pack(const float* ws, const float* bs, const float* wd, const float* bd, const float* wp, const float* bp, int chid, int cout,
                     const BlockCfg& c, std::vector<uint8_t>* blob, LaunchRec* r) {
  const int np = c.np;
  const uint64_t woff = round_up_u64(blob->size(), 256);
  blob->resize(woff + wts_bytes(np), 0);
  for (int sub = 0; sub < 2; ++sub) {
    uint8_t* base = blob->data() + woff + sub * (kSub + np * 512);
    uint16_t* e = reinterpret_cast<uint16_t*>(base);
    for (int s = 0; s < 2; ++s)
      for (int lane = 0; lane < 32; ++lane)
        for (int w = 0; w < 8; ++w) {  // halves of {fragment 0: b0, b1; fragment 1: b0, b1}
          const int f = w >> 2, hi8 = (w >> 1) & 1, lo = w & 1, n = lane >> 2, t = lane & 3;
          const int q = 2 * s + hi8;  // which word of lane t: its pair of values of window row q, or (3) the ninth of row t
          const int ky = q < 3 ? q : t, v = q < 3 ? 2 * t + lo : 8 + lo, h = channel_of(sub, f, n);
          if (h < chid && ky < 3 && v < 9) e[(s * 32 + lane) * 8 + w] = f32_to_f16_rne(ws[(static_cast<size_t>(h) * 3 + ky) * 9 + v]);
        }
    float* sbias = reinterpret_cast<float*>(base + 1024);
    uint16_t* tabl = reinterpret_cast<uint16_t*>(base + 1024 + kBiasBytes);
    float* dbias = reinterpret_cast<float*>(base + 1024 + kBiasBytes + kTableBytes);
    for (int ch = 0; ch < 16 && sub * 16 + ch < chid; ++ch) {
      sbias[ch] = bs[sub * 16 + ch];
      for (int i = 0; i < 4; ++i) dbias[ch * 4 + i] = bd[sub * 16 + ch];
    }
    for (int sl = 0; sl < 4; ++sl)
      for (int jh = 0; jh < 2; ++jh)
        for (int g = 0; g < 8; ++g) {
          const int h = sub * 16 + sl * 4 + (g >> 1);
          if (h >= chid) continue;
          uint16_t* word = tabl + ((sl * 16 + jh * 8 + g) * 4) * 2;
          for (int ky = 0; ky < 3; ++ky)
            for (int b = 0; b < 2; ++b) {
              const int dx = b * 2 + jh - (g & 1);  // input pixel of the window row, output pixel of the pair
              if (dx >= 0 && dx <= 2) word[ky * 2 + b] = f32_to_f16_rne(wd[static_cast<size_t>(ky * 3 + dx) * chid + h]);
            }
        }
    uint16_t* q = reinterpret_cast<uint16_t*>(base + kSub);
    for (int j = 0; j < np; ++j)
      for (int lane = 0; lane < 32; ++lane)
        for (int w = 0; w < 8; ++w) {
          const int f = w >> 2, hi8 = (w >> 1) & 1, lo = w & 1, n = lane >> 2, t = lane & 3;
          const int h = sub * 16 + hi8 * 8 + lo * 4 + t, co = channel_of(j, f, n);
          if (h < chid && co < cout) q[(j * 32 + lane) * 8 + w] = f32_to_f16_rne(wp[static_cast<size_t>(co) * chid + h]);
        }
  }
  std::memcpy(blob->data() + woff + 2 * (kSub + np * 512), bp, static_cast<size_t>(cout) * sizeof(float));
  r->wts = Loc{W_WEIGHTS, 0, woff};
  r->wts_bytes = wts_bytes(np);
}

unsigned int stem_block_error_word(int* cuda_err) {
  unsigned int v = 0;
  const cudaError_t e = cudaMemcpyFromSymbol(&v, g_stem_error, sizeof v);
  if (cuda_err) *cuda_err = static_cast<int>(e);
  return v;
}

int launch_stem_block(const LaunchRec& r, const Ptrs& ptr, void* stream) {
  const BlockCfg& c = r.block;
  Params p{};
  if (!layout_of(r, c, &p)) return static_cast<int>(cudaErrorInvalidConfiguration);
  p.in = static_cast<const __half*>(ptr.in0);
  p.out = static_cast<__half*>(ptr.out);
  p.wts = static_cast<const unsigned char*>(ptr.wts);
  p.H = r.H;
  p.W = r.W;
  p.Ho = r.Ho;
  p.Wo = r.Wo;
  p.Hi = r.stem_h;
  p.Wi = r.stem_w;
  p.spt = r.stem_pt;
  p.spl = r.stem_pl;
  p.pad_t = r.pt;
  p.pad_l = r.pl;
  p.tiles_x = c.tiles_x;
  p.tiles_y = c.tiles_y;
  p.units = c.units;
  p.total_bytes = static_cast<long long>(r.B) * r.stem_h * r.stem_w * 6;
  const int Po = plane_pixels(r.Ho, r.Wo);
  p.o_px = r.nhwc_out ? r.Co2 : 4;
  p.o_img = r.nhwc_out ? static_cast<long long>(r.Ho) * r.Wo * r.Co2 : Po * 4;
  p.o_sl = r.nhwc_out ? 4 : static_cast<long long>(r.B) * Po * 4;
  p.sout = slices(r.Co2);
  p.mul_gpr = magic(p.gpr);
  p.mul_per = magic(static_cast<uint64_t>(c.tiles_x) * c.tiles_y);
  p.mul_tx = magic(c.tiles_x);
  p.hi_s = r.ep.act_pre == GI_ACT_RELU6 ? 0x46004600u : kMaxFinite;  // the banded operand multiplies neighbours by zero
  p.hi_d = r.ep_mid.act_pre == GI_ACT_RELU6 ? 0x46004600u : 0x7c007c00u;
  p.hi_p = r.ep2.act_pre == GI_ACT_RELU6 ? 0x46004600u : 0x7c007c00u;
  p.wide = !r.nhwc_out && r.Wo % 2 == 0;
  p.pad_px = !r.nhwc_out && (r.Ho * r.Wo) % 2;
  // 6 bytes a pixel: with an even width and an even first column every row starts on a whole word
  const bool odd = r.stem_w % 2 != 0 || r.stem_pl % 2 != 0;
  const bool relu = r.ep2.act_pre != GI_ACT_NONE;
  auto kern = odd ? (relu ? stem_block_kernel<true, true> : stem_block_kernel<true, false>)
                  : (relu ? stem_block_kernel<false, true> : stem_block_kernel<false, false>);
  static bool attr_done_dev[kMaxDevices] = {};
  bool& attr_done = attr_done_dev[current_device_slot()];
  if (!attr_done) {
    for (auto f : {stem_block_kernel<true, true>, stem_block_kernel<true, false>, stem_block_kernel<false, true>, stem_block_kernel<false, false>}) {
      const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm / 2);
      if (e != cudaSuccess) return static_cast<int>(e);
    }
    attr_done = true;
  }
  const unsigned grid = static_cast<unsigned>(std::min<long long>(c.units, 2LL * device_sm_count()));
  return static_cast<int>(launch_pdl(kern, dim3(grid), dim3(kWarps * 32 + 32), p.off_bar + 64, static_cast<cudaStream_t>(stream), p));
}

}  // namespace gi
