// A depthwise 3x3 convolution with the convolutions around it as ONE kernel, for any plane size:
//   1x1 expansion -> depthwise 3x3 -> 1x1 projection (+ residual)   an inverted-residual block
//   3x3 stride-2 stem on a 3-channel NHWC image -> depthwise 3x3 -> 1x1   the first layers of the MobileNets: stem_block.cu
//   depthwise 3x3 -> 1x1                                            a depthwise-separable pair
// The tensors between the operators - up to six times as wide as the block's ends - never reach memory; they are rounded to
// fp16 exactly where the separate kernels would have stored them.
//
// Why the warp-level matrix instruction.  All operators run on mma.sync.m16n8k16 (fp16 operands, fp32 sums), because its
// register fragments chain: the depthwise result leaves the tensor core in the very registers in which the projection wants
// its A operand, so of the two hidden tensors one is written to shared memory once (the 3x3 window has to gather from it)
// and the other not at all.  Measured on one SM: one m16n8k16 per 2 cycles, 21 cycles of latency, one ldmatrix.x4 per 4
// cycles.  tcgen05.mma has four times that rate, but its results come back through tensor memory and its A operand goes out
// through shared memory, and a depthwise slice would occupy it for 47 cycles per instruction at N = 8.
//
// The depthwise operator as a matrix product.  A hidden pixel-slice is 4 channels (8 bytes); two neighbouring pixels are one
// 16-byte row of an ldmatrix matrix.  Stride 1: an output PAIR (x, x+1) of one slice reads 4 input pixels x 4 channels = 16
// values per window row, and produces 2 pixels x 4 channels = 8: one m16n8k16 per window row with the 3 taps in a banded
// 16 x 8 operand.  Its 16 rows are 16 pairs, and a warp walks TR output rows down, so that the fragment of a hidden row serves
// the three output rows around it in the very registers ldmatrix left it in (pairing vertical neighbours in the 16 rows needs
// fewer loads, but every other fragment then has to be put together by register moves).  Stride 2: 16 output columns,
// 4 channels x 2 output rows; 5 window rows = 5 instructions.  The N axis is ordered so that lane t of a quad holds channel t
// of both outputs: packing the results of two slices gives half of the projection's A fragment with no shuffle.  Channels are
// permuted to match when the weights are packed.
//
// Walk.  A unit is a tile of output pixels of one image (or whole small images); its CTA - or cluster of CTAs, each taking
// every ks-th chunk of the hidden channels, their partial sums stored into the shared memory of the CTA that adds them up, in
// rank order - walks the hidden channels in chunks of 16 or 32: the first operator of chunk c+1 into one of two hidden tiles while the depthwise
// operator and the projection consume chunk c from the other; one barrier per chunk.  Weights arrive by cp.async, resident
// when they fit, else through a ring of four chunks; they are requested before the previous kernel has finished.
//
// Small launches.  Where there are fewer units than SMs the chain of one unit is what a launch takes: up to 16 sets of warps
// then share a chunk, 16 hidden channels each (BlockCfg::wk), so that a warp's chain is one or two first operators, depthwise
// slices and projections; where its pixels lie is worked out before the previous kernel has finished, only the copies are
// issued behind it.  Of a launch of 14x14 64 -> 384 -> 64 at batch 1 with a cluster alone (8.7 us in a chain of such launches), 0.9
// us were the addresses, 3.3 the three chunks, 0.8 the cluster barrier and 3.0 reading the neighbours' sums one round trip after
// the other; with sets of warps and pushed sums 8.0 us a launch, 14x14 96 -> 576 -> 96 8.2 against 9.5.  Inside the networks:
// MobileNetV2 batch 1 169 -> 160 us, 8 x 192 207 -> 186, segmentation batch 1 229 -> 211.
//
// What bounds it.  Small launches: that chain.  Large ones: block_ws_kernel.  Measured on one B200 against separate kernels, stem included
// (stem_block.cu), MobileNetV2: batch 1 225 -> 155 us, 21 images of 205 pixels 340 -> 270 (248 with specialised warps), batch 256
// 1413 -> 1298 (1193); segmentation network batch 1 289 -> 207 (198), batch 16 961 -> 748 (684).
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <type_traits>

#include "bias_split.h"
#include "kernels.h"
#include "mma_frag.cuh"
#include "pdl.cuh"
#include "sm100_ptx.cuh"

namespace gi {
namespace {

using namespace ptx;
using namespace frag;

constexpr int kSubFixed = kBiasBytes + kTableBytes + kDwBiasBytes;
constexpr int kRing = 4;
constexpr int kSmemPerSm = 227 * 1024;

// How the first operator is computed: none (the input is the hidden tensor), a 1x1 expansion from up to 16 / 24 / 32 / 160
// channels
enum First { kNone = 0, kExp16 = 1, kExp24 = 2, kExp32 = 3, kExpWide = 4 };

// Bytes between the slices of a hidden tile: a constant, so that slices are immediate offsets.  32 modulo 128: the stores
// of 4 pixels x 4 slices by half a warp meet 32 different banks.
__host__ __device__ constexpr int slice_bytes(int first, bool small) { return (small ? 9 : first == kExpWide ? 18 : 36) * 128 + 32; }
__host__ __device__ constexpr int tile_pixels(int first, bool small) { return slice_bytes(first, small) / 8 - 2; }
// warps an SM holds: 128 registers a thread for 16 warps, 255 for 8 (96 sums per thread and more; tr: output rows a warp
// walks down), 168 for 12 where 64 sums and the fragments of four rows do not fit 128 (28x28 32 -> 192 -> 32 at batch 256: 77 us
// with 416 bytes of spills in the loop, 69 with 12 warps; 26x26 at batch 21 18.7 -> 16.9)
// ws: the kernel with specialised warps; 96 sums then fit 168 registers
__host__ __device__ constexpr int max_warps(int s, int np, int tr, bool ws = false) {
  return ws && np == 6 && (s == 2 || tr == 1) ? 12 : (s == 1 ? tr : 1) * np >= 6 || tr == 4 ? 8 : s == 1 && tr == 2 && np == 2 ? 12 : 16;
}
// bytes of one 16-channel sub-block of packed weights: first operator's fragments and bias, banded depthwise operands and
// bias, projection fragments
__host__ __device__ constexpr int sub_bytes(int ke, int np) { return ke * 512 + kSubFixed + np * 512; }
// ... of the kernel with specialised warps: behind it the expansion's bias as B operand, [fragment][column][two words]
constexpr int kOnesBytes = 128;
__host__ __device__ constexpr int ws_sub_bytes(int ke, int np) { return sub_bytes(ke, np) + kOnesBytes; }

struct BlockParams {
  const __half* in;
  const __half* res;
  __half* out;
  const unsigned char* wts;
  const float* bias;  // projection bias, 16 * NP floats
  int B, H, W, Ho, Wo;                  // depthwise input and output planes
  int in_px, in_img;                    // elements between pixels / images of the input
  int o_px, res_img;                    // ... between pixels of the output, images of the residual (its pixels: 4)
  long long in_sl, o_sl, o_img, res_sl; // elements between slices (and output images)
  int sin, sout;      // input and output slices
  int ke;             // 16-channel steps of a wide expansion's sum
  int pad_t, pad_l;
  int tw, nb, ni;     // output columns of a tile, bands of TR output rows, images of a unit
  int tiles_x, tiles_y, units;
  int rows, pitch, sub_px;  // hidden tile of one image: rows, pixels per row (even), rows * pitch
  int n_list, mt;           // pixels the first operator computes, in groups of 16
  int whole;                // a unit is whole images
  int compact;              // the list holds image pixels only; the border of the hidden tile stays zero
  int pw, ncols, ngroups;   // columns per band; columns and groups of 16 columns of a unit
  int eg, en;               // groups of 16 list pixels for a warp with / without a column group
  int nch, ks;              // chunks of hidden channels; CTAs sharing a unit
  int wk, nwq;              // sets of warps that share a chunk's channels; warps of a set
  int resident;
  unsigned x_pitch;
  unsigned off_bias, off_tab, off_src, off_x, off_hid, off_red;
  unsigned x_bytes, tab_bytes;  // of one of the two input tiles / tables (narrow expansions; otherwise there is one)
  unsigned mul_pitch, mul_w, mul_hw, mul_per, mul_tx;  // ceil(2^32 / d): division of a small number by d is one high multiplication
  unsigned hi_e, hi_d;  // upper clamp of the hidden activations, two halves (6; hi_e: or the largest finite value, hi_d: or infinity)
  int act_pre, act_post, has_res;
  int res_x;            // the residual is the block's input: it is still in shared memory
  int wide;             // both pixels of a pair are one aligned 16-byte store
  int pad_px;           // an odd plane holds one more pixel: zero it
};

__device__ __forceinline__ void cp_async16(unsigned dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// 8 bytes, or zeros in their place where there is nothing to read.  (A predicate: a size in a register costs 14 more instructions.)
__device__ __forceinline__ void cp_async8(unsigned dst, const void* src, bool in) {
  asm volatile("{\n\t.reg .pred none;\n\tsetp.eq.u32 none, %2, 0;\n\tcp.async.ca.shared.global [%0], [%1], 8, none;\n\t}" ::"r"(dst), "l"(src),
               "r"(static_cast<unsigned>(in))
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A barrier of `n` threads of the CTA that some only arrive at
__device__ __forceinline__ void named_sync(int id, int n) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void named_arrive(int id, int n) { asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(n) : "memory"); }

__device__ __forceinline__ void st_cluster_f4(unsigned addr, float a, float b, float c, float d) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}
// Four consecutive channels (one pixel-slice) of the projection, bias included: activation, residual, activation, fp16.
__device__ __forceinline__ uint2 finish4(const BlockParams& p, float v0, float v1, float v2, float v3, const uint2& r) {
  if (p.act_pre != GI_ACT_NONE) {
    v0 = act_f(v0, p.act_pre);
    v1 = act_f(v1, p.act_pre);
    v2 = act_f(v2, p.act_pre);
    v3 = act_f(v3, p.act_pre);
  }
  if (p.has_res) {
    const float2 r01 = __half22float2(*reinterpret_cast<const __half2*>(&r.x));
    const float2 r23 = __half22float2(*reinterpret_cast<const __half2*>(&r.y));
    v0 += r01.x;
    v1 += r01.y;
    v2 += r23.x;
    v3 += r23.y;
    if (p.act_post != GI_ACT_NONE) {
      v0 = act_f(v0, p.act_post);
      v1 = act_f(v1, p.act_post);
      v2 = act_f(v2, p.act_post);
      v3 = act_f(v3, p.act_post);
    }
  }
  return make_uint2(pack_f16x2<false>(v0, v1), pack_f16x2<false>(v2, v3));
}

struct UnitPos {
  int img0, y0, x0;  // first image, first output row / column
};
__host__ __device__ __forceinline__ UnitPos unit_pos(const BlockParams& p, int unit, int th_rows) {
  UnitPos u;
  if (p.whole || p.tiles_x * p.tiles_y == 1) {
    u.img0 = unit * p.ni;
    u.y0 = u.x0 = 0;
  } else {
    u.img0 = div_by(unit, p.mul_per);
    const int r = unit - u.img0 * (p.tiles_x * p.tiles_y);
    const int ty = p.tiles_x == 1 ? r : div_by(r, p.mul_tx);
    u.y0 = ty * th_rows;
    u.x0 = (r - ty * p.tiles_x) * p.tw;
  }
  return u;
}

// Where pixel `i` of the unit's list lies: `hid` is its pixel index in the hidden tile; (im, y, x) its place in the
// depthwise input; `in` says whether that is inside the image.
struct ListPx {
  int hid, im, y, x;
  bool in;
};
__host__ __device__ __forceinline__ ListPx list_pixel(const BlockParams& p, const UnitPos& u, int stride, int i) {
  ListPx l;
  if (p.compact) {
    l.im = div_by(i, p.mul_hw);
    const int rem = i - l.im * (p.H * p.W);
    l.y = div_by(rem, p.mul_w);
    l.x = rem - l.y * p.W;
    const int r = l.y + p.pad_t, c = l.x + p.pad_l;
    l.hid = (r < p.rows && c < p.pitch) ? l.im * p.sub_px + r * p.pitch + c : p.ni * p.sub_px;  // else: a pixel nothing reads
    l.in = u.img0 + l.im < p.B;
  } else {
    const int q = div_by(i, p.mul_pitch);
    const int c = i - q * p.pitch;
    l.im = p.ni > 1 ? q / p.rows : 0;
    l.y = u.y0 * stride - p.pad_t + (q - l.im * p.rows);
    l.x = u.x0 * stride - p.pad_l + c;
    l.hid = i;
    l.in = static_cast<unsigned>(l.y) < static_cast<unsigned>(p.H) && static_cast<unsigned>(l.x) < static_cast<unsigned>(p.W) &&
           u.img0 + l.im < p.B;
  }
  return l;
}

// Column `col` of the unit's column list -> image, band, position (pair or single column) within the band.
__host__ __device__ __forceinline__ void column_pos(const BlockParams& p, int col, int& im, int& band, int& pos) {
  const int q = col / p.pw;
  pos = col - q * p.pw;
  im = q / p.nb;
  band = q - im * p.nb;
}

// A lane's output column relative to the unit, in one word (the kernel is short of registers): image (0xff: no column), first
// row, x.
__device__ __forceinline__ unsigned lane_col(const BlockParams& p, int stride, int tr, int col) {
  int im, band, pos;
  column_pos(p, col < p.ncols ? col : 0, im, band, pos);
  return static_cast<unsigned>(col < p.ncols ? im : 0xff) << 24 | static_cast<unsigned>(band * tr) << 12 |
         static_cast<unsigned>(stride == 1 ? 2 * pos : pos);
}

// Store one column's projection results, of 16-channel blocks j0 .. j0 + NJ - 1.  a[v][j][q][f]; HALF: which half of a fragment
// the column is.  Stride 1: v = row (from v0), q = pixel of the pair; stride 2: v = row pair, q = row of it.
template <int S, int HALF, int NV, int NJ>
__device__ __forceinline__ void store_col(const BlockParams& p, const UnitPos& u, unsigned xres, unsigned col, int v0, int j0, int t,
                                          const float (&a)[NV][NJ][2][2][4]) {
  constexpr int H2 = HALF * 2;
  const int img = u.img0 + static_cast<int>(col >> 24), x = u.x0 + static_cast<int>(col & 0xfffu);
  const int y0 = u.y0 + static_cast<int>(col >> 12 & 0xfffu) + (S == 1 ? v0 : 2 * v0);
  if (col >> 24 == 0xffu || img >= p.B || x >= p.Wo) return;
  const int px0 = y0 * p.Wo + x, rows = p.Ho - y0;
  const bool two = S == 1 && x + 1 < p.Wo;
  const int o_row = p.Wo * p.o_px, r_row = p.Wo * 4;
  constexpr int kRows = S == 1 ? NV : 2 * NV;
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const int slice = 4 * (j0 + j) + t;
    if (slice >= p.sout) continue;
    __half* dst = p.out + (slice * p.o_sl + img * p.o_img + static_cast<long long>(px0) * p.o_px);
    uint2 r0[kRows], r1[kRows];  // the residual of all rows first: their latencies overlap
    if (S == 1 && p.res_x) {
      const unsigned i = (static_cast<unsigned>(img - u.img0) * p.rows + (y0 - u.y0) + p.pad_t) * p.pitch + (x - u.x0) + p.pad_l;
      unsigned at = xres + i * p.x_pitch + slice * 8;
#pragma unroll
      for (int v = 0; v < kRows; ++v, at += p.pitch * p.x_pitch) {
        r0[v] = lds64(at);
        r1[v] = lds64(at + p.x_pitch);
      }
    } else if (p.has_res) {
      const __half* rs = p.res + (slice * p.res_sl + static_cast<long long>(img) * p.res_img + static_cast<long long>(px0) * 4);
#pragma unroll
      for (int v = 0; v < kRows; ++v, rs += r_row) {
        if (v >= rows) break;
        if (S == 1 && p.wide) {
          const uint4 rr = *reinterpret_cast<const uint4*>(rs);
          r0[v] = make_uint2(rr.x, rr.y);
          r1[v] = make_uint2(rr.z, rr.w);
        } else {
          r0[v] = *reinterpret_cast<const uint2*>(rs);
          if (two) r1[v] = *reinterpret_cast<const uint2*>(rs + 4);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < kRows; ++v, dst += o_row) {
      if (v >= rows) break;
      if (S == 1) {
        const uint2 o0 = finish4(p, a[v][j][0][0][H2], a[v][j][0][0][H2 + 1], a[v][j][0][1][H2], a[v][j][0][1][H2 + 1], r0[v]);
        const uint2 o1 = finish4(p, a[v][j][1][0][H2], a[v][j][1][0][H2 + 1], a[v][j][1][1][H2], a[v][j][1][1][H2 + 1], r1[v]);
        if (p.wide) {
          *reinterpret_cast<uint4*>(dst) = make_uint4(o0.x, o0.y, o1.x, o1.y);
        } else {
          *reinterpret_cast<uint2*>(dst) = o0;
          if (two) *reinterpret_cast<uint2*>(dst + p.o_px) = o1;
          if (p.pad_px && v == rows - 1 && x + (two ? 1 : 0) == p.Wo - 1) *reinterpret_cast<uint2*>(dst + (two ? 8 : 4)) = make_uint2(0, 0);
        }
      } else {
        const float(&f)[2][4] = a[v / 2][j][v & 1];
        *reinterpret_cast<uint2*>(dst) = finish4(p, f[0][H2], f[0][H2 + 1], f[1][H2], f[1][H2 + 1], r0[v]);
        if (p.pad_px && v == rows - 1 && x == p.Wo - 1) *reinterpret_cast<uint2*>(dst + 4) = make_uint2(0, 0);
      }
    }
  }
}

// Which half of a banded weight word a lane takes, where its words lie, and whether it is a lane of the second output row (stride 2).
struct BandSel {
  unsigned a, b, a0, b0, a1, b1, entry;
  bool odd;
};
__device__ __forceinline__ BandSel band_sel(int lane) {
  const int g = lane >> 2, t = lane & 3;
  const bool band_lane = (g >> 2) == (t & 1);
  BandSel s;
  s.a = !band_lane ? 0x4444u : ((g >> 1) & 1) ? 0x1044u : 0x4410u;
  s.b = !band_lane ? 0x4444u : ((g >> 1) & 1) ? 0x3244u : 0x4432u;
  s.odd = g & 1;
  s.a0 = s.odd ? 0x4444u : s.a;  // window rows of the first output row only
  s.b0 = s.odd ? 0x4444u : s.b;
  s.a1 = s.odd ? s.a : 0x4444u;  // ... of the second only
  s.b1 = s.odd ? s.b : 0x4444u;
  s.entry = ((t >> 1) * 8 + g) * 16;
  return s;
}

// Depthwise operator and projection of HC sub-blocks of 16 hidden channels for one group of 16 columns, added to `acc`.  ws: the
// chunk's packed weights; hb: the lane's place in the hidden tile's first slice; row_b: bytes between hidden rows.
template <int S, int NP, int TR, int HC, int SL>
__device__ __forceinline__ void depthwise_project(unsigned ws, int ke, int subb, unsigned hb, unsigned row_b, int lane, unsigned hi_d,
                                                  const BandSel& sel, float (&acc)[S == 1 ? TR : TR / 2][NP][2][2][4]) {
  constexpr int NV = S == 1 ? TR : TR / 2;
  const int t = lane & 3;
  constexpr int kRows = S == 1 ? TR + 2 : 2 * TR + 1;  // hidden rows under the column
  unsigned rb[kRows];
#pragma unroll
  for (int i = 0; i < kRows; ++i) rb[i] = hb + i * row_b;
#pragma unroll
  for (int h = 0; h < HC; ++h) {
    const unsigned wd = ws + h * subb + ke * 512 + kBiasBytes;
    unsigned af[NV][2][4];
#pragma unroll
    for (int sp = 0; sp < 2; ++sp) {
      float d[2][NV][4], bd[2];
#pragma unroll
      for (int s2 = 0; s2 < 2; ++s2) {
        const int sl = sp * 2 + s2;
        const uint4 w = lds128(wd + sl * 256 + sel.entry);
        bd[s2] = __uint_as_float(lds32(wd + kTableBytes + sl * 64 + t * 16));
        if (S == 1) {
          const unsigned b0[3] = {prmt(w.x, sel.a), prmt(w.y, sel.a), prmt(w.z, sel.a)};
          const unsigned b1[3] = {prmt(w.x, sel.b), prmt(w.y, sel.b), prmt(w.z, sel.b)};
#pragma unroll
          for (int rr = 0; rr < kRows; ++rr) {
            unsigned a[4];
            ldsm4(rb[rr] + (h * 4 + sl) * SL, a);
#pragma unroll
            for (int ky = 0; ky < 3; ++ky) {
              const int v = rr - ky;
              if (v < 0 || v >= TR) continue;
              if (ky == 0) mma16816z(d[s2][v], a, b0[ky], b1[ky]);
              else mma16816(d[s2][v], a, b0[ky], b1[ky]);
            }
          }
        } else {
          const unsigned wm = sel.odd ? w.x : w.z;
          const unsigned b0[5] = {prmt(w.x, sel.a0), prmt(w.y, sel.a0), prmt(wm, sel.a), prmt(w.y, sel.a1), prmt(w.z, sel.a1)};
          const unsigned b1[5] = {prmt(w.x, sel.b0), prmt(w.y, sel.b0), prmt(wm, sel.b), prmt(w.y, sel.b1), prmt(w.z, sel.b1)};
#pragma unroll
          for (int rr = 0; rr < kRows; ++rr) {
            unsigned a[4];
            ldsm4(rb[rr] + (h * 4 + sl) * SL, a);
            const int v = rr >> 2, q = rr & 3;
            if (v < NV && q == 0) mma16816z(d[s2][v < NV ? v : 0], a, b0[q], b1[q]);
            else if (v < NV) mma16816(d[s2][v < NV ? v : 0], a, b0[q], b1[q]);
            if (q == 0 && v > 0) mma16816(d[s2][v > 0 ? v - 1 : 0], a, b0[4], b1[4]);
          }
        }
      }
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int s2 = 0; s2 < 2; ++s2) {  // the bias behind the sum: as its start value it would be moved into the accumulators
          add2(d[s2][v][0], d[s2][v][1], bd[s2], bd[s2]);
          add2(d[s2][v][2], d[s2][v][3], bd[s2], bd[s2]);
        }
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          af[v][q][sp * 2] = min_f16x2(pack_f16x2<true>(d[0][v][q], d[1][v][q]), hi_d);
          af[v][q][sp * 2 + 1] = min_f16x2(pack_f16x2<true>(d[0][v][2 + q], d[1][v][2 + q]), hi_d);
        }
    }
    const unsigned wp = wd + kTableBytes + kDwBiasBytes + lane * 16;
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const uint4 b = lds128(wp + j * 512);
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          mma16816(acc[v][j][q][0], af[v][q], b.x, b.y);
          mma16816(acc[v][j][q][1], af[v][q], b.z, b.w);
        }
    }
  }
}

// Partial sums of a cluster's CTAs and of warp sets: every tile of 16 columns x 16 channels has an owner, the CTA tile % ks;
// everybody stores into the owner's shared memory (source `src` of `n_src`), which then adds up its tiles in the order of the
// sources.  (Reading the neighbours' shared memory instead took 2.5 us: eight round trips, one after the other.)
// push_sums calls store(address, four sums).
template <int NV, int NP, class F>
__device__ __forceinline__ void push_sums(const BlockParams& p, unsigned red, int group, int src, int n_src, int lane,
                                          const float (&acc)[NV][NP][2][2][4], F&& store) {
#pragma unroll
  for (int v = 0; v < NV; ++v)
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int ti = (group * NV + v) * NP + j, slot = ti / p.ks;
      unsigned at = red + (slot * n_src + src) * 2048 + lane * 16;
      if (p.ks > 1) at = mapa_shared(at, ti - slot * p.ks);
#pragma unroll
      for (int i = 0; i < 4; ++i) store(at + i * 512, acc[v][j][i >> 1][i & 1]);
    }
}
template <int S, int TR, int NV, int NP>
__device__ __forceinline__ void add_sums(const BlockParams& p, const UnitPos& u, unsigned xs, unsigned red, int rank, int n_src, int warp,
                                         int warps, int lane) {
  const int g = lane >> 2, t = lane & 3, tiles = p.ngroups * NV * NP;
  for (int slot = warp; slot * p.ks + rank < tiles; slot += warps) {
    float s[1][1][2][2][4];
#pragma unroll
    for (int i = 0; i < 16; ++i) s[0][0][i >> 3][(i >> 2) & 1][i & 3] = 0.0f;
    unsigned at = red + slot * n_src * 2048 + lane * 16;
#pragma unroll 2
    for (int r = 0; r < n_src; ++r, at += 2048) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint4 x = lds128(at + i * 512);
        s[0][0][i >> 1][i & 1][0] += __uint_as_float(x.x);
        s[0][0][i >> 1][i & 1][1] += __uint_as_float(x.y);
        s[0][0][i >> 1][i & 1][2] += __uint_as_float(x.z);
        s[0][0][i >> 1][i & 1][3] += __uint_as_float(x.w);
      }
    }
    const int ti = slot * p.ks + rank, j = ti % NP, gv = ti / NP, gid = gv / NV, v = gv % NV;
    store_col<S, 0, 1, 1>(p, u, xs, lane_col(p, S, TR, gid * 16 + g), v, j, t, s);
    store_col<S, 1, 1, 1>(p, u, xs, lane_col(p, S, TR, gid * 16 + g + 8), v, j, t, s);
  }
}

// S: stride.  NP: 16-channel blocks of the output.  TR: output rows a warp walks down.  HC: 16-channel sub-blocks per chunk.
// SMALL: tiles of at most 146 list pixels, whose chunks several sets of warps share.
template <int S, int FIRST, int NP, int TR, int HC, bool SMALL>
__global__ void __launch_bounds__(32 * max_warps(S, NP, TR), 1) block_mma_kernel(const BlockParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const unsigned smem = smem_u32(smem_raw);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  constexpr bool kHasFirst = FIRST != kNone, kWideExp = FIRST == kExpWide;
  constexpr int SL = slice_bytes(FIRST, SMALL);
  constexpr int kSetBytes = HC * 4 * SL;
  const int wk = SMALL ? p.wk : 1, wset = SMALL ? warp / p.nwq : 0, wq = SMALL ? warp - wset * p.nwq : warp;
  const int hid_bytes = wk * kSetBytes;
  constexpr int NV = S == 1 ? TR : TR / 2;  // fragments of sums down a column: rows, or pairs of rows
  const int ke = kWideExp ? p.ke : FIRST == kNone ? 0 : FIRST == kExp16 ? 1 : 2;
  const int subb = ke * 512 + kSubFixed + NP * 512;
  const int stage_bytes = wk * HC * subb;
  const int rank = p.ks > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int unit0 = blockIdx.x / p.ks, ustep = gridDim.x / p.ks;
  const int nchl = (p.nch - rank + p.ks - 1) / p.ks;  // chunks of this CTA: rank, rank + ks, ...
  const int th_rows = p.nb * TR;
  const int my_units = unit0 < p.units ? (p.units - unit0 + ustep - 1) / ustep : 0;
  const int total = nchl * my_units;

  pdl_launch_dependents();
  if (p.ks > 1) cluster_arrive();  // (waited for before the first store into a neighbour's shared memory)

  auto load_weights = [&](int run, int c) {
    const unsigned dst = smem + (p.resident ? run : run & (kRing - 1)) * stage_bytes;
    const unsigned char* src = p.wts + static_cast<size_t>(rank + c * p.ks) * stage_bytes;
    for (int i = tid * 16; i < stage_bytes; i += nthr * 16) cp_async16(dst + i, src + i);
  };
  if (p.resident) {
    for (int c = 0; c < nchl; ++c) load_weights(c, c);
  } else {
    load_weights(0, 0);
    if (1 < total) load_weights(1, 1 % nchl);
  }
  // shared memory that must start at zero: borders of compact tiles, and the slices beyond the input's last one that the first
  // operator's steps of 16 channels read (their weights are zero, but 0 x NaN is not)
  const int step_slices = FIRST == kExp24 ? 6 : 4 * ke;
  if (p.compact || p.sin < step_slices) {
    for (unsigned i = p.off_x + tid * 16; i < p.off_red; i += nthr * 16) sts128(smem + i, 0u, 0u, 0u, 0u);
  }
  for (int i = tid; i < NP * 4; i += nthr) cp_async16(smem + p.off_bias + i * 16, reinterpret_cast<const float4*>(p.bias) + i);

  const unsigned tab0 = smem + p.off_tab, xs0 = smem + p.off_x, hid0 = smem + p.off_hid, red = smem + p.off_red;
  constexpr bool kTwoX = kHasFirst && !kWideExp;  // the next unit's input arrives during this one

  // expansion: the unit's input tile, [list pixel][channel].  The table says what a list pixel's hidden value is clamped to
  // (zero outside the image); for a wide expansion, whose list may leave out the border, also where it goes
  auto load_x = [&](const UnitPos& u, int buf) {
    const unsigned xs = xs0 + buf * p.x_bytes, tab = tab0 + buf * p.tab_bytes;
    constexpr int kSlices = FIRST == kExp16 ? 4 : FIRST == kExp24 ? 6 : FIRST == kExp32 ? 8 : 0;
    for (int i = tid; i < p.mt * 16; i += nthr) {
      const bool listed = i < p.n_list;
      const ListPx l = list_pixel(p, u, S, listed ? i : 0);
      const bool in = listed && l.in;
      if (listed) {
        const __half* src = p.in;
        if (in) src += static_cast<long long>(u.img0 + l.im) * p.in_img + static_cast<long long>(l.y * p.W + l.x) * p.in_px;
        const long long step = in ? p.in_sl : 0;
        unsigned dst = xs + i * p.x_pitch;
        if (kTwoX) {
#pragma unroll
          for (int s = 0; s < kSlices; ++s, src += step)
            if (s < p.sin) cp_async8(dst + s * 8, src, in);
        } else {
          for (int s = 0; s < p.sin; ++s, src += step, dst += 8) cp_async8(dst, src, in);
        }
      }
      if (kWideExp) sts64(tab + i * 8, static_cast<unsigned>(listed ? l.hid : p.ni * p.sub_px) * 8u, in ? p.hi_e : 0u);
      else sts32(tab + i * 4, in ? p.hi_e : 0u);
    }
  };
  // small tiles: the first unit's input in two steps: where its pixels lie is found out before the previous kernel has finished
  auto find_x = [&](const UnitPos& u) {
    for (int i = tid; i < p.mt * 16; i += nthr) {
      const bool listed = i < p.n_list;
      const ListPx l = list_pixel(p, u, S, listed ? i : 0);
      const bool in = listed && l.in;
      sts32(smem + p.off_src + i * 4, static_cast<unsigned>(in ? (u.img0 + l.im) * p.in_img + (l.y * p.W + l.x) * p.in_px : -1));
      if (kWideExp) sts64(tab0 + i * 8, static_cast<unsigned>(listed ? l.hid : p.ni * p.sub_px) * 8u, in ? p.hi_e : 0u);
      else sts32(tab0 + i * 4, in ? p.hi_e : 0u);
    }
  };
  auto copy_x = [&]() {
    const int px = p.n_list, parts = max(1, nthr / px), part = nthr >= 2 * px ? tid / px : 0;
    if (part >= parts) return;
    for (int i = tid - part * px; i < px; i += nthr) {
      const int at = static_cast<int>(lds32(smem + p.off_src + i * 4));
      const unsigned dst = xs0 + i * p.x_pitch;
      const __half* src = p.in + max(at, 0);
#pragma unroll 4
      for (int s = part; s < p.sin; s += parts) cp_async8(dst + s * 8, at >= 0 ? src + s * p.in_sl : p.in, at >= 0);
    }
  };
  // no first operator: a chunk of the input goes straight into a hidden tile (a ring of them)
  auto load_hidden = [&](int run) {
    const int k = run / nchl, c = run - k * nchl, chunk = rank + c * p.ks;
    if (c == 0) {  // a thread's own pixels of the unit, kept for its other chunks
      const UnitPos u = unit_pos(p, unit0 + k * ustep, th_rows);
      for (int i = tid; i < p.n_list; i += nthr) {
        const ListPx l = list_pixel(p, u, S, i);
        sts32(tab0 + i * 4, static_cast<unsigned>(l.in ? (u.img0 + l.im) * p.in_img + (l.y * p.W + l.x) * p.in_px : -1));
      }
    }
    unsigned dst = hid0 + (run & (kRing - 1)) * hid_bytes + tid * 8;
    const int s0 = chunk * wk * HC * 4, ns = p.sin - s0;  // slices beyond the last one are zeros: their weights are, too
    for (int i = tid; i < p.n_list; i += nthr, dst += nthr * 8) {
      const int at = static_cast<int>(lds32(tab0 + i * 4));
      const __half* src = p.in + (at < 0 ? 0 : at) + s0 * p.in_sl;
      for (int w = 0; w < wk * HC * 4; w += HC * 4)
#pragma unroll
        for (int s = w; s < w + HC * 4; ++s, src += p.in_sl) cp_async8(dst + s * SL, s < ns ? src : p.in, s < ns && at >= 0);
    }
  };
  if (SMALL && kHasFirst) find_x(unit_pos(p, unit0, th_rows));
  __syncthreads();
  pdl_wait();
  if (my_units > 0) {
    if (kHasFirst) {
      if (SMALL) copy_x();
      else load_x(unit_pos(p, unit0, th_rows), 0);
    } else {
      load_hidden(0);
      cp_async_commit();
      if (1 < total) load_hidden(1);
    }
  }
  cp_async_commit();

  // this lane's rows of the depthwise A operand, and which half of a banded weight word it takes
  unsigned dw_base;
  const unsigned row_b = p.pitch * 8;
  {
    int col = wq * 16 + (lane & 15);
    if (col >= p.ncols) col = 0;
    int im, band, pos;
    column_pos(p, col, im, band, pos);
    dw_base = static_cast<unsigned>(im * p.sub_px + band * TR * S * p.pitch) * 8u + pos * 16u + (lane >> 4) * 16u;
  }
  const unsigned col0 = lane_col(p, S, TR, wq * 16 + g), col1 = lane_col(p, S, TR, wq * 16 + g + 8);
  const BandSel sel = band_sel(lane);
  const bool has_group = wq < p.ngroups;
  // this warp's groups of 16 list pixels
  const int mt0 = has_group ? wq * p.eg : p.ngroups * p.eg + (wq - p.ngroups) * p.en;
  const int mt1 = min(p.mt, mt0 + (has_group ? p.eg : p.en));

  if (kHasFirst) cp_async_wait<0>();
  else cp_async_wait<1>();
  __syncthreads();
  int run = 0;
  for (int k = 0; k < my_units; ++k, run += nchl) {
    const int unit = unit0 + k * ustep;
    float acc[NV][NP][2][2][4];  // sums start at the bias (a cluster's: in its first CTA)
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const uint4 q = rank || wset ? make_uint4(0u, 0u, 0u, 0u) : lds128(smem + p.off_bias + (4 * j + t) * 16);
#pragma unroll
      for (int v = 0; v < NV; ++v)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[v][j][i >> 1][0][(i & 1) * 2] = __uint_as_float(q.x);
          acc[v][j][i >> 1][0][(i & 1) * 2 + 1] = __uint_as_float(q.y);
          acc[v][j][i >> 1][1][(i & 1) * 2] = __uint_as_float(q.z);
          acc[v][j][i >> 1][1][(i & 1) * 2 + 1] = __uint_as_float(q.w);
        }
    }
    const unsigned xs = xs0 + (kTwoX ? (k & 1) * p.x_bytes : 0u), tab = tab0 + (kTwoX ? (k & 1) * p.tab_bytes : 0u);
    const int steps = kHasFirst ? nchl + 1 : nchl;
#pragma unroll 1
    for (int it = 0; it < steps; ++it) {
      if (kHasFirst && !kTwoX && it == 0) cp_async_wait<0>();
      else cp_async_wait<1>();
      __syncthreads();
      if (kHasFirst) {
        if (!p.resident && it < nchl && run + it + 2 < total) load_weights(run + it + 2, it + 2 >= nchl ? (it + 2) % nchl : it + 2);
        if (k + 1 < my_units) {
          if (kTwoX && it == 0) load_x(unit_pos(p, unit + ustep, th_rows), (k + 1) & 1);
          if (kWideExp && it == nchl) load_x(unit_pos(p, unit + ustep, th_rows), 0);
        }
      } else if (run + it + 2 < total) {
        if (!p.resident) load_weights(run + it + 2, (it + 2) % nchl);
        load_hidden(run + it + 2);
      }
      cp_async_commit();

      // ---- first operator of chunk `it`
      if (kHasFirst && it < nchl && mt0 < mt1) {
        const int r = run + it;
        const unsigned ws = smem + (p.resident ? it : r & (kRing - 1)) * stage_bytes + wset * HC * subb;
        const unsigned hb = hid0 + (r & 1) * hid_bytes + wset * kSetBytes + t * SL;
        if (!kWideExp) {
          const uint4 b0 = lds128(ws + lane * 16);
          const uint4 b1 = FIRST == kExp16 ? b0 : lds128(ws + 512 + lane * 16);
          const uint4 q = lds128(ws + ke * 512 + t * 16);
          const float be[4] = {__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), __uint_as_float(q.w)};
          constexpr unsigned XP = FIRST == kExp16 || FIRST == kExp24 ? 48 : 80;
          unsigned xa = xs + (mt0 * 16 + (lane & 15)) * XP + (lane >> 4) * 16;
          unsigned xh = xs + (mt0 * 16 + (lane & 15)) * XP + 32;  // kExp24: channels 16..23
          unsigned at = hb + (mt0 * 16 + g) * 8, tb = tab + (mt0 * 16 + g) * 4;
          auto some = [&](auto count) {  // `count` groups in flight
            constexpr int N = decltype(count)::value;
            unsigned a[N][4], a2[N][4], hi[N][2];
            float c[N][2][4];
#pragma unroll
            for (int i = 0; i < N; ++i) {
              ldsm4(xa + i * 16 * XP, a[i]);
              if (FIRST == kExp24) ldsm2(xh + i * 16 * XP, a2[i][0], a2[i][1]);
              if (FIRST == kExp32) ldsm4(xa + i * 16 * XP + 32, a2[i]);
              hi[i][0] = lds32(tb + i * 64);
              hi[i][1] = lds32(tb + i * 64 + 32);
            }
#pragma unroll
            for (int i = 0; i < N; ++i) {
              mma16816c(c[i][0], a[i], b0.x, b0.y, be[0], be[1], be[0], be[1]);
              mma16816c(c[i][1], a[i], b0.z, b0.w, be[2], be[3], be[2], be[3]);
              if (FIRST == kExp24) {
                mma1688(c[i][0], a2[i][0], a2[i][1], b1.x);
                mma1688(c[i][1], a2[i][0], a2[i][1], b1.z);
              }
              if (FIRST == kExp32) {
                mma16816(c[i][0], a2[i], b1.x, b1.y);
                mma16816(c[i][1], a2[i], b1.z, b1.w);
              }
            }
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
              for (int half = 0; half < 2; ++half)
                sts64(at + i * 128 + half * 64, min_f16x2(pack_f16x2<true>(c[i][0][half * 2], c[i][0][half * 2 + 1]), hi[i][half]),
                      min_f16x2(pack_f16x2<true>(c[i][1][half * 2], c[i][1][half * 2 + 1]), hi[i][half]));
            xa += N * 16 * XP;
            xh += N * 16 * XP;
            at += N * 128;
            tb += N * 64;
          };
          int n = mt1 - mt0;
#pragma unroll 1
          for (; n >= 2; n -= 2) some(std::integral_constant<int, 2>{});
          if (n) some(std::integral_constant<int, 1>{});
        } else {
          float be[HC][4];
#pragma unroll
          for (int h = 0; h < HC; ++h) {
            const uint4 q = lds128(ws + h * subb + ke * 512 + t * 16);
            be[h][0] = __uint_as_float(q.x);
            be[h][1] = __uint_as_float(q.y);
            be[h][2] = __uint_as_float(q.z);
            be[h][3] = __uint_as_float(q.w);
          }
#pragma unroll 1
          for (int m0 = mt0; m0 < mt1; m0 += 2) {  // two groups at a time share the weight fragments
            const bool second = m0 + 1 < mt1;
            float c[2][HC][2][4];
            unsigned xa = xs + (m0 * 16 + (lane & 15)) * p.x_pitch + (lane >> 4) * 16;
            const unsigned xb = second ? 16 * p.x_pitch : 0u;
            unsigned wk = ws + lane * 16;
            auto step = [&](auto first) {
              unsigned a[2][4];
              ldsm4(xa, a[0]);
              ldsm4(xa + xb, a[1]);
#pragma unroll
              for (int h = 0; h < HC; ++h) {
                const uint4 b = lds128(wk + h * subb);
#pragma unroll
                for (int mm = 0; mm < 2; ++mm) {
                  if (decltype(first)::value) {
                    mma16816c(c[mm][h][0], a[mm], b.x, b.y, be[h][0], be[h][1], be[h][0], be[h][1]);
                    mma16816c(c[mm][h][1], a[mm], b.z, b.w, be[h][2], be[h][3], be[h][2], be[h][3]);
                  } else {
                    mma16816(c[mm][h][0], a[mm], b.x, b.y);
                    mma16816(c[mm][h][1], a[mm], b.z, b.w);
                  }
                }
              }
              xa += 32;
              wk += 512;
            };
            step(std::true_type{});
#pragma unroll 2
            for (int kk = 1; kk < ke; ++kk) step(std::false_type{});
#pragma unroll
            for (int mm = 0; mm < 2; ++mm) {
              if (mm == 1 && !second) break;
#pragma unroll
              for (int half = 0; half < 2; ++half) {
                const uint2 e = lds64(tab + ((m0 + mm) * 16 + g + half * 8) * 8);
                const unsigned at = hb + e.x;
#pragma unroll
                for (int h = 0; h < HC; ++h)
                  sts64(at + h * 4 * SL, min_f16x2(pack_f16x2<true>(c[mm][h][0][half * 2], c[mm][h][0][half * 2 + 1]), e.y),
                        min_f16x2(pack_f16x2<true>(c[mm][h][1][half * 2], c[mm][h][1][half * 2 + 1]), e.y));
              }
            }
          }
        }
      }

      // ---- depthwise and projection of the chunk before it (without a first operator: of chunk `it`)
      const int dc = kHasFirst ? it - 1 : it;
      if (dc >= 0 && has_group) {
        const int r = run + dc;
        const unsigned ws = smem + (p.resident ? dc : r & (kRing - 1)) * stage_bytes + wset * HC * subb;
        const unsigned hb = hid0 + (kHasFirst ? (r & 1) : (r & (kRing - 1))) * hid_bytes + wset * kSetBytes + dw_base;
        depthwise_project<S, NP, TR, HC, SL>(ws, ke, subb, hb, row_b, lane, p.hi_d, sel, acc);
      }
    }

    const UnitPos u = unit_pos(p, unit, th_rows);
    if (p.ks * wk == 1) {
      if (has_group) {
        store_col<S, 0, NV, NP>(p, u, xs, col0, 0, 0, t, acc);
        store_col<S, 1, NV, NP>(p, u, xs, col1, 0, 0, t, acc);
      }
    } else {
      const int src = rank * wk + wset, n_src = p.ks * wk;
      if (p.ks > 1 && k == 0) cluster_wait();  // every CTA of the cluster has started
      if (has_group)
        push_sums<NV, NP>(p, red, wq, src, n_src, lane, acc, [&](unsigned at, const float(&f)[4]) {
          if (p.ks > 1) st_cluster_f4(at, f[0], f[1], f[2], f[3]);
          else sts128(at, __float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
        });
      if (p.ks > 1) cluster_sync();
      else __syncthreads();
      add_sums<S, TR, NV, NP>(p, u, xs, red, rank, n_src, warp, nthr >> 5, lane);
      if (k + 1 < my_units) {  // nobody overwrites what a neighbour still reads
        if (p.ks > 1) cluster_sync();
        else __syncthreads();
      }
    }
  }
  cp_async_wait<0>();
}

// The same with the two halves of a chunk on warps of their own: the first p.ngroups warps each own a group of columns and run its
// depthwise operator and projection, the others compute the expansion of the chunk after it and bring weights and the next tile's
// input.  A pair of barriers per hidden tile (complete, free) lets the two run up to two chunks apart.  For units that one CTA or a
// cluster computes, with four chunks of hidden channels or more; blocks without an expansion and small tiles, whose chunks sets of
// warps share, stay on the kernel above.
//
// What it is for: with both halves in one warp the projection's sums stay live through the expansion, the register file makes the
// compiler move them, and a warp that waits for its shared memory has nobody to take its place.  Of 129 M warp instructions of 112x112
// 16 -> 96 -> 24, stride 2, at batch 256 are left 98 M (some because a bias as a sum's start value costs four moves a matrix
// instruction: the expansion's comes as a product with ones in front of the others, with 17 to 24 channels beside the last eight, the
// depthwise operator's as one two-wide addition behind the sum).  Kernel above -> this one, us on one B200: that block 63.4 -> 52.3, 56x56 24 -> 144 -> 24 at batch 64 51.4 -> 43.7, 14x14
// 64 -> 384 -> 64 at batch 64 22.2 -> 17.7, 33x33 64 -> 384 -> 64 at batch 16 29.9 -> 25.3.  MobileNetV2 at batch 256 1299 -> 1192, 21
// images of 205 pixels 271 -> 250, segmentation at batch 16 748 -> 713.  What bounds it now: shared memory's pipe (67 % of its
// wavefronts on the first of these) and the latency from ldmatrix to store with 12 to 16 warps; the matrix pipe is 30 % busy.
template <int S, int FIRST, int NP, int TR>
__global__ void __launch_bounds__(32 * max_warps(S, NP, TR, true), 1) block_ws_kernel(const BlockParams p) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const unsigned smem = smem_u32(smem_raw);
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  constexpr bool kWide = FIRST == kExpWide;
  constexpr int SL = slice_bytes(FIRST, false), HC = kWide ? 2 : 1;
  constexpr int kHidBytes = HC * 4 * SL, kSlices = FIRST == kExp16 ? 4 : FIRST == kExp24 ? 6 : 8;
  constexpr int NV = S == 1 ? TR : TR / 2;
  const int ke = kWide ? p.ke : FIRST == kExp16 ? 1 : 2;
  const int subb = ws_sub_bytes(ke, NP), stage_bytes = HC * subb;
  const unsigned XP = kWide ? p.x_pitch : FIRST == kExp32 ? 80u : 48u;  // bytes of a list pixel
  const int th_rows = p.nb * TR;
  const int rank = p.ks > 1 ? static_cast<int>(cluster_ctarank()) : 0;
  const int unit0 = p.ks > 1 ? blockIdx.x / p.ks : blockIdx.x, ustep = p.ks > 1 ? gridDim.x / p.ks : gridDim.x;
  const int nch = p.ks > 1 ? (p.nch - rank + p.ks - 1) / p.ks : p.nch;  // chunks of this CTA: rank, rank + ks, ...
  const int my_units = (p.units - unit0 + ustep - 1) / ustep;           // (of a cluster: one)
  const int total = nch * my_units;
  const unsigned tab0 = smem + p.off_tab, xs0 = smem + p.off_x, hid0 = smem + p.off_hid, red = smem + p.off_red;

  pdl_launch_dependents();
  if (p.ks > 1) cluster_arrive();  // (waited for before the first store into a neighbour's shared memory)
  auto load_weights = [&](int run, int c, int i0, int n) {
    const unsigned dst = smem + (p.resident ? c : run & (kRing - 1)) * stage_bytes;
    const unsigned char* src = p.wts + static_cast<size_t>(rank + c * p.ks) * stage_bytes;
    for (int i = i0 * 16; i < stage_bytes; i += n * 16) cp_async16(dst + i, src + i);
  };
  // a unit's input tile, [list pixel][channel], and what its hidden pixels are clamped to (zero outside the image); for a wide
  // expansion, whose list may leave out the border, also where they go
  auto load_x = [&](const UnitPos& u, int buf, int i0, int n) {
    const int yb = u.y0 * S - p.pad_t, xb = u.x0 * S - p.pad_l;
    const __half* base = p.in + static_cast<long long>(u.img0) * p.in_img;
    const unsigned xs = xs0 + buf * p.x_bytes, tab = tab0 + buf * p.tab_bytes;
    for (int i = i0; i < p.mt * 16; i += n) {
      int at, hid = i;
      bool in;
      if (kWide) {
        const bool listed = i < p.n_list;
        const ListPx l = list_pixel(p, u, S, listed ? i : 0);
        in = listed && l.in;
        hid = listed ? l.hid : p.ni * p.sub_px;
        at = l.im * p.in_img + (l.y * p.W + l.x) * p.in_px;
      } else {
        const int q = div_by(i, p.mul_pitch), x = xb + (i - q * p.pitch), y = yb + q;
        in = i < p.n_list && static_cast<unsigned>(y) < static_cast<unsigned>(p.H) && static_cast<unsigned>(x) < static_cast<unsigned>(p.W);
        at = (y * p.W + x) * p.in_px;
      }
      const __half* src = in ? base + at : p.in;
      const long long step = in ? p.in_sl : 0;
      unsigned dst = xs + i * XP;
      if (kWide) {
#pragma unroll 4
        for (int s = 0; s < p.sin; ++s, src += step, dst += 8) cp_async8(dst, src, in);
        sts64(tab + i * 8, hid * 8u, in ? p.hi_e : 0u);
      } else {
#pragma unroll
        for (int s = 0; s < kSlices; ++s, src += step)
          if (s < p.sin) cp_async8(dst + s * 8, src, in);
        sts32(tab + i * 4, in ? p.hi_e : 0u);
      }
    }
  };
  for (int c = 0; c < (p.resident ? nch : 2); ++c) load_weights(c, c, tid, nthr);
  for (int i = tid; i < NP * 4; i += nthr) cp_async16(smem + p.off_bias + i * 16, reinterpret_cast<const float4*>(p.bias) + i);
  // shared memory that must start at zero: borders of compact tiles, and the slices beyond the input's last one that the
  // expansion's steps of 16 channels read (their weights are zero, but 0 x NaN is not)
  if (p.compact || p.sin < (FIRST == kExp24 ? 6 : 4 * ke)) {
    for (unsigned i = p.off_x + tid * 16; i < p.off_red; i += nthr * 16) sts128(smem + i, 0u, 0u, 0u, 0u);
    __syncthreads();
  }
  pdl_wait();
  load_x(unit_pos(p, unit0, th_rows), 0, tid, nthr);
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();

  const int ncons = p.ngroups;
  if (warp >= ncons) {
    // ---- expansion: groups of 16 list pixels; of a wide one, every second warp takes the second 16 channels of the chunk
    const int nprod = (nthr >> 5) - ncons, w = warp - ncons, ptid = tid - ncons * 32, np = nprod * 32;
    const int half_chunk = kWide ? w & 1 : 0, wg = kWide ? w >> 1 : w, nwg = kWide ? nprod >> 1 : nprod;
    const int mt0 = wg * p.mt / nwg, cnt = (wg + 1) * p.mt / nwg - mt0;
    const unsigned a_off = (mt0 * 16 + (lane & 15)) * XP + (lane >> 4) * 16, h_off = (mt0 * 16 + (lane & 15)) * XP + 32;
    const unsigned t_off = (mt0 * 16 + g) * (kWide ? 8 : 4), ones = ones_word(t);
    int r = 0;
#pragma unroll 1
    for (int k = 0; k < my_units; ++k) {
      const unsigned xs = xs0 + (k & 1) * p.x_bytes, tab = tab0 + (k & 1) * p.tab_bytes + t_off;
      unsigned edge = 0u;  // groups (of the first 32) with pixels outside the image
#pragma unroll 1
      for (int c = 0; c < nch; ++c, ++r) {
        cp_async_wait<1>();
        if (r >= 2) named_sync(3 + (r & 1), nthr);  // the hidden tile is free, and the copies of all these warps have arrived
        if (!p.resident && r + 2 < total) load_weights(r + 2, c + 2 >= nch ? c + 2 - nch : c + 2, ptid, np);
        // (the columns' warps have finished the unit before this one: its tile may be overwritten)
        if (c == 2 && k + 1 < my_units) load_x(unit_pos(p, unit0 + (k + 1) * ustep, th_rows), (k + 1) & 1, ptid, np);
        cp_async_commit();
        const unsigned ws = smem + (p.resident ? c : r & (kRing - 1)) * stage_bytes + half_chunk * subb;
        const unsigned hid = hid0 + (r & 1) * kHidBytes + (half_chunk * 4 + t) * SL;
        unsigned one[2] = {0u, 0u};  // the bias as B operand of one more step (24 channels: in the second step)
        if (FIRST != kExp24) {
          one[0] = lds32(ws + sub_bytes(ke, NP) + g * 8 + (t & 1) * 4);
          one[1] = lds32(ws + sub_bytes(ke, NP) + 64 + g * 8 + (t & 1) * 4);
        }
        if constexpr (kWide) {
          auto some = [&](auto count, int n) {  // `count` groups in flight
            constexpr int N = decltype(count)::value;
            float d[N][2][4];
            unsigned xa = xs + a_off + n * 16 * XP, wk = ws + lane * 16;
            const unsigned step = 16 * XP;
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
              for (int f = 0; f < 2; ++f) {
                d[i][f][0] = d[i][f][1] = d[i][f][2] = d[i][f][3] = 0.0f;
                mma1688(d[i][f], ones, ones, one[f]);
              }
            unsigned a[2][N][4];
            uint4 b[2];
            auto load = [&](int s) {  // (the next step's operands are under way while this one's are multiplied)
#pragma unroll
              for (int i = 0; i < N; ++i) ldsm4(xa + i * step, a[s][i]);
              b[s] = lds128(wk);
              xa += 32;
              wk += 512;
            };
            auto mul = [&](int s) {
#pragma unroll
              for (int i = 0; i < N; ++i) {
                mma16816(d[i][0], a[s][i], b[s].x, b[s].y);
                mma16816(d[i][1], a[s][i], b[s].z, b[s].w);
              }
            };
            load(0);
            int kk = 1;
#pragma unroll 1
            for (; kk + 2 <= ke; kk += 2) {
              load(1);
              mul(0);
              load(0);
              mul(1);
            }
            if (kk < ke) {
              load(1);
              mul(0);
              mul(1);
            } else {
              mul(0);
            }
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
              for (int half = 0; half < 2; ++half) {
                const uint2 e = lds64(tab + (n + i) * 128 + half * 64);
                sts64(hid + e.x, min_f16x2(pack_f16x2<true>(d[i][0][half * 2], d[i][0][half * 2 + 1]), e.y),
                      min_f16x2(pack_f16x2<true>(d[i][1][half * 2], d[i][1][half * 2 + 1]), e.y));
              }
          };
          int n = 0;
#pragma unroll 1
          for (; n + 3 <= cnt; n += 3) some(std::integral_constant<int, 3>{}, n);
          if (n + 2 <= cnt) some(std::integral_constant<int, 2>{}, n);
          else if (n < cnt) some(std::integral_constant<int, 1>{}, n);
        } else {
          if (c == 0) {
            edge = 0u;
            for (int n = 0; n < min(cnt, 32); ++n) {
              const bool out = lds32(tab + n * 64) != p.hi_e || lds32(tab + n * 64 + 32) != p.hi_e;
              edge |= __any_sync(0xffffffffu, out) ? 1u << n : 0u;
            }
          }
          const uint4 b0 = lds128(ws + lane * 16);
          const uint4 b1 = FIRST == kExp16 ? b0 : lds128(ws + 512 + lane * 16);
          unsigned xa = xs + a_off, xh = xs + h_off, tb = tab, at = hid + (mt0 * 16 + g) * 8;
          auto some = [&](auto count, auto masked) {  // `count` groups in flight
            constexpr int N = decltype(count)::value;
            constexpr bool kMasked = decltype(masked)::value;
            unsigned a[N][4], a2[N][4], hi[N][2];
            float d[N][2][4];
#pragma unroll
            for (int i = 0; i < N; ++i) {
              ldsm4(xa + i * 16 * XP, a[i]);
              if (FIRST == kExp24) {
                ldsm2(xh + i * 16 * XP, a2[i][0], a2[i][1]);
                a2[i][2] = a2[i][3] = ones;
              }
              if (FIRST == kExp32) ldsm4(xa + i * 16 * XP + 32, a2[i]);
              hi[i][0] = kMasked ? lds32(tb + i * 64) : p.hi_e;
              hi[i][1] = kMasked ? lds32(tb + i * 64 + 32) : p.hi_e;
            }
#pragma unroll
            for (int i = 0; i < N; ++i) {
              if (FIRST == kExp24) {
                mma16816z(d[i][0], a[i], b0.x, b0.y);
                mma16816z(d[i][1], a[i], b0.z, b0.w);
              } else {  // the bias first: behind the products its sum is rounded once more (32 channels: 10 % more stored values differ)
                mma1688z(d[i][0], ones, ones, one[0]);
                mma1688z(d[i][1], ones, ones, one[1]);
              }
            }
            if (FIRST != kExp24) {
#pragma unroll
              for (int i = 0; i < N; ++i) {
                mma16816(d[i][0], a[i], b0.x, b0.y);
                mma16816(d[i][1], a[i], b0.z, b0.w);
              }
            }
            if (FIRST != kExp16) {
#pragma unroll
              for (int i = 0; i < N; ++i) {
                mma16816(d[i][0], a2[i], b1.x, b1.y);
                mma16816(d[i][1], a2[i], b1.z, b1.w);
              }
            }
#pragma unroll
            for (int i = 0; i < N; ++i)
#pragma unroll
              for (int half = 0; half < 2; ++half)
                sts64(at + i * 128 + half * 64, min_f16x2(pack_f16x2<true>(d[i][0][half * 2], d[i][0][half * 2 + 1]), hi[i][half]),
                      min_f16x2(pack_f16x2<true>(d[i][1][half * 2], d[i][1][half * 2 + 1]), hi[i][half]));
            xa += N * 16 * XP;
            xh += N * 16 * XP;
            at += N * 128;
            tb += N * 64;
          };
          auto groups = [&](auto count, unsigned edges) {
            if (edges) some(count, std::true_type{});
            else some(count, std::false_type{});
          };
          int n = 0;
#pragma unroll 1
          for (; n + 4 <= cnt; n += 4) groups(std::integral_constant<int, 4>{}, n < 29 ? edge >> n & 15u : 1u);
          if (n + 2 <= cnt) {
            groups(std::integral_constant<int, 2>{}, n < 31 ? edge >> n & 3u : 1u);
            n += 2;
          }
          if (n < cnt) groups(std::integral_constant<int, 1>{}, n < 32 ? edge >> n & 1u : 1u);
        }
        named_arrive(1 + (r & 1), nthr);
      }
    }
    cp_async_wait<0>();
    if (p.ks == 1) return;
    cluster_wait();
  } else {
    // ---- depthwise operator and projection of this warp's columns
    unsigned dw_base;
    const unsigned row_b = p.pitch * 8;
    {
      int col = warp * 16 + (lane & 15);
      if (col >= p.ncols) col = 0;
      int im, band, pos;
      column_pos(p, col, im, band, pos);
      dw_base = static_cast<unsigned>(im * p.sub_px + band * TR * S * p.pitch) * 8u + pos * 16u + (lane >> 4) * 16u;
    }
    const BandSel sel = band_sel(lane);
    int r = 0;
#pragma unroll 1
    for (int k = 0; k < my_units; ++k) {
      float acc[NV][NP][2][2][4];
#pragma unroll
      for (int j = 0; j < NP; ++j) {
        const uint4 q = rank ? make_uint4(0u, 0u, 0u, 0u) : lds128(smem + p.off_bias + (4 * j + t) * 16);
#pragma unroll
        for (int v = 0; v < NV; ++v)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            acc[v][j][i >> 1][0][(i & 1) * 2] = __uint_as_float(q.x);
            acc[v][j][i >> 1][0][(i & 1) * 2 + 1] = __uint_as_float(q.y);
            acc[v][j][i >> 1][1][(i & 1) * 2] = __uint_as_float(q.z);
            acc[v][j][i >> 1][1][(i & 1) * 2 + 1] = __uint_as_float(q.w);
          }
      }
#pragma unroll 1
      for (int c = 0; c < nch; ++c, ++r) {
        named_sync(1 + (r & 1), nthr);  // the hidden tile is complete
        const unsigned ws = smem + (p.resident ? c : r & (kRing - 1)) * stage_bytes;
        depthwise_project<S, NP, TR, HC, SL>(ws, ke, subb, hid0 + (r & 1) * kHidBytes + dw_base, row_b, lane, p.hi_d, sel, acc);
        if (r + 2 < total) named_arrive(3 + (r & 1), nthr);
      }
      if (p.ks == 1) {
        const UnitPos u = unit_pos(p, unit0 + k * ustep, th_rows);
        const unsigned xs = xs0 + (k & 1) * p.x_bytes;
        store_col<S, 0, NV, NP>(p, u, xs, lane_col(p, S, TR, warp * 16 + g), 0, 0, t, acc);
        store_col<S, 1, NV, NP>(p, u, xs, lane_col(p, S, TR, warp * 16 + g + 8), 0, 0, t, acc);
      } else {
        cluster_wait();  // every CTA of the cluster has started
        push_sums<NV, NP>(p, red, warp, rank, p.ks, lane, acc,
                          [](unsigned at, const float(&f)[4]) { st_cluster_f4(at, f[0], f[1], f[2], f[3]); });
      }
    }
    if (p.ks == 1) return;
  }
  cluster_sync();
  add_sums<S, TR, NV, NP>(p, unit_pos(p, unit0, th_rows), xs0, red, rank, p.ks, warp, nthr >> 5, lane);
}

// ---------------------------------------------------------------- host side
// Shared memory of one CTA under a configuration, and the offsets the kernel uses.
struct Layout {
  int rows, pitch, sub_px, n_list, mt, compact, pw, ncols, ngroups, nw, eg, en;
  unsigned x_pitch, x_bytes, tab_bytes, off_bias, off_tab, off_src, off_x, off_hid, off_red, bytes;
  int stage_bytes, resident, nch;
};

int ke_of(const LaunchRec& r, const BlockCfg& c) { return c.first == kNone ? 0 : (r.C + 15) / 16; }

// cost of a column group's depthwise and projection relative to a group of 16 list pixels; it only divides the list between
// warps that have a column group and warps that have none
double group_cost(const LaunchRec& r, const BlockCfg& c) {
  const int nv = c.s == 1 ? c.tr : c.tr / 2;
  const double d = 4.0 * (c.s == 1 ? 3 : 5) * nv + 4.0 * c.np * nv + 8.0;
  return d / (2.0 * ke_of(r, c) + 3.0);
}

bool layout_of(const LaunchRec& r, const BlockCfg& c, Layout* l) {
  const int th = c.nb * c.tr;
  l->rows = c.s == 1 ? th + 2 : 2 * th + 1;
  l->pitch = c.s == 1 ? c.tw + 2 : 2 * c.tw + 2;
  l->sub_px = l->rows * l->pitch;
  l->compact = c.whole && c.first == kExpWide;
  l->n_list = l->compact ? c.ni * r.H * r.W : c.ni * l->sub_px;
  l->mt = (l->n_list + 15) / 16;
  const bool small = c.wk > 0;
  const int wk = std::max(1, c.wk);
  if (c.ni * l->sub_px > tile_pixels(c.first, small) || l->mt * 16 > tile_pixels(c.first, small) + 2) return false;
  l->pw = c.s == 1 ? c.tw / 2 : c.tw;
  l->ncols = c.ni * c.nb * l->pw;
  l->ngroups = (l->ncols + 15) / 16;
  const int cap = max_warps(c.s, c.np, c.tr, c.ws);
  if (l->ngroups * wk > cap) return false;
  // warps without a column group still help with the first operator
  l->nw = std::min(cap / wk, std::max(l->ngroups, std::min(c.nw_min / wk, c.first != kNone ? (small ? l->mt : (l->mt + 1) / 2) : small ? 1 : 4)));
  {
    const double gc = group_cost(r, c);
    const double share = (l->mt + l->ngroups * gc) / l->nw;  // (of a set)
    int eg = static_cast<int>(share - gc + 0.5);
    if (l->nw == l->ngroups) eg = (l->mt + l->nw - 1) / l->nw;
    l->eg = std::max(0, std::min(eg, (l->mt + l->nw - 1) / l->nw));
    const int rest = l->mt - l->eg * l->ngroups;
    l->en = l->nw > l->ngroups ? std::max(0, (rest + l->nw - l->ngroups - 1) / (l->nw - l->ngroups)) : 0;
    if (c.first == kNone) l->eg = l->en = 0;
  }
  if (c.ws) {
    l->nw = c.nw_min;
    if (l->ngroups >= l->nw || l->nw > cap || (c.first == kExpWide && (l->nw - l->ngroups) % 2)) return false;
    l->eg = 0;
    l->en = (l->mt + l->nw - l->ngroups - 1) / (l->nw - l->ngroups);
  }
  const int ke = ke_of(r, c);
  const int chid = c.first == kNone ? r.C : r.Cmid;
  l->nch = (chid + 16 * c.hc * wk - 1) / (16 * c.hc * wk);
  if (c.ks > l->nch || (c.ws && l->nch / c.ks < 4)) return false;
  const int nchl = (l->nch + c.ks - 1) / c.ks;
  l->stage_bytes = c.hc * wk * (c.ws ? ws_sub_bytes(ke, c.np) : sub_bytes(ke, c.np));
  l->resident = nchl <= kRing || nchl * l->stage_bytes <= c.resident_kb * 1024;
  const int nslot = l->resident ? nchl : kRing;
  const int xw = ke * 2 - (c.first == kExp24 ? 1 : 0);  // 16-byte units of a list pixel; an odd number of them is free of conflicts
  l->x_pitch = c.first == kNone ? 0u : static_cast<unsigned>((xw % 2 ? xw : xw + 1) * 16);
  const int two = c.first != kNone && (c.first != kExpWide || c.ws) ? 2 : 1;
  l->tab_bytes = static_cast<unsigned>(round_up_u64(l->mt * (c.first == kExpWide ? 128 : 64), 128));
  l->x_bytes = static_cast<unsigned>(round_up_u64(l->mt * 16 * l->x_pitch, 128));
  l->off_bias = static_cast<unsigned>(nslot * l->stage_bytes);
  l->off_tab = static_cast<unsigned>(round_up_u64(l->off_bias + c.np * 64, 128));
  l->off_src = l->off_tab + two * l->tab_bytes;
  l->off_x = l->off_src + (c.first != kNone && small ? static_cast<unsigned>(round_up_u64(l->mt * 64, 128)) : 0u);
  l->off_hid = static_cast<unsigned>(round_up_u64(l->off_x + two * l->x_bytes, 128));
  l->off_red = l->off_hid + (c.first == kNone ? kRing : 2) * c.hc * wk * 4 * slice_bytes(c.first, small);
  const int tiles = l->ngroups * (c.s == 1 ? c.tr : c.tr / 2) * c.np;
  l->bytes = l->off_red + (c.ks * wk > 1 ? (tiles + c.ks - 1) / c.ks * c.ks * wk * 2048 : 0);
  l->nw *= wk;
  return l->bytes <= kSmemPerSm - 1024;
}

// (two CTAs that together ask for exactly 227 KB do not share an SM: measured)
int ctas_per_sm(const BlockCfg& c, const Layout& l) {
  return std::max(1, std::min<int>((kSmemPerSm - 1024) / (static_cast<int>(l.bytes) + 1024), max_warps(c.s, c.np, c.tr, c.ws) / l.nw));
}

// Clusters of `ks` CTAs that run at the same time with one CTA per SM: a cluster stays inside one of the chip's GPCs.  Found
// from the jump of a launch's time at one cluster more (8: 15, 4: 33, 2: 73).
int cluster_slots(int ks) { return ks == 8 ? 15 : ks == 4 ? 33 : ks == 2 ? 73 : 148; }

// Estimated time of a launch, for choosing a configuration.  Two bounds, both in SM cycles: the chain of one CTA's units (its
// chunks one after the other, `lat`), and the throughput of an SM's matrix and shared-memory pipes under all its CTAs'
// units (`thr`).  The coefficients are least-squares fits: of units that one CTA computes to 2060 measured launches (ten shapes at
// batch 2 to 256 and image sizes 128 to 513; rms error 8 %), of units that several CTAs or warp sets share to 3000 more (11 %;
// the configuration it picks takes 1.04 times the best one's time in the geometric mean).
// Specialised warps, from 35578 launches of 46 shapes (batch 1 to 256, planes of 10 to 257): within 6 % (rms) near the best; the
// configuration it picks takes 1.03 times the best one's time in the geometric mean, 1.10 at worst.  A chunk takes what the slower of
// the two kinds of warps takes.
double ws_cost_us(const LaunchRec& r, const BlockCfg& c, const Layout& l) {
  const int ke = ke_of(r, c), nv = c.s == 1 ? c.tr : c.tr / 2, nprod = l.nw - l.ngroups, nwg = c.hc == 2 ? nprod / 2 : nprod;
  const int slots = cluster_slots(c.ks) * ctas_per_sm(c, l), act = std::min(c.units, slots);
  const double upc = (c.units + act - 1) / act, per_sm = (act * c.ks + 147) / 148, nchl = (l.nch + c.ks - 1) / c.ks;
  const double rows = 4.0 * (c.s == 1 ? c.tr + 2 : 2 * c.tr + 1);
  const double first = 90.4 + 13.05 * ((l.mt + nwg - 1) / nwg) * ke, second = 29.0 + c.hc * (73.6 * c.np * nv + 7.73 * rows);
  double lat = (nchl + 1) * (44.4 + 18.7 * l.nw + std::max(first, second)) + 134.8 * c.np * nv +
               209.5 * l.n_list * slices(r.C) / (nprod * 32.0) + (c.ks > 1 ? 53.0 : 0.0);
  const double thr = nchl * c.hc * (7.83 * l.mt * ke + 116.9 * l.ngroups) + 60.0 * l.ngroups * c.np * nv;
  const double edge = 1 + 0.45 / c.tw, a = upc * lat * edge, b = upc * per_sm * thr * edge;
  return 3.8 + std::pow(std::pow(a, 1.314) + std::pow(b, 1.314), 1 / 1.314) / 1900.0;
}
double block_cost_us(const LaunchRec& r, const BlockCfg& c, const Layout& l) {
  if (c.ws) return ws_cost_us(r, c, l);
  const int ke = ke_of(r, c), nv = c.s == 1 ? c.tr : c.tr / 2;
  const int occ = ctas_per_sm(c, l), slots = cluster_slots(c.ks) * occ;
  const double upc = (c.units + std::min(c.units, slots) - 1) / std::min(c.units, slots);  // units per CTA
  const double per_sm = (std::min(c.units, slots) * c.ks + 147) / 148;
  const double nchl = (l.nch + c.ks - 1) / c.ks, ew = std::max(l.eg, l.en), thr_n = l.nw * 32.0;
  const double dw = (4.0 * (c.s == 1 ? 3 : 5) * nv + 4.0 * c.np * nv) * c.hc;
  const double wk = std::max(1, c.wk), src = c.ks * wk;
  if (src == 1) {
    const int first = c.first != kNone;
    const double e = c.hc * (4.17 + 76 * ke), d = 82.5 + 3.83 * dw + 977 * c.hc;  // a group of list pixels, of columns
    const double step = 353 + std::max(l.eg * e + d, l.en * e);                   // from one chunk's barrier to the next
    double lat = 815 + (l.nch + first) * step + 520 * c.np * nv;
    lat += first ? 4.47 * l.n_list * slices(r.C) / thr_n : 82.0 * l.nch * c.hc * l.n_list * 4 / thr_n;
    const double rows = 4.0 * (c.s == 1 ? c.tr + 2 : 2 * c.tr + 1);  // fragments of a column group's hidden rows
    double thr = 43.4 + 121 * l.ngroups * c.np * nv;
    thr += l.nch * c.hc * (l.mt * (3.75 * first + 10.74 * ke) + l.ngroups * (0.47 * dw / c.hc + 0.57 * rows + 124.9));
    thr += first ? 0.43 * l.n_list * slices(r.C) : 0.26 * l.n_list * l.nch * c.hc * 4;
    const double a = upc * lat, b = upc * per_sm * thr;
    const double us = 3.02 + std::cbrt(a * a * a + b * b * b) / 1900.0;
    // what the fit leaves on narrow expansions: long rows read and write better (56x56 24 -> 144 -> 24 at batch 256, tiles 28
    // wide 175 us, 14 wide 202), a ring of weights costs its copies; the choice is then within 1.02 of the best, else 1.05
    return c.first == kNone || c.first == kExpWide ? us : us * 0.965 * (1 + 1.0 / c.tw) * (l.resident ? 1 : 1.03);
  }
  const int tiles = l.ngroups * nv * c.np, own = (tiles + c.ks - 1) / c.ks, rounds = (own + l.nw - 1) / l.nw;  // tiles a warp adds up
  double lat = (nchl + 1) * (459.1 + 68.17 * ew * ke * c.hc + 3.99 * dw + 75.98 * l.nw) + 78.48 * c.np * nv + rounds * (1581 + 96.46 * src);
  if (c.first == kNone) lat += (nchl + 1) * 30.31 * l.n_list * 4 * wk / thr_n;
  if (c.ks > 1) lat += 1561;
  double thr = 317.1 + 130.4 * l.ngroups * c.np * nv * wk +
               nchl * wk * (3.538 * l.mt * ke * 2 * c.hc + 4.459 * l.ngroups * dw + 74.9 * l.ngroups * c.hc);
  if (c.first != kNone) thr += 1.235 * l.n_list * slices(r.C);
  const double a = upc * lat, b = upc * per_sm * thr;
  return 2.904 + std::cbrt(a * a * a + b * b * b) / 1965.0;
}

template <void (*kern)(BlockParams)>
int launch_k(const BlockParams& p, int nw, unsigned smem, int grid, cudaStream_t stream) {
  static bool attr_done_dev[kMaxDevices] = {};
  bool& attr_done = attr_done_dev[current_device_slot()];
  if (!attr_done) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemPerSm);
    if (e != cudaSuccess) return static_cast<int>(e);
    attr_done = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(nw * 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = p.ks;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = p.ks > 1 ? 2 : 1;
  return static_cast<int>(cudaLaunchKernelEx(&cfg, kern, p));
}

template <int S, int FIRST, int NP, int TR, int HC>
int launch_t(const BlockCfg& c, const BlockParams& p, int nw, unsigned smem, int grid, cudaStream_t stream) {
  if constexpr (FIRST != kNone) {
    if (c.ws) return launch_k<block_ws_kernel<S, FIRST, NP, TR>>(p, nw, smem, grid, stream);
  }
  if (c.wk > 0) return launch_k<block_mma_kernel<S, FIRST, NP, TR, 1, true>>(p, nw, smem, grid, stream);
  return launch_k<block_mma_kernel<S, FIRST, NP, TR, HC, false>>(p, nw, smem, grid, stream);
}

// rows per warp and sub-blocks per chunk follow from the channel counts (each_config)
template <int S, int FIRST>
int launch_np(const BlockCfg& c, const BlockParams& p, int nw, unsigned smem, int grid, cudaStream_t st) {
  constexpr int HC = FIRST == kExpWide ? 2 : 1;
  if constexpr (S == 2) {
    if (c.np == 2) return launch_t<2, FIRST, 2, 2, HC>(c, p, nw, smem, grid, st);
    if (c.np == 4) return launch_t<2, FIRST, 4, 2, HC>(c, p, nw, smem, grid, st);
    if constexpr (FIRST == kExpWide) {
      if (c.np == 6) return launch_t<2, FIRST, 6, 2, HC>(c, p, nw, smem, grid, st);
      if (c.np == 10) return launch_t<2, FIRST, 10, 2, HC>(c, p, nw, smem, grid, st);
    }
  } else {
    if (c.np == 2) return c.tr == 2 ? launch_t<1, FIRST, 2, 2, HC>(c, p, nw, smem, grid, st) : launch_t<1, FIRST, 2, 1, HC>(c, p, nw, smem, grid, st);
    if (c.np == 4) return c.tr == 2 ? launch_t<1, FIRST, 4, 2, HC>(c, p, nw, smem, grid, st) : launch_t<1, FIRST, 4, 1, HC>(c, p, nw, smem, grid, st);
    if constexpr (FIRST == kExpWide) {
      if (c.np == 6) return launch_t<1, FIRST, 6, 1, HC>(c, p, nw, smem, grid, st);
      if (c.np == 10) return launch_t<1, FIRST, 10, 1, HC>(c, p, nw, smem, grid, st);
    } else {
      if (c.np == 1) return c.tr == 4 ? launch_t<1, FIRST, 1, 4, HC>(c, p, nw, smem, grid, st) : launch_t<1, FIRST, 1, 2, HC>(c, p, nw, smem, grid, st);
    }
  }
  return static_cast<int>(cudaErrorInvalidConfiguration);
}

template <int S>
int launch_first(const BlockCfg& c, const BlockParams& p, int nw, unsigned smem, int grid, cudaStream_t st) {
  switch (c.first) {
    case kNone: return launch_np<S, kNone>(c, p, nw, smem, grid, st);
    case kExp16: return launch_np<S, kExp16>(c, p, nw, smem, grid, st);
    case kExp24: return launch_np<S, kExp24>(c, p, nw, smem, grid, st);
    case kExp32: return launch_np<S, kExp32>(c, p, nw, smem, grid, st);
    default: return launch_np<S, kExpWide>(c, p, nw, smem, grid, st);
  }
}

// Calls f(configuration, layout, spare) for every configuration that runs the block in `r`.  spare: the older kernel beside the
// specialised one (block_mma_choose).
template <class F>
void each_config(const LaunchRec& r, int kind, F&& f) {
  if (r.kh != 3 || r.kw != 3 || r.sh != r.sw || (r.sh != 1 && r.sh != 2) || r.dh != 1 || r.dw != 1) return;
  if (r.pt < 0 || r.pt > 2 || r.pl < 0 || r.pl > 2 || r.W < 2 || r.H < 1) return;
  if (kind == BLOCK_EXPANSION && r.Cmid < 16) return;
  BlockCfg c;
  c.s = r.sh;
  c.first = kind == BLOCK_PAIR ? kNone : r.C <= 16 ? kExp16 : r.C <= 24 ? kExp24 : r.C <= 32 ? kExp32 : kExpWide;
  const int np_raw = (r.Co2 + 15) / 16;
  if (c.first == kExpWide) {
    c.np = np_raw <= 2 ? 2 : np_raw <= 4 ? 4 : np_raw <= 6 ? 6 : np_raw <= 10 ? 10 : 0;
    if (r.C > 160) return;
  } else {
    c.np = np_raw == 1 && c.s == 1 ? 1 : np_raw <= 2 ? 2 : np_raw <= 4 ? 4 : 0;
  }
  if (c.np == 0) return;
  const int64_t in_plane = static_cast<int64_t>(plane_pixels(r.H, r.W)) * 4;
  if (r.B * in_plane * (kind == BLOCK_PAIR ? (r.C + 3) / 4 : 1) >= (1LL << 31)) return;  // offsets inside the input are 32-bit
  if (r.nhwc_in && static_cast<int64_t>(r.H) * r.W * r.C >= (1LL << 31)) return;  // and so is an image of the caller's tensor
  if (static_cast<int64_t>(r.Ho) * r.Wo * std::max(4, r.Co2) >= (1LL << 31)) return;
  c.hc = c.first == kExpWide ? 2 : 1;
  const int wo_even = (r.Wo + 1) / 2 * 2, chid = kind == BLOCK_PAIR ? r.C : r.Cmid;
  const int tr_hi = c.s == 2 ? 2 : c.np == 1 ? 4 : c.np <= 4 ? 2 : 1, tr_lo = c.s == 2 ? 2 : c.np == 1 ? 2 : 1;
  for (c.tr = tr_lo; c.tr <= tr_hi; c.tr *= 2)
    for (int tx = 1; tx <= 32; ++tx) {
      c.tw = ((wo_even + tx - 1) / tx + 1) / 2 * 2;
      c.tiles_x = (r.Wo + c.tw - 1) / c.tw;
      if (c.tiles_x != tx) continue;
      for (c.nb = 1; c.nb <= 28; ++c.nb) {
        const int th = c.nb * c.tr;
        if (th - c.tr >= r.Ho || (c.s * (th - 1) + 3) * (c.s * (c.tw - 1) + 3) > tile_pixels(c.first, false)) break;
        c.tiles_y = (r.Ho + th - 1) / th;
        c.whole = c.tiles_x == 1 && c.tiles_y == 1;
        for (c.ni = 1; c.ni <= (c.whole ? 8 : 1) && c.ni <= r.B; ++c.ni) {
          const long long units = c.whole ? (r.B + c.ni - 1) / c.ni : static_cast<long long>(r.B) * c.tiles_x * c.tiles_y;
          if (units > (1 << 28) || static_cast<uint64_t>(units) * c.tiles_x * c.tiles_y >= (1ull << 32)) continue;
          c.units = static_cast<int>(units);
          // warp sets: small tiles, while there are no more of them than SMs
          static const int kSets[] = {0, 1, 2, 3, 4, 6, 8, 12, 16};
          const int hid = c.ni * (c.s * (th - 1) + 3) * (c.s * (c.tw - 1) + 3);
          const bool sets = units <= 148 && hid <= tile_pixels(c.first, true);
          for (int wi = 0; wi < (sets ? 9 : 1); ++wi) {
            c.wk = kSets[wi];
            if ((c.wk - 1) * 16 >= chid) break;  // a set without channels
            c.hc = c.first == kExpWide && c.wk == 0 ? 2 : 1;
            // specialised warps: as many as fit one, two or three CTAs of an SM, or one less (a wide expansion's warps work in
            // pairs); wide ones, of which there are few tiles, any number.  Narrow ones stay in one CTA: their clusters are small
            // tiles for the older kernel.  Not with a bias of the expansion that has no parts (bias_split.h).
            // More than four chunks of weights come through the ring: resident they take 0.96 to 0.99 times the time near the best
            // choices where as many CTAs fit an SM, 1.1 to 1.3 times where one fewer does, which the estimate does not tell apart.
            int specialised = 0;  // cluster sizes with such a layout
            if (c.wk == 0 && c.first != kNone && r.split_bias && (c.ni == 1 || c.first == kExpWide)) {
              const int cap = max_warps(c.s, c.np, c.tr, true);
              c.ws = 1;
              for (c.ks = 1; c.ks <= (c.first == kExpWide ? 8 : 1); c.ks *= 2) {
                if (c.ks > 1 && units * c.ks > 148) break;
                for (c.nw_min = cap; c.nw_min >= 2; --c.nw_min) {
                  if (c.first != kExpWide && cap / (cap / c.nw_min) != c.nw_min && cap / (cap / (c.nw_min + 1)) != c.nw_min + 1) continue;
                  c.resident_kb = 0;
                  Layout l;
                  if (!layout_of(r, c, &l)) continue;
                  specialised |= c.ks;
                  if (c.ks == 1 || units <= cluster_slots(c.ks) * ctas_per_sm(c, l)) f(c, l, false);
                }
              }
              c.ws = 0;
            }
            const bool spare = specialised && c.first == kExpWide;
            for (c.ks = 1; c.ks <= 8; c.ks *= 2) {
              if (specialised & c.ks) continue;
              if (c.ks > 1 && units * c.ks > 148 * 2) break;  // a split pays only while SMs would be idle ...
              for (c.nw_min = 8; c.nw_min <= max_warps(c.s, c.np, c.tr); c.nw_min += max_warps(c.s, c.np, c.tr) == 12 ? 4 : 8) {
                for (int rk = 0; rk < 2; ++rk) {
                  c.resident_kb = rk ? 48 : 0;
                  Layout l;
                  if (!layout_of(r, c, &l) || (c.nw_min > 8 && l.nw <= 8)) break;  // nw_min 8 has given the same layout
                  if (rk && !l.resident) break;
                  if (spare && !l.resident) continue;
                  // ... in one wave
                  if (c.ks == 1 || units <= cluster_slots(c.ks) * ctas_per_sm(c, l)) f(c, l, spare);
                  if (l.resident) break;
                }
              }
            }
          }
        }
      }
    }
}

uint16_t half_bits(float v) { return f32_to_f16_rne(v); }

}  // namespace

// Chooses tile, image and cluster split for the block in `r` (C -> Cmid -> Co2, or C -> Co2 for BLOCK_PAIR; stride r.sh, output
// Ho x Wo).  False if no configuration runs it; `us` receives the estimate the choice was made by.
bool block_mma_choose(const LaunchRec& r, int kind, BlockCfg* best, double* us) {
  double best_cost = 0.0, spare_cost = 0.0;
  BlockCfg spare_cfg;
  bool found = false, spare_found = false;
  if (kind == BLOCK_STEM) return stem_block_choose(r, best, us);
  each_config(r, kind, [&](const BlockCfg& c, const Layout& l, bool spare) {
    const double cost = block_cost_us(r, c, l);
    bool& any = spare ? spare_found : found;
    double& least = spare ? spare_cost : best_cost;
    if (any && cost >= least) return;
    any = true;
    least = cost;
    (spare ? spare_cfg : *best) = c;
  });
  // Wide expansions on tiles for which there are specialised warps, at the cluster sizes for which there are none (fewer than four
  // chunks a CTA): the older kernel, where its weights stay in shared memory, stands in for warp sets, not for specialised warps.
  // us, it and the choice without it: 6x6 80-480-80 batch 54 10.9, 13.3; 10x10 64-384-64 batch 28 11.0, 12.1; 12x12 64-384-96 batch
  // 15 10.3, 11.3; the other way 5x5 64-384-64 batch 108 12.2, 11.7; 10x10 64-384-64 batch 17 11.6, 10.2.  Of 4000 random blocks
  // it changes the choice for 65: 0.93 times the time (geometric mean), six slower.  Set against specialised warps too it would
  // take their place where they are faster (6x6 160-960-160 batch 55 30.6, 22.1), and with a ring of weights it is slower than sets.
  if (found && spare_found && !best->ws && spare_cost < best_cost) {
    *best = spare_cfg;
    best_cost = spare_cost;
  }
  if (us) *us = best_cost;
  return found;
}

// Packs all weights of the block in sub-blocks of 16 hidden channels (layout: sub_bytes), biases in fp32.
// we: [chid][cin], for the stem [chid][3][3][3], null for a pair; wd [9][chid], wp [cout][chid].
void block_mma_pack(const float* we, const float* be, const float* wd, const float* bd, const float* wp, const float* bp, int cin,
                    int chid, int cout, const BlockCfg& c, std::vector<uint8_t>* blob, LaunchRec* r) {
  if (c.stem) return stem_block_pack(we, be, wd, bd, wp, bp, chid, cout, c, blob, r);
  const int ke = c.first == kNone ? 0 : (cin + 15) / 16, np = c.np;
  const int per = c.hc * std::max(1, c.wk), nsub = (chid + 16 * per - 1) / (16 * per) * per;
  const size_t sb = c.ws ? ws_sub_bytes(ke, np) : sub_bytes(ke, np);
  const uint64_t woff = round_up_u64(blob->size(), 256);
  const uint64_t boff = round_up_u64(woff + nsub * sb, 256);
  blob->resize(boff + static_cast<size_t>(np) * 16 * sizeof(float), 0);
  for (int sub = 0; sub < nsub; ++sub) {
    uint8_t* base = blob->data() + woff + sub * sb;
    uint16_t* e = reinterpret_cast<uint16_t*>(base);
    for (int kk = 0; kk < ke; ++kk)
      for (int lane = 0; lane < 32; ++lane)
        for (int w = 0; w < 8; ++w) {  // halves of {frag 0: b0, b1; frag 1: b0, b1}
          const int f = w >> 2, hi8 = (w >> 1) & 1, lo = w & 1;
          const int n = lane >> 2, t = lane & 3;
          const int k = kk * 16 + hi8 * 8 + 2 * t + lo, h = channel_of(sub, f, n);
          if (h < chid && k < cin) e[(kk * 32 + lane) * 8 + w] = half_bits(we[static_cast<size_t>(h) * cin + k]);
        }
    if (c.ws) {
      uint16_t* words = reinterpret_cast<uint16_t*>(base + sub_bytes(ke, np));
      for (int f = 0; f < 2; ++f)
        for (int n = 0; n < 8; ++n) {
          const int h = channel_of(sub, f, n);
          uint16_t part[4] = {};
          if (h < chid) bias_parts(be[h], part);
          std::copy(part, part + 4, words + (f * 8 + n) * 4);
          // up to 24 channels: the second step's last four values are free
          if (c.first == kExp24)
            for (int i = 0; i < 4; ++i) e[(32 + n * 4 + i / 2) * 8 + f * 4 + 2 + i % 2] = part[i];
        }
    }
    float* ebias = reinterpret_cast<float*>(base + ke * 512);
    uint16_t* tabl = reinterpret_cast<uint16_t*>(base + ke * 512 + kBiasBytes);
    float* dbias = reinterpret_cast<float*>(base + ke * 512 + kBiasBytes + kTableBytes);
    for (int ch = 0; ch < 16; ++ch) {
      const int h = sub * 16 + ch;
      if (h >= chid) break;
      if (c.first != kNone) ebias[ch] = be[h];
      for (int i = 0; i < 4; ++i) dbias[ch * 4 + i] = bd[h];
    }
    for (int sl = 0; sl < 4; ++sl)
      for (int jh = 0; jh < 2; ++jh)
        for (int g = 0; g < 8; ++g) {
          const int h = sub * 16 + sl * 4 + (g >> 1);
          if (h >= chid) continue;
          uint16_t* word = tabl + ((sl * 16 + jh * 8 + g) * 4) * 2;
          for (int ky = 0; ky < 3; ++ky)
            for (int b = 0; b < 2; ++b) {
              // stride 1: input pixel j of the window row feeds output pixel q of the pair through tap j - q;
              // stride 2: one output column, tap j
              const int j = b * 2 + jh, q = c.s == 1 ? (g & 1) : 0, dx = j - q;
              if (dx >= 0 && dx <= 2) word[ky * 2 + b] = half_bits(wd[static_cast<size_t>(ky * 3 + dx) * chid + h]);
            }
        }
    uint16_t* q = reinterpret_cast<uint16_t*>(base + ke * 512 + kSubFixed);
    for (int j = 0; j < np; ++j)
      for (int lane = 0; lane < 32; ++lane)
        for (int w = 0; w < 8; ++w) {
          const int f = w >> 2, hi8 = (w >> 1) & 1, lo = w & 1;
          const int n = lane >> 2, t = lane & 3;
          const int h = sub * 16 + hi8 * 8 + lo * 4 + t, co = channel_of(j, f, n);
          if (h < chid && co < cout) q[(j * 32 + lane) * 8 + w] = half_bits(wp[static_cast<size_t>(co) * chid + h]);
        }
  }
  float* b = reinterpret_cast<float*>(blob->data() + boff);
  for (int i = 0; i < cout; ++i) b[i] = bp[i];
  r->wts = Loc{W_WEIGHTS, 0, woff};
  r->bias = Loc{W_WEIGHTS, 0, boff};
  r->wts_bytes = nsub * sb;
}

namespace {
// Everything but the pointers.
BlockParams params_of(const LaunchRec& r, const BlockCfg& c, const Layout& l) {
  BlockParams p{};
  p.B = r.B;
  p.H = r.H;
  p.W = r.W;
  p.Ho = r.Ho;
  p.Wo = r.Wo;
  const int P = plane_pixels(r.H, r.W), Po = plane_pixels(r.Ho, r.Wo);
  p.in_px = r.nhwc_in ? r.C : 4;
  p.in_img = r.nhwc_in ? r.H * r.W * r.C : P * 4;
  p.in_sl = r.nhwc_in ? 4 : static_cast<long long>(r.B) * P * 4;
  p.o_px = r.nhwc_out ? r.Co2 : 4;
  p.o_img = r.nhwc_out ? static_cast<long long>(r.Ho) * r.Wo * r.Co2 : Po * 4;
  p.o_sl = r.nhwc_out ? 4 : static_cast<long long>(r.B) * Po * 4;
  p.res_img = Po * 4;
  p.res_sl = static_cast<long long>(r.B) * Po * 4;
  p.sin = slices(r.C);
  p.sout = slices(r.Co2);
  p.ke = ke_of(r, c);
  p.pad_t = r.pt;
  p.pad_l = r.pl;
  p.tw = c.tw;
  p.nb = c.nb;
  p.ni = c.ni;
  p.tiles_x = c.tiles_x;
  p.tiles_y = c.tiles_y;
  p.units = c.units;
  p.rows = l.rows;
  p.pitch = l.pitch;
  p.sub_px = l.sub_px;
  p.n_list = l.n_list;
  p.mt = l.mt;
  p.whole = c.whole;
  p.compact = l.compact;
  p.pw = l.pw;
  p.ncols = l.ncols;
  p.ngroups = l.ngroups;
  p.eg = l.eg;
  p.en = l.en;
  p.nch = l.nch;
  p.ks = c.ks;
  p.wk = std::max(1, c.wk);
  p.nwq = l.nw / p.wk;
  p.resident = l.resident;
  p.x_pitch = l.x_pitch;
  p.off_bias = l.off_bias;
  p.x_bytes = l.x_bytes;
  p.tab_bytes = l.tab_bytes;
  p.off_tab = l.off_tab;
  p.off_src = l.off_src;
  p.off_x = l.off_x;
  p.off_hid = l.off_hid;
  p.off_red = l.off_red;
  p.mul_pitch = magic(l.pitch);
  p.mul_w = magic(r.W);
  p.mul_hw = magic(static_cast<uint64_t>(r.H) * r.W);
  p.mul_per = magic(static_cast<uint64_t>(c.tiles_x) * c.tiles_y);
  p.mul_tx = magic(c.tiles_x);
  p.hi_e = r.ep.act_pre == GI_ACT_RELU6 ? 0x46004600u : kMaxFinite;  // the banded operand multiplies neighbours by zero
  const int dact = c.first != kNone ? r.ep_mid.act_pre : r.ep.act_pre;
  p.hi_d = dact == GI_ACT_RELU6 ? 0x46004600u : 0x7c007c00u;
  p.act_pre = r.ep2.act_pre;
  p.act_post = r.ep2.act_post;
  p.has_res = r.ep2.has_res;
  p.wide = !r.nhwc_out && r.Wo % 2 == 0;
  p.pad_px = !r.nhwc_out && (r.Ho * r.Wo) % 2;
  return p;
}
}  // namespace

int launch_block_mma(const LaunchRec& r, const Ptrs& ptr, void* stream) {
  const BlockCfg& c = r.block;
  if (c.stem) return launch_stem_block(r, ptr, stream);
  Layout l;
  if (r.dh != 1 || r.dw != 1 || !layout_of(r, c, &l)) return static_cast<int>(cudaErrorInvalidConfiguration);
  BlockParams p = params_of(r, c, l);
  p.in = static_cast<const __half*>(ptr.in0);
  p.res = static_cast<const __half*>(ptr.res);
  p.out = static_cast<__half*>(ptr.out);
  p.wts = static_cast<const unsigned char*>(ptr.wts);
  p.bias = static_cast<const float*>(ptr.bias);
  p.res_x = p.has_res && ptr.res == ptr.in0 && !r.nhwc_in && c.s == 1 && c.first != kNone && c.first != kExpWide;
  const long long slots = c.ks > 1 ? c.units : static_cast<long long>(device_sm_count()) * ctas_per_sm(c, l);
  const int grid = static_cast<int>(std::min<long long>(c.units, std::max<long long>(1, slots))) * c.ks;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return c.s == 1 ? launch_first<1>(c, p, l.nw, l.bytes, grid, st) : launch_first<2>(c, p, l.nw, l.bytes, grid, st);
}

}  // namespace gi
