// cnn.cu -- the learned initialiser of include/pty_cnn.h: bf16 implicit-GEMM convolutions on the
// tensor cores (tcgen05 with TMEM accumulators, gemm_tc.cuh: forward, input gradient, weight
// gradient), the two-channel output layer on the CUDA cores, the loss, Adam, training targets and
// stitching.
//
// Layout: activations channels-last [B][H][W][C] in bf16, so one 16-byte load gathers 8 channels of
// one tap.  GEMM views (rows x cols, reduction K):
//   forward    z[pixel][oc]   = sum_k col[pixel][k] W[oc][k],        k = (ky, kx, ic)
//   dgrad      du[pixel][ic]  = sum_k' dz[pixel'(k')][oc] Wt[ic][k'], k' = (ky, kx, oc), pixels of the
//                                (upsampled) input grid; pixel' is the output that reads it by tap
//   wgrad      dW[oc][k]      = sum_pixels dz[pixel][oc] col[pixel][k]: dz and the im2col matrix are
//                                first transposed to pixel-contiguous rows (chunks of at most 2^18
//                                pixels), then one plain GEMM per chunk, split over pixels with
//                                float atomics
// All of them run through k_gemm_ws (gemm_ws.cuh) with weights, dz and im2col transposes kept as tile images.
// Layer 6 (upsampling x4, 2 output channels) would waste 126 of 128 GEMM columns, so it runs on the
// CUDA cores: nearest upsampling makes every output pixel read, for each tap, one low-resolution
// pixel, so the per-tap channel sums P[p][tap][o] = sum_c W[o][tap][c] a5[p][c] are formed once per
// low-resolution pixel and each output adds nine of them; the backward pass runs the same
// structure in reverse.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "gemm_ws.cuh"
#include "pty_cnn.h"
#include "pty_internal.h"

namespace pty {
namespace cnn {

using bf16 = __nv_bfloat16;

struct LayerDef {
  int ic, oc, stride, up;
};
constexpr int kLayers = 6;
constexpr LayerDef kNet[kLayers] = {{1, 48, 2, 1}, {48, 96, 2, 1}, {96, 192, 2, 1},
                                    {192, 384, 2, 1}, {384, 256, 1, 2}, {256, 2, 1, 4}};
constexpr int kOut = 2;     // output channels
constexpr int kTaps6 = 18;  // layer 6: 9 taps x 2 output channels
constexpr int kC6 = 256;    // layer 6 input channels
constexpr int kPixChunk = 1 << 18;  // output pixels per weight-gradient chunk

__host__ __device__ constexpr int round64(int x) { return (x + 63) / 64 * 64; }

// ---------------------------------------------------------------------------------------------
// Plan: per-layer sizes and workspace offsets for patterns of S x S and batches of B
// ---------------------------------------------------------------------------------------------
struct Plan {
  int S, B;
  int hin[kLayers], hout[kLayers], hu[kLayers];  // input, output and upsampled-input sizes
  size_t woff[kLayers], boff[kLayers];           // offsets of weights / biases in the parameters
  int kp[kLayers], ktp[kLayers];                 // padded K of the forward and dgrad GEMMs
  // workspace pieces (byte offsets)
  size_t status, wp[kLayers], wt[kLayers], w6, act[kLayers], dz[kLayers + 1], p6, dp6, du5, lpart, colt, dzt,
      total;
  int pchunk[kLayers];  // pixels per weight-gradient chunk (multiple of 64)
  size_t colt_elems;    // elements of colt
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static bool make_plan(int S, int B, Plan* pl) {
  if (S < 16 || S > 512 || S % 16 != 0 || B < 0 || B > 1024) return false;
  Plan p;
  memset(&p, 0, sizeof(p));
  p.S = S;
  p.B = B;
  int h = S;
  size_t o = 0;
  for (int l = 0; l < kLayers; ++l) {
    p.hin[l] = h;
    p.hu[l] = h * kNet[l].up;
    p.hout[l] = (p.hu[l] + kNet[l].stride - 1) / kNet[l].stride;
    h = p.hout[l];
    p.woff[l] = o;
    o += (size_t)9 * kNet[l].ic * kNet[l].oc;
    p.boff[l] = o;
    o += kNet[l].oc;
    p.kp[l] = round64(9 * kNet[l].ic);
    p.ktp[l] = round64(9 * kNet[l].oc);
  }
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t r = off;
    off += align256(bytes);
    return r;
  };
  p.status = take(sizeof(int) * 64);
  for (int l = 0; l < 5; ++l) {
    p.wp[l] = take(sizeof(bf16) * kNet[l].oc * p.kp[l]);
    if (l > 0) p.wt[l] = take(sizeof(bf16) * kNet[l].ic * p.ktp[l]);
  }
  p.w6 = take(sizeof(float) * kTaps6 * kC6);
  for (int l = 0; l < 5; ++l) p.act[l] = take(sizeof(bf16) * (size_t)B * p.hout[l] * p.hout[l] * kNet[l].oc);
  for (int l = 0; l < 5; ++l) p.dz[l] = take(sizeof(bf16) * (size_t)B * p.hout[l] * p.hout[l] * kNet[l].oc);
  p.dz[5] = take(sizeof(bf16) * (size_t)B * p.hout[5] * p.hout[5] * kOut);
  const size_t lowres = (size_t)B * p.hout[4] * p.hout[4];
  p.p6 = take(sizeof(float) * lowres * kTaps6);
  p.dp6 = take(sizeof(float) * lowres * kTaps6);
  p.du5 = take(sizeof(float) * (size_t)B * p.hu[4] * p.hu[4] * kNet[4].ic);
  p.lpart = take(sizeof(double) * 1024);
  // weight gradients run over chunks of at most kPixChunk output pixels, with the im2col matrix and
  // dL/dz transposed to pixel-contiguous rows
  size_t colt = 0, dzt = 0;
  for (int l = 0; l < 5; ++l) {
    const size_t pix = (size_t)B * p.hout[l] * p.hout[l];
    p.pchunk[l] = (int)((pix < (size_t)kPixChunk ? (pix + 63) / 64 * 64 : (size_t)kPixChunk));
    if (p.pchunk[l] < 64) p.pchunk[l] = 64;
    colt = colt > (size_t)9 * kNet[l].ic * p.pchunk[l] ? colt : (size_t)9 * kNet[l].ic * p.pchunk[l];
    dzt = dzt > (size_t)kNet[l].oc * p.pchunk[l] ? dzt : (size_t)kNet[l].oc * p.pchunk[l];
  }
  p.colt_elems = colt;
  p.colt = take(sizeof(bf16) * colt);
  p.dzt = take(sizeof(bf16) * dzt);
  p.total = off;
  *pl = p;
  return true;
}

size_t param_count() {
  size_t n = 0;
  for (int l = 0; l < kLayers; ++l) n += (size_t)9 * kNet[l].ic * kNet[l].oc + kNet[l].oc;
  return n;
}


// ---------------------------------------------------------------------------------------------
// Weight packing: FP32 parameters -> bf16 GEMM operands (zero-padded K) and layer 6's table
// ---------------------------------------------------------------------------------------------
struct PackArgs {
  const float* params;
  bf16* wp[5];  // tile image [OC][kp]
  bf16* wt[5];  // tile image [IC][ktp] (layers 2..5)
  float* w6;    // [18][256]: row tap * 2 + o, bf16-rounded
  size_t woff[kLayers];
  int kp[kLayers], ktp[kLayers], ic[kLayers], oc[kLayers];
};

// (row, k) of element e of a tile image of `rows` rows
__device__ __forceinline__ void image_element(int e, int rows, int* row, int* k) {
  const int kb = e / (rows * 64), r = e - kb * rows * 64;
  *row = (r >> 9) * 8 + ((r >> 3) & 7);
  *k = kb * 64 + ((r >> 6) & 7) * 8 + (r & 7);
}

__global__ void k_pack(PackArgs a) {
  // segments: wp of layers 0..4, wt of layers 1..4, w6
  size_t seg[10];
  int n = 0;
  for (int l = 0; l < 5; ++l) seg[n++] = (size_t)a.oc[l] * a.kp[l];
  for (int l = 1; l < 5; ++l) seg[n++] = (size_t)a.ic[l] * a.ktp[l];
  seg[n++] = (size_t)kTaps6 * kC6;
  size_t total = 0;
  for (int q = 0; q < n; ++q) total += seg[q];
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    size_t e = i;
    int q = 0;
    while (e >= seg[q]) e -= seg[q++];
    if (q < 5) {  // forward operand of layer q: W[oc][k], k = (ky, kx, ic)
      const int l = q, K9 = 9 * a.ic[l];
      int oc, k;
      image_element((int)e, a.oc[l], &oc, &k);
      a.wp[l][e] = __float2bfloat16_rn(k < K9 ? a.params[a.woff[l] + (size_t)oc * K9 + k] : 0.f);
    } else if (q < 9) {  // dgrad operand of layer l: Wt[ic][k'] = W[oc][tap][ic], k' = tap * OC + oc
      const int l = q - 4, IC = a.ic[l], OC = a.oc[l];
      int ic, kk;
      image_element((int)e, a.ic[l], &ic, &kk);
      float w = 0.f;
      if (kk < 9 * OC) {
        const int tap = kk / OC, oc = kk % OC;
        w = a.params[a.woff[l] + ((size_t)oc * 9 + tap) * IC + ic];
      }
      a.wt[l][e] = __float2bfloat16_rn(w);
    } else {  // layer 6: w6[tap * 2 + o][c] = W[o][tap][c]
      const int j = (int)(e / kC6), c = (int)(e % kC6);
      const int tap = j / kOut, o = j % kOut;
      a.w6[e] = __bfloat162float(__float2bfloat16_rn(a.params[a.woff[5] + ((size_t)o * 9 + tap) * kC6 + c]));
    }
  }
}

// ---------------------------------------------------------------------------------------------
// GEMM operand loaders (8 consecutive reduction elements per call, zeros outside)
// ---------------------------------------------------------------------------------------------
union Pack8 {
  uint4 u;
  bf16 h[8];
};

__device__ __forceinline__ bf16 input_value(const float* I, float s_in, int S, int b, int y, int x) {
  return __float2bfloat16_rn(s_in * log1pf(__ldg(I + ((size_t)b * S + y) * S + x)));
}

// Layer 1's rows: x16[pixel][16] = the nine taps of bf16(s_in log(1 + I)) (zeros outside) and seven zeros, written once
// so that the GEMM gathers 32 contiguous bytes a row.  Rows p0 .. p0 + n - 1; one thread per row.
__global__ void __launch_bounds__(256) k_input_rows(const float* __restrict__ I, float s_in, bf16* __restrict__ x16, int S,
                                                    int hout, size_t p0, size_t n) {
  const size_t i = blockIdx.x * (size_t)256 + threadIdx.x;
  if (i >= n) return;
  const size_t m = p0 + i, hw = (size_t)hout * hout;
  const int b = (int)(m / hw), rem = (int)(m % hw), oy = rem / hout, ox = rem % hout;
  Pack8 r[2];
  r[0].u = r[1].u = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int tap = 0; tap < 9; ++tap) {
    const int y = 2 * oy + tap / 3 - 1, x = 2 * ox + tap % 3 - 1;
    if (y >= 0 && y < S && x >= 0 && x < S) r[tap / 8].h[tap % 8] = input_value(I, s_in, S, b, y, x);
  }
  uint4* o = reinterpret_cast<uint4*>(x16 + 16 * i);
  o[0] = r[0].u;
  o[1] = r[1].u;
}
struct InputRows {
  static constexpr bool kGather = true;
  const bf16* x16;
  int rows;
  struct K {
    int tap, off;
  };
  __device__ __forceinline__ const bf16* any() const { return x16; }
  __device__ __forceinline__ int tile_class(int) const { return 0; }
  __device__ __forceinline__ int kb_next(int, int kb) const { return kb; }
  __device__ __forceinline__ GatherRow row(int m) const { return GatherRow{x16 + (size_t)m * 16, m < rows ? 1u : 0u, 0u}; }
  __device__ __forceinline__ K kpos(int k, int) const { return K{0, k}; }
  __device__ __forceinline__ int offset(const GatherRow&, const K& k) const { return k.off; }
};

// Forward of layers 2..5: rows = output pixels, 8 channels of one tap of the (upsampled) input per chunk.  A tap's
// distance from tap 0 is the same for every row, or with upsampling depends on the parities of the row's pixel
// (bits 16, 17 of its mask).
template <int UP>
struct Im2col {
  static constexpr bool kGather = true;
  const bf16* a;  // [B][hin][hin][ic]
  int B, hin, hu, hout, ic, stride;
  struct K {
    int tap, y[UP], x[UP];  // elements, by the parity of the pixel; x holds the channel too
  };
  __device__ __forceinline__ const bf16* any() const { return a; }
  __device__ __forceinline__ int tile_class(int) const { return 0; }
  __device__ __forceinline__ int kb_next(int, int kb) const { return kb; }
  __device__ __forceinline__ GatherRow row(int m) const {
    if (m >= B * hout * hout) return GatherRow{a, 0u, 0u};
    const int b = m / (hout * hout), rem = m - b * hout * hout, oy = rem / hout;
    const int y0 = stride * oy - 1, x0 = stride * (rem - oy * hout) - 1;
    unsigned mask = 0;
#pragma unroll
    for (int t = 0; t < 9; ++t)
      if ((unsigned)(y0 + t / 3) < (unsigned)hu && (unsigned)(x0 + t % 3) < (unsigned)hu) mask |= 1u << t;
    if (UP == 2) mask |= (unsigned)(y0 & 1) << 16 | (unsigned)(x0 & 1) << 17;
    const long long pix = (long long)(b * hin + (y0 >> (UP - 1))) * hin + (x0 >> (UP - 1));
    return GatherRow{a + pix * ic, mask, 0u};
  }
  __device__ __forceinline__ K kpos(int k, int) const {
    K r;
    r.tap = k / ic;
    const int ky = r.tap / 3, kx = r.tap - 3 * ky;
#pragma unroll
    for (int p = 0; p < UP; ++p) {
      r.y[p] = ((p + ky) >> (UP - 1)) * hin * ic;
      r.x[p] = ((p + kx) >> (UP - 1)) * ic + k - r.tap * ic;
    }
    return r;
  }
  __device__ __forceinline__ int offset(const GatherRow& r, const K& k) const {
    if constexpr (UP == 1) return k.y[0] + k.x[0];
    else return ((r.m >> 16 & 1) ? k.y[1] : k.y[0]) + ((r.m >> 17 & 1) ? k.x[1] : k.x[0]);
  }
};

// Rows of an input gradient: the pixels of the (upsampled) input grid.  With stride 2 a pixel (uy, ux) is reached
// only by the taps with ky = uy + 1 and kx = ux + 1 (mod 2), one to four of nine, so the pixels are taken in four
// classes by their parities, whole row tiles each, and a tile skips the K blocks of the other taps: those
// would add exact zeros (about 2.6 of 9 of the blocks are left).
struct GradRows {
  int B, hu, stride, ctiles;  // ctiles: row tiles of a class
  __host__ __device__ GradRows(int B_, int hu_, int stride_) : B(B_), hu(hu_), stride(stride_) {
    const int h = hu / stride;
    ctiles = (B * h * h + 127) / 128;
  }
  int row_tiles() const { return ctiles * stride * stride; }
  __device__ __forceinline__ int tile_class(int tile) const { return stride == 2 ? tile / ctiles : 0; }
  // class, sample and place (in units of the stride) of row m; false past the end of its class
  __device__ __forceinline__ bool pixel(int m, int* cls, int* b, int* y, int* x) const {
    *cls = tile_class(m >> 7);
    const int i = m - *cls * ctiles * 128, h = hu / stride;
    if (i >= B * h * h) return false;
    *b = i / (h * h);
    const int rem = i - *b * h * h;
    *y = rem / h;
    *x = rem - *y * h;
    return true;
  }
};
// Input gradient of layers 2..5: k' = (tap, oc); the output pixel that reads (uy, ux) through tap (ky, kx) is
// ((uy + 1 - ky) / s, (ux + 1 - kx) / s).
struct DgradGather {
  static constexpr bool kGather = true;
  const bf16* dz;  // [B][hout][hout][oc]
  GradRows g;
  int hout, oc;
  unsigned long long blocks[4];  // K blocks with a tap of the class (bit kb; at most 54 blocks)
  DgradGather(const bf16* dz_, const GradRows& g_, int hout_, int oc_, int kb_all) : dz(dz_), g(g_), hout(hout_), oc(oc_) {
    for (int c = 0; c < 4; ++c) {
      blocks[c] = 0;
      for (int kb = 0; kb < kb_all; ++kb)
        for (int t = kb * kWsBlock / oc; t <= (kb * kWsBlock + kWsBlock - 1) / oc && t < 9; ++t)
          if (g.stride == 1 || (!(((c >> 1) + 1 - t / 3) & 1) && !(((c & 1) + 1 - t % 3) & 1))) blocks[c] |= 1ull << kb;
    }
  }
  struct K {
    int tap, offset;
  };
  __device__ __forceinline__ int tile_class(int tile) const { return g.tile_class(tile); }
  __device__ __forceinline__ const bf16* any() const { return dz; }
  __device__ __forceinline__ int kb_next(int c, int kb) const {
    if (g.stride == 1) return kb;
    const unsigned long long left = (c == 0 ? blocks[0] : c == 1 ? blocks[1] : c == 2 ? blocks[2] : blocks[3]) >> kb;  // kb <= 54
    return left ? kb + __ffsll((long long)left) - 1 : 64;
  }
  __device__ __forceinline__ GatherRow row(int m) const {
    int cls, b, y, x;
    if (!g.pixel(m, &cls, &b, &y, &x)) return GatherRow{dz, 0u, 0u};
    unsigned mask = 0;
    if (g.stride == 1) {  // tap (ky, kx) reads (y + 1 - ky, x + 1 - kx)
#pragma unroll
      for (int t = 0; t < 9; ++t)
        if ((unsigned)(y + 1 - t / 3) < (unsigned)hout && (unsigned)(x + 1 - t % 3) < (unsigned)hout) mask |= 1u << t;
    } else {  // the taps of the class: (y + (py + 1 - ky) / 2, ...)
      const int py = cls >> 1, px = cls & 1;
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        const int dy = py + 1 - t / 3, dx = px + 1 - t % 3;
        if (!((dy | dx) & 1) && (unsigned)(y + (dy >> 1)) < (unsigned)hout && (unsigned)(x + (dx >> 1)) < (unsigned)hout)
          mask |= 1u << t;
      }
    }
    return GatherRow{dz + ((size_t)(b * hout + y) * hout + x) * oc, mask, 0u};
  }
  // a tap's offset is the same for every row of a class
  __device__ __forceinline__ K kpos(int k, int cls) const {
    const int tap = k / oc, ky = tap / 3, kx = tap - 3 * ky, o = k - tap * oc;
    if (g.stride == 1) return K{tap, ((1 - ky) * hout + 1 - kx) * oc + o};
    return K{tap, ((((cls >> 1) + 1 - ky) >> 1) * hout + (((cls & 1) + 1 - kx) >> 1)) * oc + o};
  }
  __device__ __forceinline__ int offset(const GatherRow&, const K& k) const { return k.offset; }
};
struct ImageLoad {
  static constexpr bool kGather = false;
  ImageOperand op;
};

// ---------------------------------------------------------------------------------------------
// GEMM epilogues
// ---------------------------------------------------------------------------------------------
// epi(row, col, v): eight consecutive columns
struct FwdEpi {  // a = bf16(relu(z + bias))
  bf16* out;
  const float* bias;
  int rows, oc;
  using Row = int;
  __device__ __forceinline__ Row prep(int m) const { return m; }
  __device__ __forceinline__ void operator()(int row, int col, const float* v) const {
    if (row >= rows) return;
    Pack8 r;
#pragma unroll
    for (int e = 0; e < 8; ++e) r.h[e] = __float2bfloat16_rn(fmaxf(v[e] + __ldg(bias + col + e), 0.f));
    *reinterpret_cast<uint4*>(out + (size_t)row * oc + col) = r.u;
  }
};
struct DgradEpi {  // dz of the layer below = bf16(du * (a > 0)) (no upsampling between)
  bf16* dz;
  const bf16* a;
  GradRows g;
  int ic;
  using Row = long long;
  __device__ __forceinline__ Row prep(int m) const {  // its pixel, or -1
    int cls, b, y, x;
    if (!g.pixel(m, &cls, &b, &y, &x)) return -1;
    return ((long long)b * g.hu + g.stride * y + (g.stride == 2 ? cls >> 1 : 0)) * g.hu + g.stride * x +
           (g.stride == 2 ? cls & 1 : 0);
  }
  __device__ __forceinline__ void operator()(Row row, int col, const float* v) const {
    if (row < 0) return;
    const size_t e = (size_t)row * ic + col;
    Pack8 av, r;
    av.u = __ldg(reinterpret_cast<const uint4*>(a + e));
#pragma unroll
    for (int k = 0; k < 8; ++k) r.h[k] = __float2bfloat16_rn(__bfloat162float(av.h[k]) > 0.f ? v[k] : 0.f);
    *reinterpret_cast<uint4*>(dz + e) = r.u;
  }
};
struct StoreEpi {  // FP32 store (gradient on the upsampled grid)
  float* out;
  int rows, cols;
  using Row = int;
  __device__ __forceinline__ Row prep(int m) const { return m; }
  __device__ __forceinline__ void operator()(int row, int col, const float* v) const {
    if (row >= rows) return;
    float4* o = reinterpret_cast<float4*>(out + (size_t)row * cols + col);
    o[0] = make_float4(v[0], v[1], v[2], v[3]);
    o[1] = make_float4(v[4], v[5], v[6], v[7]);
  }
};
struct WgradImageEpi {  // split-K partial sums of dW[oc][k]; k9 a multiple of 8
  float* g;
  int oc, k9;
  using Row = int;
  __device__ __forceinline__ Row prep(int m) const { return m; }
  __device__ __forceinline__ void operator()(int row, int col, const float* v) const {
    if (row >= oc || col >= k9) return;
    float4* o = reinterpret_cast<float4*>(g + (size_t)row * k9 + col);
    atomicAdd(o, make_float4(v[0], v[1], v[2], v[3]));
    atomicAdd(o + 1, make_float4(v[4], v[5], v[6], v[7]));
  }
};
struct WgradEpi {  // the same for layer 1 (nine columns)
  float* g;
  int oc, k9;
  using Row = int;
  __device__ __forceinline__ Row prep(int m) const { return m; }
  __device__ __forceinline__ void operator()(int row, int col, const float* v) const {
    if (row >= oc) return;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (col + e < k9) atomicAdd(g + (size_t)row * k9 + col + e, v[e]);
  }
};


// ---------------------------------------------------------------------------------------------
// Layer 6 on the CUDA cores
// ---------------------------------------------------------------------------------------------
// P[p][j] = sum_c w6[j][c] a5[p][c]: one warp per low-resolution pixel, 8 channels per lane, weights in registers over
// all of a warp's pixels.  The eighteen sums over lanes are halved along with the lanes (20 shuffles; the same
// additions as eighteen butterflies, whose 90 shuffles one after the other took 102 us on 65536 pixels; 33 here).
template <int NV>
__device__ __forceinline__ void halve(float* t, int o, bool upper) {
  constexpr int H = (NV + 1) / 2;
#pragma unroll
  for (int i = 0; i < H; ++i) {
    const float hi = i + H < NV ? t[i + H] : 0.f;
    t[i] = (upper ? hi : t[i]) + __shfl_xor_sync(0xffffffffu, upper ? t[i] : hi, o);
  }
}
__global__ void __launch_bounds__(128) k_l6_sums(const bf16* __restrict__ a5, const float* __restrict__ w6,
                                                 float* __restrict__ P, int npix) {
  static_assert(kTaps6 == 18, "the halving below");
  const int lane = threadIdx.x & 31, step = gridDim.x * 4;
  float w[kTaps6][8];
#pragma unroll
  for (int j = 0; j < kTaps6; ++j)
#pragma unroll
    for (int e = 0; e < 8; ++e) w[j][e] = __ldg(w6 + j * kC6 + lane * 8 + e);
  // 18 -> 9 -> 5 -> 3 -> 2 -> 1 values: the one that this lane ends with, if it is one
  const int i4 = lane & 1, i3 = i4 + (lane & 2), i2 = i3 + (lane & 4 ? 3 : 0), i1 = i2 + (lane & 8 ? 5 : 0);
  const int mine = i1 + (lane & 16 ? 9 : 0);
  const bool valid = i3 < 3 && i2 < 5 && i1 < 9;
  int p = blockIdx.x * 4 + (threadIdx.x >> 5);
  Pack8 v, nv;
  if (p < npix) nv.u = __ldg(reinterpret_cast<const uint4*>(a5 + (size_t)p * kC6 + lane * 8));
  for (; p < npix; p += step) {
    v = nv;
    if (p + step < npix) nv.u = __ldg(reinterpret_cast<const uint4*>(a5 + (size_t)(p + step) * kC6 + lane * 8));
    float t[kTaps6];
#pragma unroll
    for (int j = 0; j < kTaps6; ++j) t[j] = 0.f;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float x = __bfloat162float(v.h[e]);
#pragma unroll
      for (int j = 0; j < kTaps6; ++j) t[j] = fmaf(w[j][e], x, t[j]);
    }
    halve<18>(t, 16, lane & 16);
    halve<9>(t, 8, lane & 8);
    halve<5>(t, 4, lane & 4);
    halve<3>(t, 2, lane & 2);
    halve<2>(t, 1, lane & 1);
    if (valid) P[(size_t)p * kTaps6 + mine] = t[0];
  }
}

// out[b][y][x][o] = bias[o] + sum_tap P[b][(y + ky - 1) / 4][(x + kx - 1) / 4][tap][o] over taps
// inside the upsampled grid (hs = 4 * hl pixels per side).
__global__ void k_l6_out(const float* __restrict__ P, const float* __restrict__ bias, float* __restrict__ out, int B,
                         int hl) {
  const int hs = 4 * hl;
  const size_t n = (size_t)B * hs * hs * kOut;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int o = (int)(i % kOut);
    const size_t px = i / kOut;
    const int x = (int)(px % hs), y = (int)((px / hs) % hs), b = (int)(px / ((size_t)hs * hs));
    float acc = bias[o];
    for (int tap = 0; tap < 9; ++tap) {
      const int uy = y + tap / 3 - 1, ux = x + tap % 3 - 1;
      if (uy < 0 || uy >= hs || ux < 0 || ux >= hs) continue;
      acc += P[(((size_t)b * hl + uy / 4) * hl + ux / 4) * kTaps6 + tap * kOut + o];
    }
    out[i] = acc;
  }
}

// Loss partial sums (FP64 per block, fixed order) and dz6 = bf16(2 (pred - Y) / n).
__global__ void __launch_bounds__(256) k_loss(const float* __restrict__ pred, const float* __restrict__ Y,
                                              bf16* __restrict__ dz6, double* __restrict__ lpart, size_t n) {
  double acc = 0.0;
  const float g = (float)(2.0 / (double)n);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float d = pred[i] - Y[i];
    acc += (double)d * d;
    dz6[i] = __float2bfloat16_rn(g * d);
  }
  __shared__ double red[256];
  red[threadIdx.x] = acc;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) lpart[blockIdx.x] = red[0];
}
__global__ void __launch_bounds__(256) k_loss_final(const double* __restrict__ lpart, int nb, size_t n, double* loss) {
  __shared__ double red[256];
  double t = 0.0;
  for (int i = threadIdx.x; i < nb; i += 256) t += lpart[i];
  red[threadIdx.x] = t;
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if ((int)threadIdx.x < h) red[threadIdx.x] += red[threadIdx.x + h];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = red[0] / (double)n;
}

// dP[p][tap][o] = sum of dz6 over the output pixels that read low-resolution pixel p through tap:
// y + ky - 1 in [4 sy, 4 sy + 3] and inside the grid.
__global__ void k_l6_dsums(const bf16* __restrict__ dz6, float* __restrict__ dP, int B, int hl) {
  const int hs = 4 * hl;
  const size_t n = (size_t)B * hl * hl * kTaps6;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(i % kTaps6), tap = j / kOut, o = j % kOut;
    const size_t p = i / kTaps6;
    const int sx = (int)(p % hl), sy = (int)((p / hl) % hl), b = (int)(p / ((size_t)hl * hl));
    const int ky = tap / 3, kx = tap % 3;
    float acc = 0.f;
    for (int dy = 0; dy < 4; ++dy) {
      const int y = 4 * sy + dy + 1 - ky;
      if (y < 0 || y >= hs) continue;
      for (int dx = 0; dx < 4; ++dx) {
        const int x = 4 * sx + dx + 1 - kx;
        if (x < 0 || x >= hs) continue;
        acc += __bfloat162float(dz6[(((size_t)b * hs + y) * hs + x) * kOut + o]);
      }
    }
    dP[i] = acc;
  }
}

// dz5[p][c] = bf16((a5[p][c] > 0) sum_j dP[p][j] w6[j][c]) and dW6[o][tap][c] += sum over the CTA's pixels of dP[p][tap 2 + o]
// a5[p][c]: thread c keeps its channel's weights and sums in registers, eight pixels' operands in flight (a
// CTA per pixel, and a pass over a5 per tap and output: 64 + 131 us on 65536 pixels).
__global__ void __launch_bounds__(kC6) k_l6_grad(const float* __restrict__ dP, const float* __restrict__ w6,
                                                 const bf16* __restrict__ a5, bf16* __restrict__ dz5, float* __restrict__ gW6,
                                                 int npix) {
  constexpr int U = 8;
  __shared__ float d[U * kTaps6];
  const int c = threadIdx.x;
  float w[kTaps6], g[kTaps6];
#pragma unroll
  for (int j = 0; j < kTaps6; ++j) {
    w[j] = __ldg(w6 + j * kC6 + c);
    g[j] = 0.f;
  }
  for (int p0 = blockIdx.x * U; p0 < npix; p0 += gridDim.x * U) {
    const int n = min(U, npix - p0);
    __syncthreads();
    if (c < n * kTaps6) d[c] = dP[(size_t)p0 * kTaps6 + c];
    float a[U];
#pragma unroll
    for (int u = 0; u < U; ++u) a[u] = u < n ? __bfloat162float(a5[(size_t)(p0 + u) * kC6 + c]) : 0.f;
    __syncthreads();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (u >= n) break;
      float acc = 0.f;
#pragma unroll
      for (int j = 0; j < kTaps6; ++j) {
        const float dj = d[u * kTaps6 + j];
        acc = fmaf(dj, w[j], acc);
        g[j] = fmaf(dj, a[u], g[j]);
      }
      dz5[(size_t)(p0 + u) * kC6 + c] = __float2bfloat16_rn(a[u] > 0.f ? acc : 0.f);
    }
  }
#pragma unroll
  for (int j = 0; j < kTaps6; ++j) atomicAdd(gW6 + ((size_t)(j % kOut) * 9 + j / kOut) * kC6 + c, g[j]);
}

// ---------------------------------------------------------------------------------------------
// Bias gradients, upsampling adjoint, Adam
// ---------------------------------------------------------------------------------------------
// gb[c] += sum over a chunk of pixels of dz[p][c].
__global__ void k_bias_grad(const bf16* __restrict__ dz, float* __restrict__ gb, size_t npix, int C, int chunk) {
  const size_t p0 = (size_t)blockIdx.x * chunk;
  const size_t p1 = p0 + chunk < npix ? p0 + chunk : npix;
  for (int c = threadIdx.x; c < C; c += blockDim.x) {
    float acc = 0.f;
    for (size_t p = p0; p < p1; ++p) acc += __bfloat162float(dz[p * C + c]);
    atomicAdd(gb + c, acc);
  }
}

// dz[b][y][x][c] = bf16((a > 0) sum of the f x f block of du on the upsampled grid), four channels a thread.
__global__ void __launch_bounds__(256) k_upsample_grad(const float* __restrict__ du, const bf16* __restrict__ a,
                                                       bf16* __restrict__ dz, int B, int h, int C, int f) {
  const size_t n = (size_t)B * h * h * C / 4;
  const int hu = h * f;
  for (size_t i = blockIdx.x * (size_t)256 + threadIdx.x; i < n; i += (size_t)gridDim.x * 256) {
    const int c = 4 * (int)(i % (C / 4));
    const size_t px = i / (C / 4);
    const int x = (int)(px % h), y = (int)((px / h) % h), b = (int)(px / ((size_t)h * h));
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int dy = 0; dy < f; ++dy)
      for (int dx = 0; dx < f; ++dx) {
        const float4 v = *reinterpret_cast<const float4*>(du + (((size_t)b * hu + f * y + dy) * hu + f * x + dx) * C + c);
        acc.x += v.x;
        acc.y += v.y;
        acc.z += v.z;
        acc.w += v.w;
      }
    union {
      uint2 u;
      bf16 e[4];
    } av, r;
    av.u = *reinterpret_cast<const uint2*>(a + px * C + c);
    r.e[0] = __float2bfloat16_rn(__bfloat162float(av.e[0]) > 0.f ? acc.x : 0.f);
    r.e[1] = __float2bfloat16_rn(__bfloat162float(av.e[1]) > 0.f ? acc.y : 0.f);
    r.e[2] = __float2bfloat16_rn(__bfloat162float(av.e[2]) > 0.f ? acc.z : 0.f);
    r.e[3] = __float2bfloat16_rn(__bfloat162float(av.e[3]) > 0.f ? acc.w : 0.f);
    *reinterpret_cast<uint2*>(dz + px * C + c) = r.u;
  }
}

__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v, const float* __restrict__ g,
                       size_t n, float lr, float b1, float b2, float eps, float bc1, float bc2_sqrt) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= (lr / bc1) * mi / (sqrtf(vi) / bc2_sqrt + eps);
  }
}

// ---------------------------------------------------------------------------------------------
// Targets and stitching
// ---------------------------------------------------------------------------------------------
__device__ __forceinline__ void window_corner(const float* pos, int j, int S, int H, int W, int* i0, int* i1) {
  float r0 = rintf(pos[2 * j]), r1 = rintf(pos[2 * j + 1]);  // half to even, as the forward model
  if (!isfinite(r0)) r0 = 0.f;
  if (!isfinite(r1)) r1 = 0.f;
  *i0 = (int)fminf(fmaxf(r0, 0.f), (float)(H - S));
  *i1 = (int)fminf(fmaxf(r1, 0.f), (float)(W - S));
}

__global__ void k_targets(int S, int Nz, int H, int W, const float* __restrict__ amp, const float* __restrict__ phase,
                          const float* __restrict__ pos, const int32_t* __restrict__ idx, int B, float* __restrict__ Y) {
  const int h = S / 2, q = S / 4;
  const size_t n = (size_t)B * h * h;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % h), y = (int)((i / h) % h), b = (int)(i / ((size_t)h * h));
    int i0, i1;
    window_corner(pos, idx[b], S, H, W, &i0, &i1);
    const size_t e = (size_t)(i0 + q + y) * W + (i1 + q + x);
    double ph = 0.0, la = 0.0;
    for (int s = 0; s < Nz; ++s) {
      ph += phase[(size_t)s * H * W + e];
      la += log((double)amp[(size_t)s * H * W + e]);
    }
    Y[2 * i] = (float)ph;
    Y[2 * i + 1] = (float)la;
  }
}

__global__ void k_stitch(int S, int H, int W, const float* __restrict__ pred, const float* __restrict__ pos,
                         const int32_t* __restrict__ idx, int B, const float* __restrict__ wgt, float* __restrict__ num,
                         float* __restrict__ den) {
  const int h = S / 2, q = S / 4;
  const size_t n = (size_t)B * h * h;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int x = (int)(i % h), y = (int)((i / h) % h), b = (int)(i / ((size_t)h * h));
    int i0, i1;
    window_corner(pos, idx[b], S, H, W, &i0, &i1);
    const size_t e = (size_t)(i0 + q + y) * W + (i1 + q + x);
    const float w = wgt[y * h + x];
    atomicAdd(num + 2 * e, w * pred[2 * i]);
    atomicAdd(num + 2 * e + 1, w * pred[2 * i + 1]);
    atomicAdd(den + e, w);
  }
}

__global__ void k_stitch_finish(int Nz, int H, int W, const float* __restrict__ num, const float* __restrict__ den,
                                float* __restrict__ amp, float* __restrict__ phase) {
  const size_t n = (size_t)H * W;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float d = den[i];
    const float ph = d > 0.f ? num[2 * i] / d / Nz : 0.f;
    const float am = d > 0.f ? expf(num[2 * i + 1] / d / Nz) : 1.f;
    for (int s = 0; s < Nz; ++s) {
      phase[(size_t)s * n + i] = ph;
      amp[(size_t)s * n + i] = am;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Weight-gradient operands with pixel-contiguous rows
// ---------------------------------------------------------------------------------------------
// Tile image of colT[k][m - p0] = im2col[m][k] for k = (tap, ic) < 9 IC and output pixels m in [p0, p0 + P); zero past the
// last pixel (layers 2..5, ic a multiple of 16).  A warp takes 16 pixels by two groups of 8 channels: per tap each
// lane loads its pixel's 16 bytes, eight lanes transpose 8 pixels x 8 channels, and every store is one core
// matrix row, 128 contiguous bytes per eight lanes.
__global__ void __launch_bounds__(256) k_im2col_t(const bf16* __restrict__ a, bf16* __restrict__ colt, int B, int hin, int hu,
                                                  int hout, int ic, int stride, int up, int p0, int P) {
  const int hw = hout * hout, pixels = B * hw, pairs = ic / 16, k9 = 9 * ic, lane = threadIdx.x & 31;
  const size_t warps = (size_t)pairs * (P / 16), step = (size_t)gridDim.x * 8;
  const int sh = up == 2 ? 1 : 0;
  for (size_t w = blockIdx.x * (size_t)8 + (threadIdx.x >> 5); w < warps; w += step) {
    const int mm = (int)(w / pairs) * 16 + (lane & 15), c0 = (int)(w % pairs) * 16 + 8 * (lane >> 4), m = p0 + mm;
    int b = 0, y0 = -1 << 20, x0 = -1 << 20;
    if (m < pixels) {
      b = m / hw;
      const int rem = m % hw;
      y0 = stride * (rem / hout) - 1;
      x0 = stride * (rem % hout) - 1;
    }
    const bf16* img = a + (size_t)b * hin * hin * ic + c0;
#pragma unroll
    for (int tap = 0; tap < 9; ++tap) {
      const int uy = y0 + tap / 3, ux = x0 + tap % 3;
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (uy >= 0 && uy < hu && ux >= 0 && ux < hu)
        v = __ldg(reinterpret_cast<const uint4*>(img + ((size_t)(uy >> sh) * hin + (ux >> sh)) * ic));
      uint32_t r[4] = {v.x, v.y, v.z, v.w};
      transpose8(r, lane);
      // this lane now holds channel c0 + lane % 8 of the eight pixels from mm & ~7
      *reinterpret_cast<uint4*>(colt + image_index(tap * ic + c0 + (lane & 7), (size_t)(mm & ~7), k9)) =
          make_uint4(r[0], r[1], r[2], r[3]);
    }
  }
}

// Layer 1 (one channel from the patterns): tile image of sixteen rows, taps 0..8 and zeros, of pixels [p0, p0 + P).
__global__ void __launch_bounds__(256) k_im2col_t1(const float* __restrict__ I, float s_in, bf16* __restrict__ colt, int B,
                                                   int S, int hout, int p0, int P) {
  const int hw = hout * hout, pixels = B * hw, lane = threadIdx.x & 31;
  for (int mm = blockIdx.x * 256 + threadIdx.x; mm < P; mm += gridDim.x * 256) {  // P a multiple of 64: whole warps
    const int m = p0 + mm;
    Pack8 lo, hi;
    lo.u = hi.u = make_uint4(0u, 0u, 0u, 0u);
    if (m < pixels) {
      const int b = m / hw, rem = m % hw, oy = rem / hout, ox = rem % hout;
#pragma unroll
      for (int tap = 0; tap < 9; ++tap) {
        const int y = 2 * oy + tap / 3 - 1, x = 2 * ox + tap % 3 - 1;
        if (y >= 0 && y < S && x >= 0 && x < S) (tap < 8 ? lo : hi).h[tap & 7] = input_value(I, s_in, S, b, y, x);
      }
    }
    uint32_t r[4] = {lo.u.x, lo.u.y, lo.u.z, lo.u.w}, t[4] = {hi.u.x, 0u, 0u, 0u};
    transpose8(r, lane);
    transpose8(t, lane);
    bf16* o = colt + image_index(lane & 7, (size_t)(mm & ~7), 16);
    *reinterpret_cast<uint4*>(o) = make_uint4(r[0], r[1], r[2], r[3]);
    *reinterpret_cast<uint4*>(o + 512) = make_uint4(t[0], t[1], t[2], t[3]);  // rows 8..15
  }
}

// Tile image of dzT[c][m - p0] = dz[m][c] for m in [p0, p0 + P) (zero past the last pixel; P a multiple of 64, C of 16), and the
// bias gradient: gb[c] += the sum over the pixels.  blockIdx.y takes 16 channels; a warp takes 16 pixels at a time and
// transposes as k_im2col_t (32 x 32 tiles through shared memory, two bytes a thread: 283 us a step, now 96).
__global__ void __launch_bounds__(256) k_dz_t(const bf16* __restrict__ dz, bf16* __restrict__ dzt, float* __restrict__ gb,
                                              int pixels, int C, int p0, int P) {
  const int lane = threadIdx.x & 31, c0 = blockIdx.y * 16 + 8 * (lane >> 4);
  float sum = 0.f;
  for (int w = blockIdx.x * 8 + (threadIdx.x >> 5); w < P / 16; w += gridDim.x * 8) {
    const int mm = 16 * w + (lane & 15), m = p0 + mm;
    const uint4 v = m < pixels ? __ldg(reinterpret_cast<const uint4*>(dz + (size_t)m * C + c0)) : make_uint4(0u, 0u, 0u, 0u);
    uint32_t r[4] = {v.x, v.y, v.z, v.w};
    transpose8(r, lane);
    *reinterpret_cast<uint4*>(dzt + image_index(c0 + (lane & 7), (size_t)(mm & ~7), C)) = make_uint4(r[0], r[1], r[2], r[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) sum += __uint_as_float(r[i] << 16) + __uint_as_float(r[i] & 0xffff0000u);
  }
  sum += __shfl_xor_sync(0xffffffffu, sum, 8);  // the warp's other eight pixels
  __shared__ float part[8][16];
  if (!(lane & 8)) part[threadIdx.x >> 5][(lane & 7) + 8 * (lane >> 4)] = sum;
  __syncthreads();
  if (threadIdx.x < 16) {
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += part[k][threadIdx.x];
    atomicAdd(gb + blockIdx.y * 16 + threadIdx.x, t);
  }
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
#define CNN_CHECK(what)                                                  \
  do {                                                                   \
    cudaError_t e_ = cudaGetLastError();                                 \
    if (e_ != cudaSuccess) {                                             \
      set_error("%s launch failed: %s", what, cudaGetErrorString(e_));   \
      return PTY_ECUDA;                                                  \
    }                                                                    \
    note_launch();                                                       \
  } while (0)

static unsigned blocks_for(size_t n, unsigned cap = 152 * 16) {
  const size_t b = (n + 255) / 256;
  return (unsigned)(b < 1 ? 1 : (b > cap ? cap : b));
}

static int gemm_result(cudaError_t e, const char* what) {
  if (e != cudaSuccess) {
    set_error("%s launch failed: %s", what, cudaGetErrorString(e));
    return PTY_ECUDA;
  }
  note_launch();
  return PTY_OK;
}
// C = A B^T over row_tiles x 128 rows and b.rows columns in tiles of BN, which divides them, K = 64 kb_all
template <int BN, int KS = 4, class LA, class Epi>
static int gemm(const LA& la, const ImageOperand& b, int row_tiles, int kb_all, const Epi& epi, int* status,
                cudaStream_t st, int splits = 1) {
  return gemm_result(launch_gemm_ws<BN, KS>(la, b, WsWork{row_tiles, b.rows / BN, splits, kb_all, 0}, epi, status, st),
                     "k_gemm_ws");
}

struct Buffers {
  int* status;
  bf16 *wp[5], *wt[5], *act[5], *dz[6];
  float *w6, *p6, *dp6, *du5;
  double* lpart;
  bf16 *colt, *dzt;
};

static Buffers carve(const Plan& pl, void* ws) {
  char* base = static_cast<char*>(ws);
  Buffers b;
  memset(&b, 0, sizeof(b));
  b.status = reinterpret_cast<int*>(base + pl.status);
  for (int l = 0; l < 5; ++l) {
    b.wp[l] = reinterpret_cast<bf16*>(base + pl.wp[l]);
    if (l > 0) b.wt[l] = reinterpret_cast<bf16*>(base + pl.wt[l]);
    b.act[l] = reinterpret_cast<bf16*>(base + pl.act[l]);
    b.dz[l] = reinterpret_cast<bf16*>(base + pl.dz[l]);
  }
  b.dz[5] = reinterpret_cast<bf16*>(base + pl.dz[5]);
  b.w6 = reinterpret_cast<float*>(base + pl.w6);
  b.p6 = reinterpret_cast<float*>(base + pl.p6);
  b.dp6 = reinterpret_cast<float*>(base + pl.dp6);
  b.du5 = reinterpret_cast<float*>(base + pl.du5);
  b.lpart = reinterpret_cast<double*>(base + pl.lpart);
  b.colt = reinterpret_cast<bf16*>(base + pl.colt);
  b.dzt = reinterpret_cast<bf16*>(base + pl.dzt);
  return b;
}

// Pack the weights and run layers 1..6; pred[B][S/2][S/2][2].
static int run_forward(const Plan& pl, const Buffers& bu, const float* params, const float* I, float s_in, float* pred,
                       cudaStream_t st) {
  PackArgs pa;
  pa.params = params;
  for (int l = 0; l < 5; ++l) {
    pa.wp[l] = bu.wp[l];
    pa.wt[l] = bu.wt[l];
  }
  pa.w6 = bu.w6;
  for (int l = 0; l < kLayers; ++l) {
    pa.woff[l] = pl.woff[l];
    pa.kp[l] = pl.kp[l];
    pa.ktp[l] = pl.ktp[l];
    pa.ic[l] = kNet[l].ic;
    pa.oc[l] = kNet[l].oc;
  }
  if (cudaMemsetAsync(bu.status, 0, sizeof(int), st) != cudaSuccess) {
    set_error("cudaMemsetAsync failed: %s", cudaGetErrorString(cudaGetLastError()));
    return PTY_ECUDA;
  }
  k_pack<<<152 * 16, 256, 0, st>>>(pa);
  CNN_CHECK("k_pack");
  const int B = pl.B;
  if (B == 0) return PTY_OK;
  for (int l = 0; l < 5; ++l) {
    const LayerDef& L = kNet[l];
    const size_t rows = (size_t)B * pl.hout[l] * pl.hout[l];
    const ImageOperand w{bu.wp[l], L.oc};
    int rc;
    if (l == 0) {  // rows of 16 in the weight gradients' scratch, in pieces that fit it
      const size_t fit = pl.colt_elems / 16 / 128 * 128;
      for (size_t p0 = 0; p0 < rows; p0 += fit) {
        const size_t n = rows - p0 < fit ? rows - p0 : fit;
        k_input_rows<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(I, s_in, bu.colt, pl.S, pl.hout[0], p0, n);
        CNN_CHECK("k_input_rows");
        FwdEpi epi{bu.act[0] + p0 * L.oc, params + pl.boff[0], (int)n, L.oc};
        if ((rc = gemm<48, 1>(InputRows{bu.colt, (int)n}, w, (int)((n + 127) / 128), 1, epi, bu.status, st))) return rc;
      }
    } else {
      FwdEpi epi{bu.act[l], params + pl.boff[l], (int)rows, L.oc};
      const int tiles = (int)((rows + 127) / 128), kb = pl.kp[l] / 64;
      const Im2col<1> la{bu.act[l - 1], B, pl.hin[l], pl.hu[l], pl.hout[l], L.ic, L.stride};
      const Im2col<2> la2{bu.act[l - 1], B, pl.hin[l], pl.hu[l], pl.hout[l], L.ic, L.stride};
      rc = l == 1 ? gemm<96>(la, w, tiles, kb, epi, bu.status, st)
         : l == 4 ? gemm<256>(la2, w, tiles, kb, epi, bu.status, st) : gemm<192>(la, w, tiles, kb, epi, bu.status, st);
      if (rc) return rc;
    }
  }
  const int hl = pl.hout[4], npix = B * hl * hl;
  k_l6_sums<<<npix < 4 * 152 * 4 ? (npix + 3) / 4 : 152 * 4, 128, 0, st>>>(bu.act[4], bu.w6, bu.p6, npix);
  CNN_CHECK("k_l6_sums");
  k_l6_out<<<blocks_for((size_t)B * 16 * hl * hl * kOut), 256, 0, st>>>(bu.p6, params + pl.boff[5], pred, B, hl);
  CNN_CHECK("k_l6_out");
  return PTY_OK;
}

// Loss, then gradients of every layer (grad zeroed here).
static int run_backward(const Plan& pl, const Buffers& bu, const float* I, float s_in, const float* pred, const float* Y,
                        double* loss, float* grad, cudaStream_t st) {
  const int B = pl.B;
  if (cudaMemsetAsync(grad, 0, sizeof(float) * param_count(), st) != cudaSuccess) {
    set_error("cudaMemsetAsync failed");
    return PTY_ECUDA;
  }
  if (B == 0) {
    if (cudaMemsetAsync(loss, 0, sizeof(double), st) != cudaSuccess) {
      set_error("cudaMemsetAsync failed");
      return PTY_ECUDA;
    }
    return PTY_OK;
  }
  const int hs = pl.hout[5], hl = pl.hout[4];
  const size_t nout = (size_t)B * hs * hs * kOut;
  const unsigned lb = blocks_for(nout, 1024);
  k_loss<<<lb, 256, 0, st>>>(pred, Y, bu.dz[5], bu.lpart, nout);
  CNN_CHECK("k_loss");
  k_loss_final<<<1, 256, 0, st>>>(bu.lpart, (int)lb, nout, loss);
  CNN_CHECK("k_loss_final");
  // layer 6
  const int npix = B * hl * hl;
  k_l6_dsums<<<blocks_for((size_t)npix * kTaps6), 256, 0, st>>>(bu.dz[5], bu.dp6, B, hl);
  CNN_CHECK("k_l6_dsums");
  k_l6_grad<<<npix < 8 * 152 * 4 ? (npix + 7) / 8 : 152 * 4, kC6, 0, st>>>(bu.dp6, bu.w6, bu.act[4], bu.dz[4],
                                                                          grad + pl.woff[5], npix);
  CNN_CHECK("k_l6_grad");
  const size_t pix6 = (size_t)B * hs * hs;
  k_bias_grad<<<(unsigned)((pix6 + 1023) / 1024), 256, 0, st>>>(bu.dz[5], grad + pl.boff[5], pix6, kOut, 1024);
  CNN_CHECK("k_bias_grad");
  // layers 5..1
  for (int l = 4; l >= 0; --l) {
    const LayerDef& L = kNet[l];
    const int pixels = B * pl.hout[l] * pl.hout[l];
    const int k9 = 9 * L.ic;
    // dW[oc][k] = sum over pixels of dz[m][oc] im2col[m][k], chunk by chunk, both operands
    // transposed to pixel-contiguous rows first (plain 16-byte loads in the GEMM)
    const int P = pl.pchunk[l];
    for (int p0 = 0; p0 < pixels; p0 += P) {
      const unsigned xb = (unsigned)((P / 16 + 7) / 8), cap = 152 * 16 / (L.oc / 16);
      k_dz_t<<<dim3(xb < cap ? xb : cap, L.oc / 16), 256, 0, st>>>(bu.dz[l], bu.dzt, grad + pl.boff[l], pixels, L.oc, p0, P);
      CNN_CHECK("k_dz_t");
      if (l == 0)
        k_im2col_t1<<<blocks_for((size_t)P), 256, 0, st>>>(I, s_in, bu.colt, B, pl.S, pl.hout[0], p0, P);
      else
        k_im2col_t<<<blocks_for((size_t)L.ic / 16 * P * 2), 256, 0, st>>>(bu.act[l - 1], bu.colt, B, pl.hin[l], pl.hu[l],
                                                                         pl.hout[l], L.ic, L.stride, L.up, p0, P);
      CNN_CHECK("k_im2col_t");
      // 9 ic = 432, 864, 1728 or 3456 columns: tiles of 144 divide them; layer 1: one tile of 16
      const ImageLoad la{ImageOperand{bu.dzt, L.oc}};
      const int row_tiles = (L.oc + 127) / 128, tiles = row_tiles * (l == 0 ? 1 : k9 / 144), splits = 2 * 152 / tiles;
      const int rc = l == 0 ? gemm<16>(la, ImageOperand{bu.colt, 16}, row_tiles, P / 64,
                                       WgradEpi{grad + pl.woff[l], L.oc, k9}, bu.status, st, splits)
                            : gemm<144>(la, ImageOperand{bu.colt, k9}, row_tiles, P / 64,
                                        WgradImageEpi{grad + pl.woff[l], L.oc, k9}, bu.status, st, splits);
      if (rc) return rc;
    }
    if (l == 0) break;
    const GradRows gr(B, pl.hu[l], L.stride);
    const int kb = pl.ktp[l] / 64;
    const DgradGather ga(bu.dz[l], gr, pl.hout[l], L.oc, kb);
    const ImageOperand wt{bu.wt[l], L.ic};
    int rc;
    if (L.up == 1) {
      const DgradEpi epi{bu.dz[l - 1], bu.act[l - 1], gr, L.ic};
      rc = l == 1 ? gemm<48>(ga, wt, gr.row_tiles(), kb, epi, bu.status, st)
         : l == 2 ? gemm<96>(ga, wt, gr.row_tiles(), kb, epi, bu.status, st)
                  : gemm<192>(ga, wt, gr.row_tiles(), kb, epi, bu.status, st);
    } else {
      rc = gemm<192>(ga, wt, gr.row_tiles(), kb, StoreEpi{bu.du5, B * pl.hu[l] * pl.hu[l], L.ic}, bu.status, st);
      if (rc) return rc;
      k_upsample_grad<<<blocks_for((size_t)B * pl.hin[l] * pl.hin[l] * L.ic / 4), 256, 0, st>>>(
          bu.du5, bu.act[l - 1], bu.dz[l - 1], B, pl.hin[l], L.ic, L.up);
      CNN_CHECK("k_upsample_grad");
    }
    if (rc) return rc;
  }
  return PTY_OK;
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

static int check(int S, int B, const void* ws, size_t ws_bytes, Plan* pl) {
  if (!make_plan(S, B, pl)) {
    set_error("S = %d, B = %d not supported (S a multiple of 16 in [16, 512], 0 <= B <= 1024)", S, B);
    return PTY_EINVAL;
  }
  if (!ws || ((uintptr_t)ws & 255)) {
    set_error("workspace is NULL or not 256-byte aligned");
    return PTY_EINVAL;
  }
  if (ws_bytes < pl->total) {
    set_error("workspace has %zu bytes, %zu needed", ws_bytes, pl->total);
    return PTY_EWORKSPACE;
  }
  return PTY_OK;
}

__global__ void k_to_f32(const bf16* __restrict__ x, float* __restrict__ y, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    y[i] = __bfloat162float(x[i]);
}

}  // namespace cnn
}  // namespace pty

using namespace pty;
using namespace pty::cnn;

extern "C" {

size_t pty_cnn_param_count(void) { return param_count(); }

size_t pty_cnn_workspace_size(int S, int B) {
  Plan pl;
  if (!make_plan(S, B, &pl)) {
    set_error("S = %d, B = %d not supported (S a multiple of 16 in [16, 512], 0 <= B <= 1024)", S, B);
    return 0;
  }
  return pl.total;
}

int pty_cnn_forward(int S, int B, const float* params, const float* I, float s_in, float* pred, void* ws,
                    size_t ws_bytes, void* stream) {
  Plan pl;
  int rc = check(S, B, ws, ws_bytes, &pl);
  if (rc) return rc;
  if (!params || !aligned16(params) || (B > 0 && (!I || !pred || !aligned16(I) || !aligned16(pred)))) {
    set_error("params, I and pred must be non-NULL and 16-byte aligned");
    return PTY_EINVAL;
  }
  return run_forward(pl, carve(pl, ws), params, I, s_in, pred, (cudaStream_t)stream);
}

int pty_cnn_loss_grad(int S, int B, const float* params, const float* I, const float* Y, float s_in, double* loss,
                      float* grad, float* pred, void* ws, size_t ws_bytes, void* stream) {
  Plan pl;
  int rc = check(S, B, ws, ws_bytes, &pl);
  if (rc) return rc;
  if (!params || !grad || !loss || !aligned16(params) || !aligned16(grad) ||
      (B > 0 && (!I || !Y || !aligned16(I) || !aligned16(Y))) || (pred && !aligned16(pred))) {
    set_error("params, grad, loss, I and Y must be non-NULL and 16-byte aligned");
    return PTY_EINVAL;
  }
  const Buffers bu = carve(pl, ws);
  float* out = pred ? pred : bu.du5;  // du5 is free until layer 5's input gradient
  if ((size_t)B * pl.hout[5] * pl.hout[5] * kOut > (size_t)B * pl.hu[4] * pl.hu[4] * kNet[4].ic && !pred) {
    set_error("internal: prediction scratch too small");
    return PTY_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)stream;
  rc = run_forward(pl, bu, params, I, s_in, out, st);
  if (rc) return rc;
  return run_backward(pl, bu, I, s_in, out, Y, loss, grad, st);
}

int pty_cnn_adam(float* params, float* m, float* v, const float* grad, int step, float lr, float beta1, float beta2,
                 float eps, void* stream) {
  if (!params || !m || !v || !grad || step < 1 || !(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) ||
      !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f)) {
    set_error("bad Adam arguments");
    return PTY_EINVAL;
  }
  const double bc1 = 1.0 - pow((double)beta1, step), bc2 = 1.0 - pow((double)beta2, step);
  const size_t n = param_count();
  k_adam<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(params, m, v, grad, n, lr, beta1, beta2, eps, (float)bc1,
                                                          (float)sqrt(bc2));
  CNN_CHECK("k_adam");
  return PTY_OK;
}

int pty_cnn_train_step(int S, int B, float* params, float* m, float* v, float* grad, int step, float lr,
                       const float* I, const float* Y, float s_in, double* loss, void* ws, size_t ws_bytes,
                       void* stream) {
  int rc = pty_cnn_loss_grad(S, B, params, I, Y, s_in, loss, grad, nullptr, ws, ws_bytes, stream);
  if (rc) return rc;
  return pty_cnn_adam(params, m, v, grad, step, lr, 0.9f, 0.999f, 1e-8f, stream);
}

int pty_cnn_targets(int S, int Nz, int H, int W, const float* amp, const float* phase, const float* pos,
                    const int32_t* idx, int B, float* Y, void* stream) {
  if (S < 16 || S % 16 || Nz < 1 || H < S || W < S || B < 0 || (B > 0 && (!amp || !phase || !pos || !idx || !Y))) {
    set_error("bad target arguments");
    return PTY_EINVAL;
  }
  if (B == 0) return PTY_OK;
  k_targets<<<blocks_for((size_t)B * S * S / 4), 256, 0, (cudaStream_t)stream>>>(S, Nz, H, W, amp, phase, pos, idx, B,
                                                                                Y);
  CNN_CHECK("k_targets");
  return PTY_OK;
}

int pty_cnn_stitch(int S, int H, int W, const float* pred, const float* pos, const int32_t* idx, int B,
                   const float* weight, float* num, float* den, void* stream) {
  if (S < 16 || S % 16 || H < S || W < S || B < 0 || !weight || !num || !den || (B > 0 && (!pred || !pos || !idx))) {
    set_error("bad stitch arguments");
    return PTY_EINVAL;
  }
  if (B == 0) return PTY_OK;
  k_stitch<<<blocks_for((size_t)B * S * S / 4), 256, 0, (cudaStream_t)stream>>>(S, H, W, pred, pos, idx, B, weight,
                                                                               num, den);
  CNN_CHECK("k_stitch");
  return PTY_OK;
}

int pty_cnn_stitch_finish(int Nz, int H, int W, const float* num, const float* den, float* amp, float* phase,
                          void* stream) {
  if (Nz < 1 || H < 1 || W < 1 || !num || !den || !amp || !phase) {
    set_error("bad stitch arguments");
    return PTY_EINVAL;
  }
  k_stitch_finish<<<blocks_for((size_t)H * W), 256, 0, (cudaStream_t)stream>>>(Nz, H, W, num, den, amp, phase);
  CNN_CHECK("k_stitch_finish");
  return PTY_OK;
}

int pty_cnn_read_state(int S, int B, const void* ws, size_t ws_bytes, int layer, int what, float* out,
                       void* stream) {
  Plan pl;
  int rc = check(S, B, ws, ws_bytes, &pl);
  if (rc) return rc;
  if (layer < 1 || layer > kLayers || what < 0 || what > 1 || (what == 0 && layer == kLayers) || (B > 0 && !out)) {
    set_error("bad state request: layer %d, what %d", layer, what);
    return PTY_EINVAL;
  }
  const Buffers bu = carve(pl, const_cast<void*>(ws));
  const int l = layer - 1;
  const size_t n = (size_t)B * pl.hout[l] * pl.hout[l] * kNet[l].oc;
  if (n == 0) return PTY_OK;
  k_to_f32<<<blocks_for(n), 256, 0, (cudaStream_t)stream>>>(what == 0 ? bu.act[l] : bu.dz[l], out, n);
  CNN_CHECK("k_to_f32");
  return PTY_OK;
}

}  // extern "C"
