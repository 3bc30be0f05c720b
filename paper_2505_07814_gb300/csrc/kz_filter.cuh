// kz_filter.cuh -- the k_z filter (Eq. 10-12): the periodic 3D DFT of z = amp + i phase, the real even
// filter W_a, and the inverse, in five passes over a complex workspace volume.
//
//   x lines, forward   amp, phase [Nz][H][W]  ->  z in blocks of eight x positions, [x / 8][s][y][x % 8]
//   y lines, forward   in place, eight lines (one block of one slice, contiguous) side by side
//   depth              per (k_y, k_x) column, in place
//   y lines, inverse   in place
//   x lines, inverse   z  ->  amp, phase with the relaxation
//
// Line transforms.  One CTA transforms C lines at a time in shared memory, each pass one read and one
// write of it with a 16- or 8-point DFT in registers (fft_smem.cuh), so a line of 1024 takes three
// barriers where one radix-2 stage at a time took ten.  The forward passes decimate in frequency
// and leave the spectrum in the digit order of their radices; the depth step asks kz_bin() for the
// bin of a position and the inverse passes consume that order, so nothing is ever reordered.  Lines
// whose length is not a power of two are Bluestein convolutions (L. I. Bluestein, IEEE Trans. Audio
// Electroacoustics 18(4), 1970) with P >= 2 L - 1 points, the chirp's spectrum kept in shared
// memory and every CTA running many tiles so that it is built rarely.
//
// Depth step.  W_a is real and even in k_z, so "DFT over depth, filter, inverse DFT" is a circular
// convolution of the column with a real kernel h(d) = sum_k W_a(k) cos(2 pi k d / Nz), h(d) = h(Nz - d):
// 2 FMAs per pair of slices where the two DFTs take 8.
//
// Measured (GB300, one call; before: one radix-2 stage per barrier, direct DFTs for other lengths, a DFT
// pair over depth): 20 x 1024 x 1024 1954 -> 751 us, 6 x 614 x 614 5226 -> 256 us.  The five passes
// move 88 bytes per voxel: 2.5 TB/s on the large volume, bound by the latency of each tile's load,
// barrier-separated passes and store with two CTAs on an SM; the ragged lines are bound by their arithmetic.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "fft_smem.cuh"
#include "pty_internal.h"

namespace pty {

constexpr int kMaxLine = 8192;
constexpr int kKzThreads = 256;
constexpr int kKzSmem = 224 * 1024;  // shared memory of one CTA at most
constexpr float kKzEps = 1e-3f;      // per square angstrom, the stabilising constant under Eq. 10

enum { KZ_POW2 = 0, KZ_BLUESTEIN = 1, KZ_DIRECT = 2 };

// One line length: the transform's points P, its passes (log2 of their radices, 3 or 4) and how it
// is computed.  Bluestein needs two P-point arrays in shared memory, which fit up to P = 8192; longer
// lines that are not powers of two (L > 4096) take the direct O(L^2) sum.
struct KzLine {
  int L, P, lgP, npass, kind;
  unsigned radices;  // four bits per pass
  __host__ __device__ int lgR(int i) const { return (radices >> (4 * i)) & 15; }
};
inline KzLine kz_line(int L) {
  KzLine k;
  memset(&k, 0, sizeof(k));
  k.L = L;
  const bool pow2 = (L & (L - 1)) == 0;
  k.kind = pow2 ? KZ_POW2 : L <= 4096 ? KZ_BLUESTEIN : KZ_DIRECT;
  const int least = pow2 ? L : 2 * L - 1;
  while ((1 << k.lgP) < least) ++k.lgP;
  k.P = 1 << k.lgP;
  k.npass = (k.lgP + 3) / 4;  // L >= 64, so every pass gets 3 or 4 levels
  for (int i = 0; i < k.npass; ++i) k.radices |= (unsigned)(k.lgP / k.npass + (i < k.lgP % k.npass ? 1 : 0)) << (4 * i);
  return k;
}
// Shared-memory place of element i: one float2 of padding per 16 keeps the strided accesses of the
// later passes (8 or 16 apart) off each other's banks.
__host__ __device__ constexpr int kz_pad(int i) { return i + (i >> 4); }
// Distance of the lines of a tile, chosen mod 16 so that a half warp's accesses in z's order meet no
// bank twice: x tiles take 8 positions of 2 lines at once (8 mod 16), y tiles 2 positions of 8 lines (2).
__host__ __device__ inline int kz_line_stride(int P, bool x) {
  const int n = P + P / 16;
  return n + (((x ? 8 : 2) - n) & 15);
}
// Element (x position, slice, y) of z: blocks of 8 x positions (the last one narrower), so that neither the
// x passes nor the y passes touch less than a run of the block's width.
__host__ __device__ inline size_t kz_block(int b, int Nz, int H) { return (size_t)8 * b * Nz * H; }
__host__ __device__ inline int kz_width(int b, int W) { return W - 8 * b < 8 ? W - 8 * b : 8; }
inline size_t kz_table_bytes(const KzLine& k) {
  if (k.kind == KZ_DIRECT) return sizeof(float2) * (size_t)k.L;
  return sizeof(float2) * ((size_t)k.P / 2 + (k.kind == KZ_BLUESTEIN ? (size_t)k.L + 1 + kz_line_stride(k.P, true) : 0));
}
inline size_t kz_lines_bytes(const KzLine& k, int C) {
  return sizeof(float2) * (k.kind == KZ_DIRECT ? 2 * (size_t)k.L : (size_t)C * (k.P + k.P / 16 + 16));
}
// Bin of spectrum position p.
__host__ __device__ inline int kz_bin(const KzLine& k, int p) {
  if (k.kind != KZ_POW2) return p;
  int f = 0, mul = 0, rem = k.lgP;
  for (int i = 0; i < k.npass; ++i) {
    rem -= k.lgR(i);
    f += (p >> rem) << mul;
    p &= (1 << rem) - 1;
    mul += k.lgR(i);
  }
  return f;
}

// DFT frequency of bin i of n samples spaced d, in cycles per unit of d (numpy's fftfreq)
__device__ __forceinline__ float fft_freq(int i, int n, float d) {
  return (float)(i < (n + 1) / 2 ? i : i - n) / ((float)n * d);
}
// exp(-i pi t / n) for 0 <= t < 2 n: t / n is split into a float and its remainder, so that the angle is
// exact to second order
__device__ __forceinline__ float2 kz_root(int t, int n) {
  if (t > n) t -= 2 * n;
  const float hi = (float)t / (float)n, lo = fmaf(-hi, (float)n, (float)t) / (float)n;
  float s, c;
  sincospif(hi, &s, &c);
  const float d = 3.14159265358979f * lo;
  return make_float2(fmaf(-d, s, c), -fmaf(d, c, s));
}

// v[i] times W^i (its conjugate for INV), W = tw[e]; the powers of W come from four (R = 16) or three (R = 8)
// table entries and at most two products.
template <int R, bool INV>
__device__ __forceinline__ void kz_twiddle(float2* v, const float2* tw, int e) {
  float2 w[R];
  w[1] = tw[e];
  w[2] = tw[2 * e];
  w[4] = tw[4 * e];
  if constexpr (R == 16) w[8] = tw[8 * e];
  w[3] = cmul(w[2], w[1]);
#pragma unroll
  for (int i = 1; i < R; ++i) {
    if (i > 4 && i != 8) w[i] = cmul(w[i >= 8 ? 8 : 4], w[i - (i >= 8 ? 8 : 4)]);
    v[i] = INV ? cmulc(w[i], v[i]) : cmul(w[i], v[i]);
  }
}
// One pass of the P-point transform of `lines` lines: sub-transforms of n = 2^lgn points, radix R.
// Forward (decimation in frequency): DFT over elements n / R apart, times W_n^{jk}; inverse: its mirror.
// tw[t] = exp(-2 pi i t / P), t < P / 2.
template <int R, bool INV>
__device__ __forceinline__ void kz_pass(float2* buf, int lines, int ls, int lgP, int lgn, const float2* tw) {
  constexpr int LR = R == 16 ? 4 : 3;
  const int lgm = lgn - LR, per = lgP - LR, total = lines << per;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const int q = t & ((1 << per) - 1), j = q & ((1 << lgm) - 1);
    float2* line = buf + (t >> per) * ls;
    const int base = ((q >> lgm) << lgn) + j;
    float2 v[R];
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = line[kz_pad(base + (i << lgm))];
    if (!INV) dft<R, false>(v);
    if (lgm > 0) kz_twiddle<R, INV>(v, tw, j << (lgP - lgn));
    if (INV) dft<R, true>(v);
#pragma unroll
    for (int i = 0; i < R; ++i) line[kz_pad(base + (i << lgm))] = v[i];
  }
  __syncthreads();
}
// natural order -> digit order; LAST: all passes, else all but the last (n = R)
template <bool LAST = true>
__device__ __forceinline__ void kz_forward(float2* buf, int lines, int ls, const KzLine& k, const float2* tw) {
  int lgn = k.lgP;
  for (int i = 0; i < k.npass - (LAST ? 0 : 1); ++i) {
    if (k.lgR(i) == 4) kz_pass<16, false>(buf, lines, ls, k.lgP, lgn, tw);
    else kz_pass<8, false>(buf, lines, ls, k.lgP, lgn, tw);
    lgn -= k.lgR(i);
  }
}
// digit order -> natural order, conjugate sign, not normalised; FIRST: all passes, else all but the first (n = R)
template <bool FIRST = true>
__device__ __forceinline__ void kz_inverse(float2* buf, int lines, int ls, const KzLine& k, const float2* tw) {
  int lgn = FIRST ? 0 : k.lgR(k.npass - 1);
  for (int i = k.npass - (FIRST ? 1 : 2); i >= 0; --i) {
    lgn += k.lgR(i);
    if (k.lgR(i) == 4) kz_pass<16, true>(buf, lines, ls, k.lgP, lgn, tw);
    else kz_pass<8, true>(buf, lines, ls, k.lgP, lgn, tw);
  }
}
// The middle of a convolution: the last forward pass, the product with the kernel's spectrum bhat and the
// first inverse pass work on the same R consecutive elements, so they share one trip through registers.
template <int R>
__device__ __forceinline__ void kz_middle(float2* buf, int lines, int ls, int lgP, const float2* bhat) {
  constexpr int LR = R == 16 ? 4 : 3;
  const int per = lgP - LR, total = lines << per;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    float2* line = buf + (t >> per) * ls;
    const int base = (t & ((1 << per) - 1)) << LR;
    float2 v[R];
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = line[kz_pad(base + i)];
    dft<R, false>(v);
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = cmul(v[i], bhat[kz_pad(base + i)]);
    dft<R, true>(v);
#pragma unroll
    for (int i = 0; i < R; ++i) line[kz_pad(base + i)] = v[i];
  }
  __syncthreads();
}

enum KzMode { KZ_X_FWD, KZ_X_INV, KZ_Y_FWD, KZ_Y_INV };

template <int BYTES>
__device__ __forceinline__ void kz_copy(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem),
               "n"(BYTES)
               : "memory");
}

struct KzArgs {
  float2* z;            // blocked volume (kz_block)
  float *amp, *phase;   // [Nz][H][W]
  float relax;
  int Nz, H, W, C;
  long long tiles;
  KzLine line;
};

// Every CTA takes tiles blockIdx.x, + gridDim.x, ...  x modes: C lines y0 .. y0 + C - 1 of one slice; y modes: C
// of the lines of one block and slice.
template <int MODE, int KIND>
__global__ void __launch_bounds__(kKzThreads, 2) k_kz_lines(KzArgs a) {
  constexpr bool INV = MODE == KZ_X_INV || MODE == KZ_Y_INV, X = MODE == KZ_X_FWD || MODE == KZ_X_INV;
  extern __shared__ __align__(16) float2 kz_sm[];
  const KzLine& k = a.line;
  const int L = k.L, P = k.P, C = a.C, tid = threadIdx.x, T = blockDim.x;
  const int ls = KIND == KZ_DIRECT ? L : kz_line_stride(P, X);
  float2* tw = kz_sm;
  float2* chirp = tw + P / 2;             // Bluestein: exp(-i pi j^2 / L)
  float2* bhat = chirp + ((L + 1) & ~1);  // Bluestein: spectrum of the conjugate chirp / P
  float2* buf = KIND == KZ_DIRECT ? tw + L : KIND == KZ_POW2 ? tw + P / 2 : bhat + kz_line_stride(P, true);
  if (KIND == KZ_DIRECT) {
    for (int t = tid; t < L; t += T) tw[t] = kz_root(2 * t, L);
  } else {
    for (int t = tid; t < P / 2; t += T) {
      float s, c;
      sincospif(-2.0f * (float)t / (float)P, &s, &c);
      tw[t] = make_float2(c, s);
    }
  }
  if (KIND == KZ_BLUESTEIN) {
    for (int j = tid; j < L; j += T) chirp[j] = kz_root((int)(((long long)j * j) % (2 * L)), L);
    __syncthreads();
    for (int i = tid; i < P; i += T) {
      const int j = i < L ? i : P - i;  // the chirp and its mirror image around 0 (mod P)
      bhat[kz_pad(i)] = j < L ? cconj(chirp[j]) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    kz_forward(bhat, 1, ls, k, tw);
    for (int i = tid; i < P; i += T) bhat[kz_pad(i)] = cscale(bhat[kz_pad(i)], 1.0f / (float)P);
  }
  __syncthreads();

  const int parts = X ? (a.H + C - 1) / C : 8 / C;  // tiles per slice / per block and slice
  for (long long tile = blockIdx.x; tile < a.tiles; tile += gridDim.x) {
    const int part = (int)(tile % parts), l0 = part * C;
    const int s = (int)(tile / parts % a.Nz), b = X ? 0 : (int)(tile / parts / a.Nz);
    const int width = X ? 0 : kz_width(b, a.W);
    const int lines = X ? min(C, a.H - l0) : min(C, width - l0);
    if (lines <= 0) continue;  // the narrow last block
    auto get = [&](int l, int j) {
      if (KIND == KZ_POW2) return buf[l * ls + kz_pad(j)];
      const float2 v = KIND == KZ_BLUESTEIN ? cmul(buf[l * ls + kz_pad(j)], chirp[j]) : buf[L + j];
      return INV ? cconj(v) : v;
    };
    // the tile in z's order: f(line, position, element of z), consecutive threads on consecutive elements
    auto each_z = [&](auto&& f) {
      if (X) {  // C lines by 8 positions are contiguous in each block
        const int sub = tid & 7, row = tid >> 3;
        for (int e = row; e < (L + 7) / 8 * C; e += T / 8) {
          const int l = e & (C - 1), xb = e / C, j = 8 * xb + sub;
          if (l < lines && j < L) f(l, j, kz_block(xb, a.Nz, a.H) + ((size_t)s * a.H + l0 + l) * kz_width(xb, a.W) + sub);
        }
      } else {
        const size_t base = kz_block(b, a.Nz, a.H) + (size_t)s * a.H * width + l0;
        const int l = tid & (C - 1);
        if (l < lines)
          for (int j = tid / C; j < L; j += T / C) f(l, j, base + (size_t)j * width + l);
      }
    };
    // asynchronous loads of the whole tile: every element is in flight at once, where a loop of loads into
    // registers waited for each round of them (20 x 1024 x 1024, y lines: 257 us a
    // pass, now 130)
    auto place = [&](int l, int j) { return buf + l * ls + (KIND == KZ_DIRECT ? j : kz_pad(j)); };
    if (MODE == KZ_X_FWD) {
      for (int l = 0; l < lines; ++l) {
        const size_t e = ((size_t)s * a.H + l0 + l) * a.W;
        for (int j = tid; j < L; j += T) {
          float2* d = place(l, j);
          kz_copy<4>(&d->x, a.amp + e + j);
          kz_copy<4>(&d->y, a.phase + e + j);
        }
      }
    } else {
      each_z([&](int l, int j, size_t e) { kz_copy<8>(place(l, j), a.z + e); });
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (KIND != KZ_POW2) {  // conjugate for the inverse, times the chirp, zeros up to P
      for (int l = 0; l < lines; ++l)
        for (int j = tid; j < (KIND == KZ_DIRECT ? L : P); j += T) {
          float2 v = make_float2(0.f, 0.f);
          if (j < L) {
            v = *place(l, j);
            if (INV) v = cconj(v);
            if (KIND == KZ_BLUESTEIN) v = cmul(v, chirp[j]);
          }
          *place(l, j) = v;
        }
      __syncthreads();
    }
    if (KIND == KZ_POW2) {
      if (INV) kz_inverse(buf, lines, ls, k, tw);
      else kz_forward(buf, lines, ls, k, tw);
    } else if (KIND == KZ_BLUESTEIN) {
      kz_forward<false>(buf, lines, ls, k, tw);
      if (k.lgR(k.npass - 1) == 4) kz_middle<16>(buf, lines, ls, k.lgP, bhat);
      else kz_middle<8>(buf, lines, ls, k.lgP, bhat);
      kz_inverse<false>(buf, lines, ls, k, tw);
    } else {
      for (int f = tid; f < L; f += T) {
        float2 acc = make_float2(0.f, 0.f);
        int t = 0;  // (j f) mod L
        for (int j = 0; j < L; ++j) {
          const float2 x = buf[j], w = tw[t];
          acc.x = fmaf(x.x, w.x, fmaf(-x.y, w.y, acc.x));
          acc.y = fmaf(x.x, w.y, fmaf(x.y, w.x, acc.y));
          t += f;
          if (t >= L) t -= L;
        }
        buf[L + f] = acc;
      }
      __syncthreads();
    }
    if (MODE == KZ_X_INV) {
      for (int l = 0; l < lines; ++l) {
        float* x = a.amp + ((size_t)s * a.H + l0 + l) * a.W;
        float* y = a.phase + ((size_t)s * a.H + l0 + l) * a.W;
        for (int j0 = tid; j0 < L; j0 += 4 * T) {  // four loads of each in flight
          float xv[4], yv[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j0 + u * T;
            xv[u] = j < L ? x[j] : 0.f;
            yv[u] = j < L ? y[j] : 0.f;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int j = j0 + u * T;
            if (j < L) {
              const float2 v = get(l, j);
              x[j] = xv[u] + a.relax * (v.x - xv[u]);
              y[j] = yv[u] + a.relax * (v.y - yv[u]);
            }
          }
        }
      }
    } else {
      each_z([&](int l, int j, size_t e) { a.z[e] = get(l, j); });
    }
    __syncthreads();  // the tile's lines are free
  }
}

// Depth step: CTA (chunk of a block's columns, block), one thread per column.  Shared memory: the chunk's column
// values [Nz][T], W_a and h [Nz / 2 + 1][T], the cosines [Nz] and the fold of a slice distance onto h's index.
// Outputs are formed eight at a time from eight inputs and the fifteen kernel values between them.
constexpr int kDepthThreads = 128;
inline size_t kz_depth_bytes(int Nz) {
  const size_t q = (size_t)Nz / 2 + 1;
  return sizeof(float2) * Nz * kDepthThreads + sizeof(float) * (2 * q * kDepthThreads + Nz) +
         sizeof(int) * (2 * (size_t)Nz + 32);
}
__global__ void __launch_bounds__(kDepthThreads)
    k_kz_depth(float2* __restrict__ z, int Nz, int H, int W, float dx, const float* __restrict__ dz, float beta,
               float alpha, KzLine lx, KzLine ly) {
  constexpr int T = kDepthThreads;
  extern __shared__ __align__(16) float2 kz_sm[];
  const int q = Nz / 2 + 1, tid = threadIdx.x;
  float2* col = kz_sm;                                       // [Nz][T]
  float* wk = reinterpret_cast<float*>(col + (size_t)Nz * T);  // [q][T]
  float* h = wk + (size_t)q * T;                             // [q][T]
  float* ct = h + (size_t)q * T;                             // cos(2 pi t / Nz)
  int* fold = reinterpret_cast<int*>(ct + Nz);               // of distance i - Nz - 15
  const int width = kz_width(blockIdx.y, W), c = blockIdx.x * T + tid;
  const bool in = c < H * width;
  const int y = c / width, px = 8 * blockIdx.y + c % width;
  const size_t row = (size_t)H * width;
  float2* zc = z + kz_block(blockIdx.y, Nz, H) + c;
  if (in)
    for (int s = 0; s < Nz; ++s) kz_copy<8>(col + s * T + tid, zc + s * row);
  for (int t = tid; t < Nz; t += T) ct[t] = cospif(2.0f * (float)t / (float)Nz);
  for (int i = tid; i < 2 * Nz + 31; i += T) {
    int d = i - Nz - 15;
    d = (d < 0 ? -d : d) % Nz;
    fold[i] = d <= Nz - d ? d : Nz - d;
  }
  if (in) {
    const float kx = fft_freq(kz_bin(lx, px), W, dx), ky = fft_freq(kz_bin(ly, y), H, dx);
    const float kr2 = kx * kx + ky * ky, dzv = *dz;
    const float lateral = expf(-alpha * kr2) / ((float)Nz * ((float)H * (float)W));
    const float b2 = beta * beta, den = kr2 + kKzEps;
    for (int k = 0; k < q; ++k) {
      const float kz = fft_freq(k, Nz, dzv);
      const float w = (1.0f - 0.63661977236758134f * atanf(b2 * kz * kz / den)) * lateral;  // 2 / pi
      // bins k and Nz - k together, except bin 0 and (even Nz) bin Nz / 2
      wk[k * T + tid] = (k == 0 || 2 * k == Nz) ? w : 2.0f * w;
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (!in) return;
  for (int d = 0; d < q; ++d) {
    float acc = 0.f;
    int t = 0;  // (k d) mod Nz
    for (int k = 0; k < q; ++k) {
      acc = fmaf(wk[k * T + tid], ct[t], acc);
      t += d;
      if (t >= Nz) t -= Nz;
    }
    h[d * T + tid] = acc;
  }
  for (int s0 = 0; s0 < Nz; s0 += 8) {
    float2 acc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) acc[u] = make_float2(0.f, 0.f);
    for (int t0 = 0; t0 < Nz; t0 += 8) {
      float w[15];  // h at distances s0 - t0 - 7 .. s0 - t0 + 7
#pragma unroll
      for (int i = 0; i < 15; ++i) w[i] = h[fold[s0 - t0 - 7 + i + Nz + 15] * T + tid];
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const float2 x = t0 + v < Nz ? col[(t0 + v) * T + tid] : make_float2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          acc[u].x = fmaf(w[u - v + 7], x.x, acc[u].x);
          acc[u].y = fmaf(w[u - v + 7], x.y, acc[u].y);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (s0 + u < Nz) zc[(s0 + u) * row] = acc[u];
  }
}

}  // namespace pty
