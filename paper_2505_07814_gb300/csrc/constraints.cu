// constraints.cu -- the constraints applied after an optimiser step (pty_constrain, include/pty.h;
// Sec. "Physical constraints").
//
//   probe orthogonalisation  k_gram (FP64 Gram-matrix partials of the probe modes), k_ortho_eig
//                            (one CTA: complex Jacobi eigensolver in FP64, disjoint rotations side by
//                            side, modes sorted by power), k_ortho_apply (each pixel's modes mixed
//                            by the eigenvectors, in place);
//   k_z filter (Eq. 10-12)   kz_filter.cuh: k_kz_lines along x and y, k_kz_depth, k_kz_lines back;
//   depth blur, positivity   k_constrain (Eq. 13 and the phase clip).
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include "kz_filter.cuh"
#include "pty_internal.h"

namespace pty {

// ---------------------------------------------------------------------------------------------
// Depth blur and positivity.  One CTA per (tile of T x V pixels of the plane, array): cp.async
// copies the tile's Nz slices to shared memory (each element is read from HBM once), each thread
// blurs its V pixel columns along depth with the Gaussian taps held in shared memory and writes
// every output once; the phase CTAs apply the relaxed positivity clip on the way out.
// HBM-bound: 8 bytes per element and array.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxBlurSlices = 128;
constexpr int kConstrainSmem = 200 * 1024;

template <int V>
__global__ void k_constrain(float* __restrict__ x0, float* __restrict__ x1, int Nz, size_t plane, float sigma, int R,
                            float rz_relax, float pos_relax) {
  extern __shared__ __align__(16) unsigned char c_smem[];
  float* taps = reinterpret_cast<float*>(c_smem);  // w(d) = exp(-d^2 / (2 sigma^2)), d = 0 .. R
  float* rden = taps + kMaxBlurSlices;             // 1 / (sum of slice s's taps inside the volume)
  float* tile = rden + kMaxBlurSlices;             // [Nz][T * V]
  float* x = blockIdx.y ? x1 : x0;
  const float clip = x == x1 ? pos_relax : 0.f;  // x1 is the phase
  const int T = blockDim.x, tid = threadIdx.x;
  const size_t p = (blockIdx.x * (size_t)T + tid) * V;
  const bool in = p < plane;  // V = 4 needs plane % 4 == 0, so the whole vector is inside

  if (!(sigma > 0.f)) {  // positivity alone
    if (in) {
      for (int s = 0; s < Nz; ++s) {
        float* q = x + (size_t)s * plane + p;
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const float y = q[v];
          if (y < 0.f) q[v] = y - clip * y;
        }
      }
    }
    return;
  }
  for (int s = 0; s < Nz; ++s) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(tile + ((size_t)s * T + tid) * V);
    const float* g = x + (size_t)s * plane + (in ? p : 0);
    if (V == 4)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(g), "r"(in ? 16 : 0) : "memory");
    else
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(g), "r"(in ? 4 : 0) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int d = tid; d <= R; d += T) {
    const float u = (float)d / sigma;
    taps[d] = expf(-0.5f * u * u);
  }
  __syncthreads();
  for (int s = tid; s < Nz; s += T) {
    const int t0 = s - R > 0 ? s - R : 0, t1 = s + R < Nz - 1 ? s + R : Nz - 1;
    float den = 0.f;
    for (int t = t0; t <= t1; ++t) den += taps[t > s ? t - s : s - t];
    rden[s] = 1.f / den;
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  if (!in) return;
  for (int s = 0; s < Nz; ++s) {
    const int t0 = s - R > 0 ? s - R : 0, t1 = s + R < Nz - 1 ? s + R : Nz - 1;
    float acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = 0.f;
    for (int t = t0; t <= t1; ++t) {
      const float w = taps[t > s ? t - s : s - t];
      const float* src = tile + ((size_t)t * T + tid) * V;
      if constexpr (V == 4) {
        const float4 q = *reinterpret_cast<const float4*>(src);
        acc[0] = fmaf(w, q.x, acc[0]);
        acc[1] = fmaf(w, q.y, acc[1]);
        acc[2] = fmaf(w, q.z, acc[2]);
        acc[3] = fmaf(w, q.w, acc[3]);
      } else {
        acc[0] = fmaf(w, src[0], acc[0]);
      }
    }
    const float* own = tile + ((size_t)s * T + tid) * V;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const float v0 = own[v];
      float y = v0 + rz_relax * (acc[v] * rden[s] - v0);
      if (y < 0.f) y -= clip * y;
      acc[v] = y;
    }
    float* dst = x + (size_t)s * plane + p;
    if constexpr (V == 4)
      *reinterpret_cast<float4*>(dst) = make_float4(acc[0], acc[1], acc[2], acc[3]);
    else
      dst[0] = acc[0];
  }
}

// The dynamic shared memory that launches of `kern` may ask for.  The limit belongs to the function and not to a launch, and
// host threads with other sizes share it: every call that needs more than the default sets the same number, the
// largest that any call needs.
template <class Kern>
static int allow_smem(Kern kern, size_t bytes, size_t largest, const char* what) {
  if (bytes > 48 * 1024 &&
      cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)largest) != cudaSuccess) {
    set_error("cudaFuncSetAttribute(%s) failed: %s", what, cudaGetErrorString(cudaGetLastError()));
    return PTY_ECUDA;
  }
  return PTY_OK;
}

template <int V>
static int launch_constrain(float* amp, float* phase, int Nz, size_t plane, float sigma, float rz_relax,
                            float pos_relax, cudaStream_t st) {
  const bool blur = sigma > 0.f;
  int T = 128;
  size_t smem = 0;
  if (blur) {
    const size_t fixed = 2 * kMaxBlurSlices * sizeof(float);
    T = (int)((kConstrainSmem - fixed) / ((size_t)Nz * V * sizeof(float)));
    T = T >= 128 ? 128 : T / 32 * 32;
    smem = fixed + (size_t)Nz * T * V * sizeof(float);
    if (int rc = allow_smem(k_constrain<V>, smem, kConstrainSmem, "k_constrain")) return rc;
  }
  const int R0 = (int)ceilf(4.0f * sigma);
  const int R = blur ? (R0 < Nz - 1 ? R0 : Nz - 1) : 0;
  const size_t per = (size_t)T * V;
  const dim3 grid((unsigned)((plane + per - 1) / per), blur ? 2 : 1);
  // without the blur only the phase is touched: the single row of CTAs takes x0 = phase
  k_constrain<V><<<grid, T, smem, st>>>(blur ? amp : phase, phase, Nz, plane, sigma, R, rz_relax, pos_relax);
  return PTY_OK;
}

// ---------------------------------------------------------------------------------------------
// Probe orthogonalisation (mixed-state probe, Sec. "Physical constraints").  With the modes as the
// rows of A (M x N^2): G = A A^H = U diag(lambda) U^H, Q = U^H A, modes ordered by decreasing
// power lambda; each column of U is turned so that its largest-magnitude entry is real positive.
// ---------------------------------------------------------------------------------------------
constexpr int kMaxOrthoModes = 32;
constexpr int kGramChunk = 256;    // pixels per k_gram CTA
constexpr int kGramTile = 128;     // pixels in shared memory at a time
constexpr int kJacobiSweeps = 60;  // cyclic sweeps at most (convergence is quadratic; a handful suffice)

__device__ __forceinline__ void pair_of(int pair, int M, int* m, int* n) {
  int r = pair, i = 0;
  while (r >= M - i) {  // row i holds the pairs (i, i .. M-1)
    r -= M - i;
    ++i;
  }
  *m = i;
  *n = i + r;
}

// partial[pair][chunk] = sum over the chunk's pixels of P_m conj(P_n), m <= n.  A CTA converts its pixels'
// modes to FP64 once in shared memory and every thread sums one mode pair over one of `groups` shares
// of the pixels, so the pass is bound by the FP64 units (4 products per pixel and pair); one CTA per
// (chunk, pair) read and converted every mode M times (N = 256, M = 12: 132 us, now
// 50).
__global__ void __launch_bounds__(256) k_gram(const float2* __restrict__ probe, int M, int NN,
                                              double2* __restrict__ partial) {
  extern __shared__ __align__(16) double2 g_px[];  // [kGramTile][M], then [256] partial sums
  double2* red = g_px + (size_t)kGramTile * M;
  const int tid = threadIdx.x, np = M * (M + 1) / 2, c0 = blockIdx.x * kGramChunk;
  // np <= 528: up to three pairs a thread.  M = 2 and 3 take 16 shares a pair instead of 85 and 42, whose addition
  // one after the other was most of the pass (N = 64: 9.6 and 8.0 us, now 6.5 and 6.7)
  const int groups = np < 8 ? 16 : np < 256 ? 256 / np : 1;
  const int grp = np < 256 ? tid / np : 0;
  double re[3] = {0.0, 0.0, 0.0}, im[3] = {0.0, 0.0, 0.0};
  int pm[3], pn[3], cnt = 0;
  for (int p = np < 256 ? tid % np : tid; p < np && cnt < 3 && grp < groups; p += np < 256 ? np : 256, ++cnt)
    pair_of(p, M, &pm[cnt], &pn[cnt]);
  for (int t0 = c0; t0 < min(NN, c0 + kGramChunk); t0 += kGramTile) {
    __syncthreads();
    for (int e = tid; e < kGramTile * M; e += 256) {
      const int m = e / kGramTile, p = e % kGramTile;
      const float2 v = t0 + p < NN ? probe[(size_t)m * NN + t0 + p] : make_float2(0.f, 0.f);
      g_px[p * M + m] = make_double2(v.x, v.y);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (k >= cnt) break;
      for (int p = grp; p < kGramTile; p += groups) {
        const double2 x = g_px[p * M + pm[k]], y = g_px[p * M + pn[k]];
        re[k] = fma(x.y, y.y, fma(x.x, y.x, re[k]));
        im[k] = fma(-x.x, y.y, fma(x.y, y.x, im[k]));
      }
    }
  }
  if (np >= 256) {
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (k < cnt) partial[(size_t)(tid + 256 * k) * gridDim.x + blockIdx.x] = make_double2(re[k], im[k]);
    return;
  }
  red[tid] = make_double2(re[0], im[0]);
  __syncthreads();
  if (tid < np) {
    double2 t = red[tid];
    for (int g = 1; g < groups; ++g) {
      t.x += red[g * np + tid].x;
      t.y += red[g * np + tid].y;
    }
    partial[(size_t)tid * gridDim.x + blockIdx.x] = t;
  }
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zlin(double a, double2 x, double2 b, double2 y) {  // a x + b y
  return make_double2(fma(a, x.x, fma(b.x, y.x, -b.y * y.y)), fma(a, x.y, fma(b.x, y.y, b.y * y.x)));
}

// One CTA: reduce the Gram partials, diagonalise with cyclic complex Jacobi rotations in FP64, sort,
// fix the phases; writes U (column k = eigenvector of the k-th largest power) and lambda.
// A sweep is M - 1 rounds of a round-robin tournament (M even; an odd M sits one mode out): a round's
// M / 2 rotations touch disjoint mode pairs, so they run side by side.  What bounds it is the chain of FP64
// operations of a round (an FP64 instruction occupies a scheduler for many clocks, however few of its
// lanes are live), so a thread forms one entry of one 2 x 2 block, the rotations come from two reciprocal
// square roots, and V follows G one round behind on the warps that would wait for them.  One rotation after the
// other by one warp took 1.10 ms at M = 12; this 0.18-0.20.
__global__ void __launch_bounds__(256) k_ortho_eig(const double2* __restrict__ partial, int M, int chunks,
                                                    double2* __restrict__ Uout, double* __restrict__ lam_out) {
  constexpr int kMaxPairs = kMaxOrthoModes / 2;
  __shared__ double2 G[kMaxOrthoModes][kMaxOrthoModes + 1];
  __shared__ double2 V[kMaxOrthoModes][kMaxOrthoModes + 1];
  __shared__ double lam[kMaxOrthoModes];
  __shared__ double rc[2][kMaxPairs];  // this round's rotations and the last one's (V follows a round behind)
  __shared__ double2 rs[2][kMaxPairs];
  __shared__ int rp[2][kMaxPairs], rq[2][kMaxPairs];
  __shared__ int done;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int npairs = M * (M + 1) / 2;
  for (int pr = warp; pr < npairs; pr += 8) {
    int m, n;
    pair_of(pr, M, &m, &n);
    double x = 0.0, y = 0.0;
    for (int c = lane; c < chunks; c += 32) {
      const double2 v = partial[(size_t)pr * chunks + c];
      x += v.x;
      y += v.y;
    }
    for (int o = 16; o > 0; o >>= 1) {
      x += __shfl_xor_sync(0xffffffffu, x, o);
      y += __shfl_xor_sync(0xffffffffu, y, o);
    }
    if (lane == 0) {
      G[m][n] = make_double2(x, m == n ? 0.0 : y);
      G[n][m] = make_double2(x, m == n ? 0.0 : -y);
    }
  }
  for (int i = tid; i < M * M; i += 256) V[i / M][i % M] = make_double2(i / M == i % M ? 1.0 : 0.0, 0.0);
  __syncthreads();
  const int n = (M + 1) & ~1, half = n / 2, tri = half * (half + 1) / 2;
  const double2 zero = make_double2(0.0, 0.0);
  // V <- V U for the rotations in slot k; the two threads of a pair of entries are neighbours, t0 a warp's
  // multiple of 32
  auto turn_v = [&](int k, int t0, int step) {
    for (int b = t0 + lane; b < (2 * M * half + 31) / 32 * 32; b += step) {
      const int row = b / 2 / half, j = b / 2 % half, d = b & 1;
      const bool on = row < M && rq[k][j] < M;  // the mode that sits out is left alone
      const int p = rp[k][j], q = rq[k][j];
      double2 v = zero;
      if (on) {
        const double2 s = rs[k][j], vp = V[row][p], vq = V[row][q];
        v = zlin(rc[k][j], d ? vq : vp, make_double2(d ? s.x : -s.x, s.y), d ? vp : vq);
      }
      __syncwarp();
      if (on) V[row][d ? q : p] = v;
    }
  };
  int rounds = 0;
  for (int sweep = 0; sweep < kJacobiSweeps; ++sweep) {
    if (warp == 0) {
      double off = 0.0, diag = 0.0;
      for (int i = lane; i < M; i += 32) {
        diag += G[i][i].x * G[i][i].x;
        for (int j = i + 1; j < M; ++j) off += G[i][j].x * G[i][j].x + G[i][j].y * G[i][j].y;
      }
      for (int o = 16; o > 0; o >>= 1) {
        off += __shfl_xor_sync(0xffffffffu, off, o);
        diag += __shfl_xor_sync(0xffffffffu, diag, o);
      }
      if (lane == 0) done = !(off > 1e-30 * diag);  // also ends on an all-zero matrix
    }
    __syncthreads();
    if (done) break;
    for (int r = 0; r < n - 1; ++r, ++rounds) {
      const int k = rounds & 1;
      if (warp == 0) {  // rotation `lane` of the round: the modes that meet at this table
        if (lane < half) {
          int p = lane == 0 ? n - 1 : (r + lane) % (n - 1), q = lane == 0 ? r : (r - lane + n - 1) % (n - 1);
          if (p > q) {
            const int t = p;
            p = q;
            q = t;
          }
          // c and the complex s of U_pp = U_qq = c, U_pq = s, U_qp = -conj(s), which zeroes g = G_pq.  With
          // d = G_qq - G_pp and r = sqrt(d^2 + 4 |g|^2): c^2 = (1 + |d| / r) / 2, s = sign(d) g / (r c)
          double c = 1.0;
          double2 s = zero;
          if (q < M) {
            const double2 g = G[p][q];
            const double g2 = fma(g.x, g.x, g.y * g.y), d = G[q][q].x - G[p][p].x, r2 = fma(d, d, 4.0 * g2);
            if (g2 > 1e-290) {  // else g is zero (or its square is denormal)
              const double ir = rsqrt(r2), c2 = fma(0.5 * fabs(d), ir, 0.5), ic = rsqrt(c2);
              const double f = (d >= 0.0 ? ir : -ir) * ic;
              c = c2 * ic;
              s = make_double2(g.x * f, g.y * f);
            }
          }
          rp[k][lane] = p;
          rq[k][lane] = q;
          rc[k][lane] = c;
          rs[k][lane] = s;
        }
      } else if (warp >= 3 && rounds > 0) {
        turn_v(k ^ 1, 32 * (warp - 3), 32 * 5);
      }
      __syncthreads();
      // G <- U^H G U, one thread per entry of the 2 x 2 blocks (rows of rotation i, columns of rotation j, i <= j),
      // the four of a block neighbours in one warp; blocks below the diagonal get the conjugates
      for (int b = tid; b < (4 * tri + 31) / 32 * 32; b += 256) {
        const bool in = b < 4 * tri;
        const int a = (b >> 1) & 1, d = b & 1;
        int i = 0, j = 0;
        if (in) pair_of(b >> 2, half, &i, &j);
        const int p = rp[k][j], q = rq[k][j], ip = rp[k][i], iq = rq[k][i];
        const bool okc = q < M, okr = iq < M;
        const bool on = in && (d ? okc : true) && (a ? okr : true);
        double2 g = zero;
        if (on) {
          const double2 b00 = G[ip][p], b01 = okc ? G[ip][q] : zero, b10 = okr ? G[iq][p] : zero,
                        b11 = okc && okr ? G[iq][q] : zero;
          const double c = rc[k][j], ci = rc[k][i];
          const double2 s = rs[k][j], si = rs[k][i], m = make_double2(d ? s.x : -s.x, s.y);
          const double2 x = zlin(c, d ? b01 : b00, m, d ? b00 : b01), y = zlin(c, d ? b11 : b10, m, d ? b10 : b11);
          g = zlin(ci, a ? y : x, make_double2(a ? si.x : -si.x, -si.y), a ? x : y);
          if (i == j) {  // the rotation's own block: exactly diagonal and real
            g.y = 0.0;
            if (a != d) g.x = 0.0;
          }
        }
        __syncwarp();
        if (on) {
          const int row = a ? iq : ip, col = d ? q : p;
          G[row][col] = g;
          if (i != j) G[col][row] = make_double2(g.x, -g.y);
        }
      }
      __syncthreads();
    }
  }
  if (rounds > 0) turn_v((rounds - 1) & 1, 32 * warp, 256);
  if (tid < M) lam[tid] = G[tid][tid].x;
  __syncthreads();
  if (tid < M) {
    // rank of this eigenpair by decreasing power (ties keep the index order)
    const double lk = lam[tid];
    int rank = 0;
    for (int j = 0; j < M; ++j) rank += (lam[j] > lk) || (lam[j] == lk && j < tid);
    int mstar = 0;
    double best = -1.0;
    for (int m = 0; m < M; ++m) {
      const double a = V[m][tid].x * V[m][tid].x + V[m][tid].y * V[m][tid].y;
      if (a > best) {
        best = a;
        mstar = m;
      }
    }
    const double2 vs = V[mstar][tid];
    const double av = sqrt(vs.x * vs.x + vs.y * vs.y);
    const double2 ph = av > 0.0 ? make_double2(vs.x / av, -vs.y / av) : make_double2(1.0, 0.0);
    for (int m = 0; m < M; ++m) Uout[(size_t)m * M + rank] = zmul(V[m][tid], ph);
    lam_out[rank] = lk;
  }
}

// Q_k[p] = sum_m conj(U[m][k]) P_m[p], in place; one thread per pixel, its M modes in shared memory, converted
// to FP64 once (bound by the FP64 units: 4 M^2 products per pixel; N = 256, M = 12: 170 us
// before, now 81).
__global__ void __launch_bounds__(128) k_ortho_apply(float2* __restrict__ probe, int M, int NN,
                                                      const double2* __restrict__ U) {
  extern __shared__ __align__(16) unsigned char o_smem[];
  double2* u = reinterpret_cast<double2*>(o_smem);  // [M][M]
  double2* px = u + (size_t)M * M;                  // [M][128]
  const int tid = threadIdx.x;
  for (int i = tid; i < M * M; i += 128) u[i] = U[i];
  const int p = blockIdx.x * 128 + tid;
  if (p < NN)
    for (int m = 0; m < M; ++m) {
      const float2 v = probe[(size_t)m * NN + p];
      px[m * 128 + tid] = make_double2(v.x, v.y);
    }
  __syncthreads();
  if (p >= NN) return;
  for (int k = 0; k < M; ++k) {
    double re = 0.0, im = 0.0;
    for (int m = 0; m < M; ++m) {
      const double2 w = u[m * M + k], x = px[m * 128 + tid];  // conj(w) * x
      re = fma(w.y, x.y, fma(w.x, x.x, re));
      im = fma(-w.y, x.x, fma(w.x, x.y, im));
    }
    probe[(size_t)k * NN + p] = make_float2((float)re, (float)im);
  }
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
static size_t round256(size_t b) { return (b + 255) & ~(size_t)255; }

static bool kz_on(const pty_constraints* c) { return c->kz_relax > 0.f && (c->kz_beta > 0.f || c->kz_alpha > 0.f); }

struct ConstrainLayout {
  size_t z, partial, U, lam, total;
};

static ConstrainLayout constrain_layout(const pty_geom* g, const pty_constraints* c) {
  ConstrainLayout L = {0, 0, 0, 0, 0};
  size_t off = 0;
  if (kz_on(c)) {
    L.z = off;
    off += round256(sizeof(float2) * (size_t)g->Nz * g->H * g->W);
  }
  if (c->probe_orthogonalize && g->M > 1) {
    const size_t NN = (size_t)g->N * g->N, chunks = (NN + kGramChunk - 1) / kGramChunk;
    L.partial = off;
    off += round256(sizeof(double2) * (size_t)g->M * (g->M + 1) / 2 * chunks);
    L.U = off;
    off += round256(sizeof(double2) * (size_t)g->M * g->M);
    L.lam = off;
    off += round256(sizeof(double) * g->M);
  }
  L.total = off;
  return L;
}

static int launched(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_error("%s launch failed: %s", what, cudaGetErrorString(e));
    return PTY_ECUDA;
  }
  note_launch();
  return PTY_OK;
}

static int check_constraints(const pty_geom* geom, const pty_constraints* c) {
  int rc = validate_geom(geom);
  if (rc) return rc;
  REQUIRE(c, "constraints are NULL");
  REQUIRE(c->phase_positivity >= 0.f && c->phase_positivity <= 1.f, "phase_positivity %g outside [0, 1]",
          c->phase_positivity);
  REQUIRE(c->rz_relax >= 0.f && c->rz_relax <= 1.f, "rz_relax %g outside [0, 1]", c->rz_relax);
  REQUIRE(c->rz_sigma >= 0.f && isfinite(c->rz_sigma), "rz_sigma %g must be finite and >= 0", c->rz_sigma);
  REQUIRE(c->kz_relax >= 0.f && c->kz_relax <= 1.f, "kz_relax %g outside [0, 1]", c->kz_relax);
  REQUIRE(c->kz_beta >= 0.f && isfinite(c->kz_beta) && c->kz_alpha >= 0.f && isfinite(c->kz_alpha),
          "kz_beta %g and kz_alpha %g must be finite and >= 0", c->kz_beta, c->kz_alpha);
  const bool blur = c->rz_sigma > 0.f && c->rz_relax > 0.f;
  REQUIRE(!blur || geom->Nz <= kMaxBlurSlices, "the depth blur supports Nz <= %d", kMaxBlurSlices);
  REQUIRE(!kz_on(c) || (geom->H <= kMaxLine && geom->W <= kMaxLine && geom->Nz <= kMaxBlurSlices),
          "the k_z filter supports H, W <= %d and Nz <= %d", kMaxLine, kMaxBlurSlices);
  REQUIRE(!c->probe_orthogonalize || geom->M <= kMaxOrthoModes, "orthogonalisation supports M <= %d modes",
          kMaxOrthoModes);
  return PTY_OK;
}

// One pass of line transforms.  C lines per tile, a power of two up to 8 while two CTAs fit an SM, at least
// one; as many CTAs as fit the chip at once take the tiles in turn.
template <int MODE, int KIND>
static int run_lines_of(KzArgs a, cudaStream_t st) {
  constexpr bool X = MODE == KZ_X_FWD || MODE == KZ_X_INV;
  const size_t tables = kz_table_bytes(a.line);
  a.C = KIND == KZ_DIRECT ? 1 : 8;
  while (a.C > 1 && tables + kz_lines_bytes(a.line, a.C) > kKzSmem / 2) a.C /= 2;
  const size_t smem = tables + kz_lines_bytes(a.line, a.C);
  a.tiles = X ? (long long)a.Nz * ((a.H + a.C - 1) / a.C) : (long long)((a.W + 7) / 8) * a.Nz * (8 / a.C);
  if (int rc = allow_smem(k_kz_lines<MODE, KIND>, smem, kKzSmem, "k_kz_lines")) return rc;
  long long per_sm = (long long)(kKzSmem / (smem + 1024));
  per_sm = per_sm < 1 ? 1 : per_sm > 4 ? 4 : per_sm;
  const long long grid = a.tiles < 152 * per_sm ? a.tiles : 152 * per_sm;
  k_kz_lines<MODE, KIND><<<(unsigned)grid, kKzThreads, smem, st>>>(a);
  return launched("k_kz_lines");
}
template <int MODE>
static int run_lines(const KzArgs& a, cudaStream_t st) {
  return a.line.kind == KZ_POW2 ? run_lines_of<MODE, KZ_POW2>(a, st)
       : a.line.kind == KZ_BLUESTEIN ? run_lines_of<MODE, KZ_BLUESTEIN>(a, st) : run_lines_of<MODE, KZ_DIRECT>(a, st);
}

static int run_kz_filter(const pty_geom* g, float* amp, float* phase, const float* dz, const pty_constraints* c,
                         float2* z, cudaStream_t st) {
  KzArgs a;
  memset(&a, 0, sizeof(a));
  a.z = z;
  a.amp = amp;
  a.phase = phase;
  a.relax = c->kz_relax;
  a.Nz = g->Nz;
  a.H = g->H;
  a.W = g->W;
  const KzLine lx = kz_line(g->W), ly = kz_line(g->H);
  int rc;
  a.line = lx;
  if ((rc = run_lines<KZ_X_FWD>(a, st))) return rc;
  a.line = ly;
  if ((rc = run_lines<KZ_Y_FWD>(a, st))) return rc;
  const size_t smem = kz_depth_bytes(g->Nz);
  if ((rc = allow_smem(k_kz_depth, smem, kz_depth_bytes(kMaxBlurSlices), "k_kz_depth"))) return rc;
  const int columns = g->H * (g->W < 8 ? g->W : 8);  // of a block
  k_kz_depth<<<dim3((columns + kDepthThreads - 1) / kDepthThreads, (g->W + 7) / 8), kDepthThreads, smem, st>>>(
      z, g->Nz, g->H, g->W, g->dx, dz, c->kz_beta, c->kz_alpha, lx, ly);
  if ((rc = launched("k_kz_depth"))) return rc;
  if ((rc = run_lines<KZ_Y_INV>(a, st))) return rc;
  a.line = lx;
  return run_lines<KZ_X_INV>(a, st);
}

static int run_orthogonalize(const pty_geom* g, float* probe, const ConstrainLayout& L, char* ws, cudaStream_t st) {
  const int M = g->M, NN = g->N * g->N;
  const int chunks = (NN + kGramChunk - 1) / kGramChunk;
  double2* partial = reinterpret_cast<double2*>(ws + L.partial);
  double2* U = reinterpret_cast<double2*>(ws + L.U);
  double* lam = reinterpret_cast<double*>(ws + L.lam);
  float2* P = reinterpret_cast<float2*>(probe);
  int rc;
  auto gram_smem = [](int m) { return sizeof(double2) * ((size_t)kGramTile * m + 256); };
  auto apply_smem = [](int m) { return sizeof(double2) * ((size_t)m * m + (size_t)m * 128); };
  if ((rc = allow_smem(k_gram, gram_smem(M), gram_smem(kMaxOrthoModes), "k_gram"))) return rc;
  k_gram<<<chunks, 256, gram_smem(M), st>>>(P, M, NN, partial);
  if ((rc = launched("k_gram"))) return rc;
  k_ortho_eig<<<1, 256, 0, st>>>(partial, M, chunks, U, lam);
  if ((rc = launched("k_ortho_eig"))) return rc;
  if ((rc = allow_smem(k_ortho_apply, apply_smem(M), apply_smem(kMaxOrthoModes), "k_ortho_apply"))) return rc;
  k_ortho_apply<<<(NN + 127) / 128, 128, apply_smem(M), st>>>(P, M, NN, U);
  return launched("k_ortho_apply");
}

}  // namespace pty

using namespace pty;

extern "C" {

size_t pty_constrain_workspace_size(const pty_geom* geom, const pty_constraints* c) {
  if (check_constraints(geom, c)) return 0;
  return constrain_layout(geom, c).total;
}

int pty_constrain(const pty_geom* geom, float* amp, float* phase, float* probe, const float* dz,
                  const pty_constraints* c, void* ws, size_t ws_bytes, void* stream) {
  int rc = check_constraints(geom, c);
  if (rc) return rc;
  const bool blur = c->rz_sigma > 0.f && c->rz_relax > 0.f;
  const bool kz = kz_on(c), ortho = c->probe_orthogonalize != 0;
  REQUIRE(!(blur || kz || c->phase_positivity > 0.f) || (amp && phase), "amp or phase is NULL");
  REQUIRE(!amp || (aligned(amp, 4) && aligned(phase, 4)), "float arrays must be 4-byte aligned");
  REQUIRE(!kz || dz, "the k_z filter needs the slice spacing dz (device pointer)");
  REQUIRE(!ortho || (probe && aligned(probe, 8)), "probe is NULL or not 8-byte aligned");
  const ConstrainLayout L = constrain_layout(geom, c);
  REQUIRE(ws_bytes >= L.total, "workspace of %zu bytes is smaller than the %zu needed", ws_bytes, L.total);
  REQUIRE(L.total == 0 || (ws && aligned(ws, 256)), "workspace is NULL or not 256-byte aligned");
  cudaStream_t st = (cudaStream_t)stream;
  char* w = static_cast<char*>(ws);
  if (ortho && geom->M > 1 && (rc = run_orthogonalize(geom, probe, L, w, st))) return rc;
  const size_t plane = (size_t)geom->H * geom->W, vol = (size_t)geom->Nz * plane;
  const int Ko = geom->obj_modes > 1 ? geom->obj_modes : 1;
  for (int n = 0; n < Ko; ++n) {  // each object mode is its own volume (the k_z workspace is reused)
    float* a = amp ? amp + n * vol : nullptr;
    float* p = phase ? phase + n * vol : nullptr;
    if (kz && (rc = run_kz_filter(geom, a, p, dz, c, reinterpret_cast<float2*>(w + L.z), st))) return rc;
    if (!blur && c->phase_positivity == 0.f) continue;
    const bool vec = plane % 4 == 0 && aligned(a, 16) && aligned(p, 16);
    const float sigma = blur ? c->rz_sigma : 0.f;
    rc = vec ? launch_constrain<4>(a, p, geom->Nz, plane, sigma, c->rz_relax, c->phase_positivity, st)
             : launch_constrain<1>(a, p, geom->Nz, plane, sigma, c->rz_relax, c->phase_positivity, st);
    if (rc || (rc = launched("k_constrain"))) return rc;
  }
  return PTY_OK;
}

}  // extern "C"
