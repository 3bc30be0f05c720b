// dftgemm.cuh -- the same pass with every per-slice 2D DFT computed as tensor-core GEMMs in split
// precision (pty_geom.fft_impl = PTY_FFT_SPLIT_BF16, _FP16 or SPLIT3_BF16), for N = 64 and 128.
//
// A 2D DFT of every wave of the batch is two row GEMMs over all waves at once: the first transforms
// along axis 1 and stores its result transposed per wave, the second transforms along the other axis.
// A complex row x times a complex matrix F is the real product [xr xi] [[Fr Fi]; [-Fi Fr]], and each
// real operand is cut into 16-bit pieces: with two pieces x F ~ xh Fh + xh Fl + xl Fh, every product
// accumulated in FP32 (k_dft_gemm).  The DFT
// matrices are permuted so that k-space comes out in exactly the digit order of the shared-memory
// FFT (kbin0 / kbin1), so patterns, loss, hooks and finalisers are shared with the FP32 path.
// Elementwise work between transforms runs as per-wave pointwise kernels (k_stage) that apply the same
// hooks to the wave and write the next transform's operand pieces.  FP32 FFTs remain for the probe
// spectra and the probe-gradient finaliser (once per call, not per slice).
//
// fp16 has a 5-bit exponent, so before each fp16 GEMM the batch is scaled by a power of two that
// puts its largest magnitude near 2^14; bf16 keeps FP32's exponent range and needs no scaling.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "gemm_ws.cuh"
#include "pipeline.cuh"

namespace pty {

// Split formats.  Each operand is cut into kPieces 16-bit pieces (piece 0 = the value rounded to 16
// bits, piece q = the remainder after pieces 0..q-1 rounded to 16 bits), and the product keeps the
// piece pairs (A piece p, B piece q) with p + q < kPieces, whose weight is above the format's rounding:
//   P = 1 (bf16, 2 pieces): h*h + h*l + l*h, 16 significant bits;
//   P = 2 (fp16, 2 pieces): h*h + h*l + l*h, 22 significant bits (after power-of-two scaling);
//   P = 3 (bf16, 3 pieces): h*h + h*m + h*l + m*h + m*m + l*h, 24 significant bits.
template <int P>
struct SplitType;
template <>
struct SplitType<PTY_FFT_SPLIT_BF16> {
  using H = __nv_bfloat16;
  static constexpr bool kScale = false;
  static constexpr int kPieces = 2;
  __device__ static H to(float x) { return __float2bfloat16_rn(x); }
  __device__ static float from(H h) { return __bfloat162float(h); }
};
template <>
struct SplitType<PTY_FFT_SPLIT_FP16> {
  using H = __half;
  static constexpr bool kScale = true;
  static constexpr int kPieces = 2;
  __device__ static H to(float x) { return __float2half_rn(x); }
  __device__ static float from(H h) { return __half2float(h); }
};
template <>
struct SplitType<PTY_FFT_SPLIT3_BF16> {
  using H = __nv_bfloat16;
  static constexpr bool kScale = false;
  static constexpr int kPieces = 3;
  __device__ static H to(float x) { return __float2bfloat16_rn(x); }
  __device__ static float from(H h) { return __bfloat162float(h); }
};

// Operand image: the rows of the batch as kPieces x 2N / 64 blocks of 64 (piece, real or imaginary part, 64
// positions), each a tile image (gemm_ws.cuh), so the 128 rows of a tile are one bulk copy a block.
//
// store_pieces: eight lanes (lane % 8 = i) hold x[e] of row r0 + e at position c8 + i of one part, e < 8; lane i
// stores row r0 + i, positions c8 .. c8 + 7 of every piece.
template <int N, int P>
__device__ __forceinline__ void store_pieces(typename SplitType<P>::H* out, int rows, int r0, int c8, int part,
                                             float (&x)[8], int lane) {
  using S = SplitType<P>;
  const int r = r0 + (lane & 7);
  typename S::H* o = out + (size_t)(part * (N / 64) + c8 / 64) * rows * 64 + (size_t)(r >> 3) * 512 + (c8 & 63) * 8 + (r & 7) * 8;
#pragma unroll
  for (int q = 0; q < S::kPieces; ++q) {
    union {
      uint32_t r[4];
      typename S::H h[8];
    } p;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      p.h[e] = S::to(x[e]);
      x[e] -= S::from(p.h[e]);  // exact: each piece removes the leading bits
    }
    transpose8(p.r, lane);
    *reinterpret_cast<uint4*>(o + (size_t)q * (2 * N / 64) * rows * 64) = make_uint4(p.r[0], p.r[1], p.r[2], p.r[3]);
  }
}

// The operand from complex rows X[rows][N] times the fp16 scale: eight lanes take the same 8 rows at 8 positions.
template <int N, int P>
__global__ void __launch_bounds__(256) k_split(const float2* __restrict__ X, typename SplitType<P>::H* __restrict__ Xs,
                                               int rows, const float* scale) {
  const size_t n = (size_t)(rows / 8) * N;  // a multiple of 32
  const float sc = *scale;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int r0 = 8 * (int)(i / N), c = (int)(i % N);
    float re[8], im[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float2 v = X[(size_t)(r0 + e) * N + c];
      re[e] = v.x * sc;
      im[e] = v.y * sc;
    }
    store_pieces<N, P>(Xs, rows, r0, c & ~7, 0, re, threadIdx.x & 31);
    store_pieces<N, P>(Xs, rows, r0, c & ~7, 1, im, threadIdx.x & 31);
  }
}

// ---------------------------------------------------------------------------------------------
// k_dft_gemm: rows x split DFT matrix
// ---------------------------------------------------------------------------------------------
// A CTA keeps 64 output positions' part of the matrix in shared memory and streams the operand's rows past it.  Per
// 64 of K and piece the resident block has 192 rows, -Fi, Fr and Fi of the 64 positions: rows 64..191 are [Fr Fi], what
// a real part multiplies, and rows 0..127 are [-Fi Fr], what an imaginary part does, so both are one 128 x 128 MMA
// operand and the matrix takes 147 KB (three pieces, N = 128), which leaves a ring of five 16 KB stages for the rows.
// Streaming matrix and rows together would move 768 KB a 128 x 256 tile from L2 where this moves 384 KB: L2 -> SM
// copies bound it.  K runs over (part, 64 positions).  Of every such block the tensor cores sum the h*h products into a
// fresh TMEM region (two in turn), and of a whole tile the smaller piece pairs into another (two in turn); each
// region is added to FP32 registers with round-to-nearest adds.  The small pairs' sum is 2^-8 of the result, so what
// their accumulation rounds does not show; h*h, whose would, keeps to 64 of K.  All pairs of a block in one region
// made an intensity error 1.15 times larger; a region for every pair of a block made 24 promotions a tile, whose
// regions the MMAs waited for while the warps promoted and stored (92 us a GEMM).
//   warps 0-7  promote and store (warp w: rows 32 (w % 4) .., positions 32 (w / 4) .. of the tile)
//   warp 8     one thread: bulk copies;   warp 9  one thread: MMAs
// Waits are bounded as in k_gemm_ws.
// The GEMMs of the three-piece format on 49152 rows of N = 128: 200 us each with both operands gathered by cp.async
// and one block in flight, 50 here (HBM traffic alone: 20-25).
constexpr int DFT_THREADS = 320;
template <int N, int P>
struct DftShape {
  static constexpr int PC = SplitType<P>::kPieces, KB = N / 64, PARTS = N / 64;  // K blocks of a part; column parts
  static constexpr int B_BLOCK = 192 * 128, B_BYTES = KB * PC * B_BLOCK, STAGE = 128 * 128;
  static constexpr int STAGES = (229376 - B_BYTES) / STAGE < 8 ? (229376 - B_BYTES) / STAGE : 8;
  static constexpr size_t SMEM = (size_t)B_BYTES + STAGES * STAGE + 1024 + 256;
  static_assert(8 * (2 * STAGES + 9) + 8 <= 256, "barriers, TMEM slot, abort flag");
  static constexpr size_t TABLE = (size_t)PARTS * B_BYTES / 2;  // elements of one matrix
};

// Split DFT matrices: [mat][column part][K block][piece] resident blocks.  mat 0: axis 1 forward (natural c ->
// position p1); 1: axis 0 forward (r -> p0); 2: axis 0 inverse (p0 -> r); 3: axis 1 inverse (p1 -> c).
template <int N, int P>
__global__ void k_init_dft_tables(typename SplitType<P>::H* Bt) {
  using S = SplitType<P>;
  using D = DftShape<N, P>;
  const size_t n = 4 * D::TABLE;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const int e = (int)(i % (D::B_BLOCK / 2));
    const int blk = (int)(i / (D::B_BLOCK / 2));
    const int piece = blk % D::PC, kb = blk / D::PC % D::KB, np = blk / D::PC / D::KB % D::PARTS, mat = (int)(i / D::TABLE);
    const int row = 8 * (e / 512) + (e % 64) / 8, k = 8 * (e % 512 / 64) + e % 8;  // image_index inverted
    const int qin = 64 * kb + k, jout = 64 * np + row % 64;
    int a, b;
    double sign;
    switch (mat) {
      case 0: a = qin; b = kbin1<N>(jout); sign = -1.0; break;
      case 1: a = qin; b = kbin0<N>(jout); sign = -1.0; break;
      case 2: a = kbin0<N>(qin); b = jout; sign = 1.0; break;
      default: a = kbin1<N>(qin); b = jout; sign = 1.0; break;
    }
    double sn, cs;
    sincospi(2.0 * (double)((a * b) % N) / N, &sn, &cs);
    double g = row < 64 ? -sign * sn : row < 128 ? cs : sign * sn;
    // pieces from the FP64 value (the FP32 rounding of g would cap the table at 24 bits)
    typename S::H h = S::to((float)g);
    for (int r = 0; r < piece; ++r) {
      g -= (double)S::from(h);
      h = S::to((float)g);
    }
    Bt[i] = h;
  }
}

// Epilogues: a warp's 32 rows (lane: one row; all valid) x 32 output positions from c0.
// Second GEMM (or fp16): complex FP32, row by row or, TRANSPOSE, row a of wave w at position (w, c, a).
template <int N, bool TRANSPOSE>
struct DftEpilogue {
  float2* out;
  const float* scale;  // fp16: undo the input scaling
  __device__ __forceinline__ void operator()(int row0, int lane, int c0, float (&re)[32], float (&im)[32]) const {
    const int row = row0 + lane;
    if (scale) {
      const float s = 1.0f / *scale;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        re[i] *= s;
        im[i] *= s;
      }
    }
    if constexpr (TRANSPOSE) {
      float2* o = out + ((size_t)(row / N) * N + c0) * N + row % N;
#pragma unroll
      for (int i = 0; i < 32; ++i) o[(size_t)i * N] = make_float2(re[i], im[i]);
    } else {
      float4* o = reinterpret_cast<float4*>(out + (size_t)row * N + c0);
#pragma unroll
      for (int i = 0; i < 32; i += 2) o[i / 2] = make_float4(re[i], im[i], re[i + 1], im[i + 1]);
    }
  }
};
// First GEMM, unscaled formats: the result, transposed per wave, goes straight into the pieces of the
// second GEMM's operand.
template <int N, int P>
struct DftSplitEpilogue {
  typename SplitType<P>::H* out;
  int rows;
  __device__ __forceinline__ void operator()(int row0, int lane, int c0, float (&re)[32], float (&im)[32]) const {
    const int a8 = row0 % N + (lane & 24), r0 = row0 / N * N + c0;
#pragma unroll
    for (int g = 0; g < 32; g += 8) {
      float x[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = re[g + e];
      store_pieces<N, P>(out, rows, r0 + g, a8, 0, x, lane);
#pragma unroll
      for (int e = 0; e < 8; ++e) x[e] = im[g + e];
      store_pieces<N, P>(out, rows, r0 + g, a8, 1, x, lane);
    }
  }
};

template <int N, int P, class Epi>
__global__ void __launch_bounds__(DFT_THREADS, 1)
    k_dft_gemm(const typename SplitType<P>::H* __restrict__ A, int rows, const typename SplitType<P>::H* __restrict__ Bt,
               Epi epi, int* status, long spin) {
  using D = DftShape<N, P>;
  constexpr int ST = D::STAGES, KBLOCKS = 2 * D::KB;
  extern __shared__ __align__(1024) unsigned char ws_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)ws_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* ring = base + D::B_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(ring + ST * D::STAGE);
  // barriers: [ST] stage full, [ST] stage free, [4] region done (two of h*h, two of small pairs), [4] region free, matrix landed
  const uint32_t full = tc_smem_u32(bars), empty = full + 8 * ST, done = empty + 8 * ST, rfree = done + 32, matrix = rfree + 32;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2 * ST + 9);
  volatile int* abort = reinterpret_cast<volatile int*>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    auto init = [](uint32_t bar, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(n)); };
    for (int i = 0; i < ST; ++i) {
      init(full + 8 * i, 1);
      init(empty + 8 * i, 1);
    }
    for (int i = 0; i < 4; ++i) {
      init(done + 8 * i, 1);
      init(rfree + 8 * i, 8);
    }
    init(matrix, 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  // the grid is a multiple of PARTS: CTAs side by side take the parts of the same rows
  const int part = blockIdx.x % D::PARTS, tile0 = blockIdx.x / D::PARTS, step = gridDim.x / D::PARTS;
  const int tiles = (rows + 127) / 128;
  auto fail = [&]() {
    *abort = 1;
    atomicOr(status, PTY_ETIMEOUT);
  };

  if (warp < 8) {
    const int sub = warp & 3, half = warp >> 2;
    const uint32_t col = ((uint32_t)(32 * sub) << 16) + 32 * half;
    int q = 0, it = 0;
    bool ok = true;
    for (int t = tile0; t < tiles && ok; t += step, ++it) {
      float re[32], im[32];
#pragma unroll
      for (int j = 0; j < 32; ++j) re[j] = im[j] = 0.f;
      for (int b = 0; b <= KBLOCKS; ++b) {  // the h*h blocks, then the small pairs
        const int r = b < KBLOCKS ? q & 1 : 2 + (it & 1), use = b < KBLOCKS ? q >> 1 : it >> 1;
        ok = __all_sync(0xffffffffu, ws_wait(done + 8 * r, (uint32_t)use & 1, spin, abort)) != 0;
        if (!ok) {
          if (lane == 0) fail();
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t region = tmem + 128 * r + col;
        tc_ld_add<32>(region, re);
        tc_ld_add<32>(region + 64, im);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) ws_arrive(rfree + 8 * r);
        if (b < KBLOCKS) ++q;
      }
      if (!ok) break;
      const int row0 = t * 128 + 32 * sub;
      if (row0 < rows) epi(row0, lane, 64 * part + 32 * half, re, im);  // rows: a multiple of 64
    }
  } else if (warp == 8) {
    if (lane == 0) {
      const typename SplitType<P>::H* bp = Bt + (size_t)part * (D::B_BYTES / 2);
      ws_expect(matrix, D::B_BYTES);
      for (int i = 0; i < D::KB * D::PC; ++i)
        ws_bulk(tc_smem_u32(base + i * D::B_BLOCK), bp + (size_t)i * (D::B_BLOCK / 2), D::B_BLOCK, matrix);
      int n = 0;
      bool ok = true;
      for (int t = tile0; t < tiles && ok; t += step) {
        const uint32_t bytes = (uint32_t)min(128, rows - t * 128) * 128;
        const typename SplitType<P>::H* ap = A + (size_t)t * 128 * 64;
        for (int i = 0; i < KBLOCKS * D::PC; ++i, ++n) {
          const int s = n % ST;
          if (n >= ST && !ws_wait(empty + 8 * s, (uint32_t)(n / ST - 1) & 1, spin, abort)) {
            fail();
            ok = false;
            break;
          }
          ws_expect(full + 8 * s, bytes);
          ws_bulk(tc_smem_u32(ring + s * D::STAGE), ap + (size_t)((D::PC - 1 - i % D::PC) * KBLOCKS + i / D::PC) * rows * 64, bytes, full + 8 * s);
        }
      }
      // every copy has landed before the CTA can end (only after an abort is there one to wait for)
      tc_wait(matrix, 0);
      for (int i = n > ST ? n - ST : 0; i < n; ++i) tc_wait(full + 8 * (i % ST), (uint32_t)(i / ST) & 1);
    }
  } else if (lane == 0) {
    constexpr uint32_t id = tc_idesc<typename SplitType<P>::H, 128>();
    int n = 0, q = 0, it = 0;
    bool ok = ws_wait(matrix, 0, spin, abort);
    if (!ok) fail();
    for (int t = tile0; t < tiles && ok; t += step, ++it) {
      const int small = 2 + (it & 1);
      uint32_t accum = 0u;  // of the small pairs' region
      ok = it < 2 || ws_wait(rfree + 8 * small, (uint32_t)((it >> 1) - 1) & 1, spin, abort);
      for (int pk = 0; pk < KBLOCKS && ok; ++pk) {
        // a real part's block meets [Fr Fi] (8 KB in), an imaginary part's [-Fi Fr]
        const uint32_t sb0 = tc_smem_u32(base) + pk % D::KB * D::PC * D::B_BLOCK + (pk < D::KB ? 8192 : 0);
#pragma unroll
        for (int pa = D::PC - 1; pa >= 0; --pa, ++n) {
          const int s = n % ST;
          ok = ok && ws_wait(full + 8 * s, (uint32_t)(n / ST) & 1, spin, abort) &&
               (pa > 0 || q < 2 || ws_wait(rfree + 8 * (q & 1), (uint32_t)((q >> 1) - 1) & 1, spin, abort));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t sa = tc_smem_u32(ring + s * D::STAGE);
#pragma unroll
          for (int pb = 0; pb < D::PC - pa; ++pb) {
            const bool hh = pa == 0 && pb == 0;
            const uint32_t d = tmem + 128 * (hh ? q & 1 : small);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const uint64_t da = tc_desc(sa + k * 256), db = tc_desc(sb0 + pb * D::B_BLOCK + k * 256);
              asm volatile(
                  "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                  "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
                  "l"(da), "l"(db), "r"(id), "r"(hh ? (uint32_t)(k > 0) : accum));
              if (!hh) accum = 1u;
            }
            if (hh) ws_commit(done + 8 * (q & 1));
          }
          if (pa == 0) ++q;
          ws_commit(empty + 8 * s);
        }
      }
      if (!ok) {
        fail();
        break;
      }
      ws_commit(done + 8 * small);
    }
    // the last MMAs are complete before the tensor memory is released: every stage's are committed to its barrier
    if (n > 0) tc_wait(empty + 8 * ((n - 1) % ST), (uint32_t)((n - 1) / ST) & 1);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// fp16 scaling: largest |re|, |im| of the batch, then the power of two that maps it near 2^14.
static __global__ void k_absmax(const float* __restrict__ x, size_t n, unsigned* out) {
  float m = 0.f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf(x[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));  // non-negative floats order as ints
}
static __global__ void k_pow2_scale(const unsigned* amax, float* scale) {
  const float m = __uint_as_float(*amax);
  *scale = (m > 0.f && isfinite(m)) ? exp2f(14.0f - ceilf(log2f(m))) : 1.0f;
}

// ---------------------------------------------------------------------------------------------
// Pointwise stages on a wave in global memory (one CTA of 256 threads per wave)
// ---------------------------------------------------------------------------------------------
enum GemmStage { GS_SHIFT, GS_TRANS, GS_PROP, GS_FAR, GS_FARGRAD, GS_ADJTRANS, GS_ADJPROP, GS_PROBE };

struct StageArgs {
  FwdArgs f;     // geometry, parameters, checkpoint / far-field outputs (forward stages)
  AdjArgs a;     // adjoint inputs and accumulators
  float2* wave;  // [waves][N*N] current wave (natural or k-space layout)
  void* pieces;  // unscaled formats: the next transform's operand, written instead of the wave
  int sl;        // slice
};

template <int N>
__host__ __device__ constexpr size_t stage_smem_bytes() {
  return sizeof(float2) * 4 * N + sizeof(float) * 6 * N + sizeof(double) * 5 * 8;
}

// A thread holds 8 consecutive rows of one column, so the 8 x 8 transpose of eight lanes gives each a row's 8
// columns: one 16-byte store per piece and part, 512 contiguous bytes a warp, in the GEMM's tile image.  Writing the
// pieces here replaces the FP32 wave and a kernel that split it.
template <int N, int ST, int P>
__global__ void __launch_bounds__(256) k_stage(StageArgs g) {
  constexpr int T = 256, NN = N * N, STEP = T / N;
  extern __shared__ __align__(16) float2 sm[];
  float2* t0p = sm;  // forward: ra0 / ra1 / pm0 / pm1; adjoint: cm0 / cm1 / cr0 / cr1
  float2* t1p = t0p + N;
  float2* t2p = t1p + N;
  float2* t3p = t2p + N;
  float* e0 = reinterpret_cast<float*>(t3p + N);
  float* e1 = e0 + N;
  float* c0 = e1 + N;
  float* c1 = c0 + N;
  float* f0 = c1 + N;
  float* f1 = f0 + N;
  double* red = reinterpret_cast<double*>(f1 + N);
  const FwdArgs& a = g.f;
  const int tid = threadIdx.x, bm = blockIdx.x;
  const int b = bm / (a.M * a.Ko), m = (bm / a.Ko) % a.M;  // waves: (position, probe mode, object mode)
  const int j = checked_index(a.idx, b, a.Ntot, a.status);
  int i0, i1;
  float d0, d1;
  patch_corner<N>(a.pos, j, a.H, a.W, &i0, &i1, &d0, &d1, a.status);
  const Pair* wc = a.wc + (size_t)b * kWaveConsts;
  constexpr bool kAdj = ST >= GS_FARGRAD;
  if (kAdj) {
    adj_tables<N>(t0p, t1p, t2p, t3p, e0, e1, c0, c1, f0, f1, d0, d1, wc);
  } else {
    fwd_tables<N>(t0p, t1p, t2p, t3p, d0, d1, wc);
  }
  __syncthreads();
  const size_t plane = (size_t)a.H * a.W, patch = (size_t)(bm % a.Ko) * a.Nz * plane + (size_t)i0 * a.W + i1;
  float2* X = g.wave + (size_t)bm * NN;
  const int sl = g.sl;
  float acc[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
  constexpr int U = 8;
  // natural stages: thread owns column tid % N, 8 rows from 8 (tid / N + STEP i); k-space stages: row p0 = tid % N,
  // 8 columns p1 (the buffer is stored p1 * N + p0)
  const int lo = tid % N, hi0 = tid / N;
  for (int i = 0; i < N / (STEP * U); ++i) {
    float2 v[U];
    const int h = (hi0 + i * STEP) * U;
    if constexpr (ST != GS_SHIFT && ST != GS_FARGRAD) {  // those two replace the wave
#pragma unroll
      for (int u = 0; u < U; ++u) v[u] = X[(size_t)(h + u) * N + lo];
    }
    if constexpr (ST == GS_SHIFT) {
      ShiftLoad<N> hk{a.Phat + (size_t)m * NN, t0p, t1p};
      hk.template operator()<U>(lo, 0, h, 1, v);
    } else if constexpr (ST == GS_TRANS) {
      TransLoad<N> hk{a.T + sl * plane + patch, a.W, a.ckpt ? a.ckpt + ((size_t)bm * a.Nz + sl) * NN : nullptr};
      hk.template operator()<U>(h, 1, lo, 0, v);
    } else if constexpr (ST == GS_PROP) {
      PropStore<N> hk{t2p, t3p, a.vhat ? a.vhat + ((size_t)bm * (a.Nz - 1) + sl) * NN : nullptr};
      hk.template operator()<U>(lo, 0, h, 1, v);
    } else if constexpr (ST == GS_FAR) {
      FarStore<N> hk{a.Psi ? a.Psi + (size_t)bm * NN : nullptr, a.Imode + (size_t)bm * NN};
      hk.template operator()<U>(lo, 0, h, 1, v);
    } else if constexpr (ST == GS_FARGRAD) {
      FarGradLoad<N> hk{g.a.u + (size_t)b * NN, g.a.Psi + (size_t)bm * NN,
                        g.a.u_scaled ? 1.0f : (float)(2.0 * g.a.scal[0] / N)};
      hk.template operator()<U>(lo, 0, h, 1, v);
    } else if constexpr (ST == GS_ADJTRANS) {
      const bool obj = (g.a.grad_mask & (PTY_GRAD_AMP | PTY_GRAD_PHASE)) != 0;
      AdjTransLoad<N> hk{a.T + sl * plane + patch, g.a.gT + sl * plane + patch,
                         obj ? g.a.ckpt + ((size_t)bm * a.Nz + sl) * NN : nullptr, a.W};
      hk.template operator()<U>(h, 1, lo, 0, v);
    } else if constexpr (ST == GS_ADJPROP) {
      AdjPropStore<N> hk{t0p, t1p, g.a.vhat ? g.a.vhat + ((size_t)bm * (a.Nz - 1) + sl - 1) * NN : nullptr,
                         e0, e1, c0, c1, acc[4], acc[2], acc[3]};
      hk.template operator()<U>(lo, 0, h, 1, v);
    } else {
      ProbeStore<N> hk{(g.a.grad_mask & PTY_GRAD_PROBE) ? g.a.gPhat + (size_t)m * NN : nullptr,
                       a.Phat + (size_t)m * NN, t2p, t3p, f0, f1, (g.a.grad_mask & PTY_GRAD_POS) != 0, acc[0], acc[1]};
      hk.template operator()<U>(lo, 0, h, 1, v);
    }
    if constexpr (ST != GS_FAR && ST != GS_PROBE) {
      if constexpr (SplitType<P>::kScale) {
#pragma unroll
        for (int u = 0; u < U; ++u) X[(size_t)(h + u) * N + lo] = v[u];
      } else {
        typename SplitType<P>::H* out = reinterpret_cast<typename SplitType<P>::H*>(g.pieces);
        const int rows = (int)gridDim.x * N, r0 = bm * N + h;
        float x[8];
#pragma unroll
        for (int part = 0; part < 2; ++part) {
#pragma unroll
          for (int u = 0; u < U; ++u) x[u] = part ? v[u].y : v[u].x;
          store_pieces<N, P>(out, rows, r0, lo & ~7, part, x, tid & 31);
        }
      }
    }
  }
  if constexpr (ST == GS_ADJPROP || ST == GS_PROBE) {  // FP64 CTA sums into the per-wave partials
    double s5[5] = {acc[0], acc[1], acc[2], acc[3], acc[4]};
#pragma unroll
    for (int q = 0; q < 5; ++q)
      for (int o = 16; o > 0; o >>= 1) s5[q] += __shfl_down_sync(0xffffffffu, s5[q], o);
    if ((tid & 31) == 0) {
#pragma unroll
      for (int q = 0; q < 5; ++q) red[5 * (tid >> 5) + q] = s5[q];
    }
    __syncthreads();
    if (tid < 5) {
      double t = 0.0;
      for (int w = 0; w < T / 32; ++w) t += red[5 * w + tid];
      g.a.spart[(size_t)bm * 5 + tid] += t;
    }
  }
}

}  // namespace pty

namespace pty {

// Split DFT matrices of one device, built on the device on first use (one synchronous init per
// device and precision).
template <int N, int P>
__device__ __align__(256) typename SplitType<P>::H g_dft_tables[4 * DftShape<N, P>::TABLE];

template <int N, int P>
const typename SplitType<P>::H* dft_tables(cudaStream_t st) {
  static void* addr[256] = {nullptr};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 256) return nullptr;
  if (!addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_dft_tables<N, P>) != cudaSuccess || !p) return nullptr;
    k_init_dft_tables<N, P><<<152 * 4, 256, 0, st>>>(reinterpret_cast<typename SplitType<P>::H*>(p));
    if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) return nullptr;
    note_launch();
    addr[dev] = p;
  }
  return reinterpret_cast<const typename SplitType<P>::H*>(addr[dev]);
}

// One pass with split-precision DFT-GEMMs in place of the shared-memory FFT (checkpoint every slice).
template <int N, int P>
struct GemmPass {
  using S = SplitType<P>;
  using H = typename S::H;
  static constexpr int NN = N * N;
  Pass<N> base;
  const Problem& pb;
  const Workspace& ws;
  cudaStream_t st;
  const H* tables = nullptr;

  explicit GemmPass(const Problem& p) : base(p), pb(p), ws(p.ws), st(p.stream) {}

  // fp16 batch scale of `src` into ws.gscal (returns the device scale pointer)
  int fp16_scale(const float2* src, const float** sc) {
    const int rows = pb.B * pb.M * pb.Ko * N;
    unsigned* amax = reinterpret_cast<unsigned*>(ws.gscal);
    float* scale = reinterpret_cast<float*>(ws.gscal) + 1;
    if (cudaMemsetAsync(amax, 0, sizeof(unsigned), st) != cudaSuccess) return base.memset_failed();
    k_absmax<<<152 * 4, 256, 0, st>>>(reinterpret_cast<const float*>(src), (size_t)rows * N * 2, amax);
    PTY_LAUNCH_CHECK("k_absmax", -1);
    k_pow2_scale<<<1, 1, 0, st>>>(amax, scale);
    PTY_LAUNCH_CHECK("k_pow2_scale", -1);
    *sc = scale;
    return PTY_OK;
  }
  template <class Epi>
  int gemm(int mat, const void* operand, const Epi& epi) {
    using D = DftShape<N, P>;
    const int rows = pb.B * pb.M * pb.Ko * N, items = (rows + 127) / 128 * D::PARTS;
    auto kern = k_dft_gemm<N, P, Epi>;
    static bool ready[256] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess && (dev < 0 || dev >= 256)) e = cudaErrorInvalidDevice;
    if (e == cudaSuccess && !__atomic_load_n(&ready[dev], __ATOMIC_ACQUIRE)) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)D::SMEM);
      if (e == cudaSuccess) __atomic_store_n(&ready[dev], true, __ATOMIC_RELEASE);
    }
    if (e == cudaSuccess) {
      kern<<<items < 152 ? items : 152, DFT_THREADS, D::SMEM, st>>>(reinterpret_cast<const H*>(operand), rows,
                                                                  tables + (size_t)mat * D::TABLE, epi, ws.status,
                                                                  stage_wait_limit());
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
      set_error("k_dft_gemm launch failed: %s", cudaGetErrorString(e));
      return PTY_ECUDA;
    }
    PTY_LAUNCH_CHECK("k_dft_gemm", -1);
    return PTY_OK;
  }
  int split(const float2* src, void* dst, const float* sc) {
    const int rows = pb.B * pb.M * pb.Ko * N;
    const size_t n = (size_t)(rows / 8) * N;
    const unsigned blocks = (unsigned)((n + 255) / 256 < 152 * 16 ? (n + 255) / 256 : 152 * 16);
    k_split<N, P><<<blocks, 256, 0, st>>>(src, reinterpret_cast<H*>(dst), rows, sc);
    PTY_LAUNCH_CHECK("k_split", -1);
    return PTY_OK;
  }
  // The stage before has left the pieces of the wave in pieces0 (bf16 formats: the first GEMM writes the pieces of the
  // second's operand) or the wave in FP32 (fp16: scaled and split before each GEMM).
  int transform(int mat_a, int mat_b) {
    int rc;
    const float* sc = nullptr;
    if constexpr (S::kScale) {
      if ((rc = fp16_scale(ws.wave, &sc))) return rc;
      if ((rc = split(ws.wave, ws.pieces0, sc))) return rc;
      if ((rc = gemm(mat_a, ws.pieces0, DftEpilogue<N, true>{ws.tmp, sc}))) return rc;
      if ((rc = fp16_scale(ws.tmp, &sc))) return rc;
      if ((rc = split(ws.tmp, ws.pieces1, sc))) return rc;
    } else {
      if ((rc = gemm(mat_a, ws.pieces0, DftSplitEpilogue<N, P>{reinterpret_cast<H*>(ws.pieces1), pb.B * pb.M * pb.Ko * N}))) return rc;
    }
    return gemm(mat_b, ws.pieces1, DftEpilogue<N, false>{ws.wave, sc});
  }
  // natural [w][r][c] -> k-space [w][p1][p0] and back
  int dft2() { return transform(0, 1); }
  int idft2() { return transform(2, 3); }
  template <int ST>
  int stage(const FwdArgs& fa, const AdjArgs& aa, int sl, int prof) {
    StageArgs g{fa, aa, ws.wave, ws.pieces0, sl};
    k_stage<N, ST, P><<<pb.B * pb.M * pb.Ko, 256, stage_smem_bytes<N>(), st>>>(g);
    PTY_LAUNCH_CHECK("k_stage", prof);
    return PTY_OK;
  }

  int forward(const float* I_meas) {
    tables = dft_tables<N, P>(st);
    if (!tables) {
      set_error("split DFT tables could not be set up: %s", cudaGetErrorString(cudaGetLastError()));
      return PTY_ECUDA;
    }
    int rc = base.forward_begin();
    if (rc || pb.B == 0) return rc;
    const FwdArgs fa = base.fwd_args_saved();
    const AdjArgs aa = base.adj_args();
    const int Nz = pb.Nz;
#define PTY_TRY(x)         \
  do {                     \
    int r_ = (x);          \
    if (r_) return r_;     \
  } while (0)
    PTY_TRY(stage<GS_SHIFT>(fa, aa, 0, -1));
    PTY_TRY(idft2());
    for (int sl = 0; sl < Nz; ++sl) {
      PTY_TRY(stage<GS_TRANS>(fa, aa, sl, -1));
      PTY_TRY(dft2());
      if (sl + 1 < Nz) {
        PTY_TRY(stage<GS_PROP>(fa, aa, sl, -1));
        PTY_TRY(idft2());
      } else {
        PTY_TRY(stage<GS_FAR>(fa, aa, sl, 2));
      }
    }
    return base.loss_phase(I_meas);
  }

  int adjoint() {
    PTY_TRY(base.adjoint_begin());
    if (pb.B > 0) {
      AdjArgs aa = base.adj_args();
      aa.ckpt = ws.ckpt;
      aa.vhat = base.want_prop ? ws.vhat : nullptr;
      const FwdArgs fa = base.fwd_args();
      const int Nz = pb.Nz;
      PTY_TRY(stage<GS_FARGRAD>(fa, aa, Nz - 1, -1));
      PTY_TRY(idft2());
      for (int sl = Nz - 1; sl >= 0; --sl) {
        PTY_TRY(stage<GS_ADJTRANS>(fa, aa, sl, -1));
        if (sl > 0) {
          PTY_TRY(dft2());
          PTY_TRY(stage<GS_ADJPROP>(fa, aa, sl, -1));
          PTY_TRY(idft2());
        } else if (base.want_probe || (pb.grad_mask & PTY_GRAD_POS)) {
          PTY_TRY(dft2());
          PTY_TRY(stage<GS_PROBE>(fa, aa, sl, -1));
        }
      }
      prof_mark(5, st);
    }
    return base.finalize();
#undef PTY_TRY
  }
};

template <int N, int P>
int run_pipeline_gemm(const Problem& pb) {
  GemmPass<N, P> ps(pb);
  int rc = ps.base.set_attributes();
  if (rc) return rc;
  switch (pb.mode) {
    case MODE_FORWARD:
    case MODE_FORWARD_SAVE:
      return ps.forward(nullptr);
    case MODE_GRAD:
      rc = ps.forward(pb.I_meas);
      if (rc) return rc;
      if (pb.B == 0 && pb.loss_out) {
        if (cudaMemsetAsync(pb.loss_out, 0, sizeof(double), pb.stream) != cudaSuccess) return ps.base.memset_failed();
      }
      return ps.adjoint();
    case MODE_STATS:
      if (pb.loss == PTY_LOSS_POISSON) return ps.base.stats();  // the measured patterns only
      rc = ps.forward(pb.I_meas);
      if (rc) return rc;
      return ps.base.stats_write(pb.B * loss_parts<N>());
    case MODE_BACKWARD:
      rc = ps.base.external_dldi(pb.dldi);
      if (rc) return rc;
      ps.tables = dft_tables<N, P>(pb.stream);
      if (!ps.tables) {
        set_error("split DFT tables could not be set up");
        return PTY_ECUDA;
      }
      return ps.adjoint();
    default:
      set_error("unknown pass mode %d", pb.mode);
      return PTY_EINVAL;
  }
}

}  // namespace pty
