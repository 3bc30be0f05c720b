// gemm_ws.cuh -- C = A * B^T on the 5th-generation tensor cores with a role for every warp, for the learned
// initialiser's layers.  K in blocks of 64, each summed by the tensor cores into a fresh TMEM region and added to
// FP32 registers with round-to-nearest adds, in K order.
//
// One CTA per SM, which takes the 128 x BN tiles blockIdx.x, + gridDim.x, ...:
//   warps 0-7   promote: read a finished block's TMEM region, add it to their registers, run the epilogue;
//   2 or 4 warps gather the A tile with cp.async (im2col rows: 8 rows x 64 bytes a warp instruction), two blocks
//               behind their own loads when they announce a stage; a row is a pointer and a mask of its
//               valid taps, decoded once per tile, so a chunk costs a bit test and an add.  One thread also
//               issues the bulk copies of operands that are kept as tile images (B always; A when it is one);
//   last warp   one thread issues the MMAs.
// Stages pass between them on mbarriers, so the loads of later blocks and tiles, the MMAs and the promotion
// overlap; where eight warps do all three in turn, one block ahead, with two barriers a block, the
// 65536 x 256 x 3456 layer takes 5500 clocks a block where its MMAs need 512 (507 us; 232 here).
//
// Tile images.  An operand of R rows (a multiple of 8) is stored by K block: block kb holds, for every 8 rows, the
// eight 8 x 8 core matrices along K (128 bytes each), which is the tensor core's canonical K-major layout without
// swizzle, so the rows of one tile and block are one contiguous run and one bulk copy.
//
// Every wait is bounded and watches the CTA's abort flag: a role whose wait runs out sets the flag and PTY_ETIMEOUT,
// every role leaves its loop, what is in flight (copies, MMAs) is waited for with the full limit, and the
// tensor memory is released.
#pragma once
#include "gemm_tc.cuh"

namespace pty {

constexpr int WS_PROMOTE = 256;
constexpr int kWsBlock = 64;  // K per block and tile image

// Element (row, k) of a tile-image operand of `rows` rows, in elements.
__host__ __device__ __forceinline__ size_t image_index(int row, size_t k, int rows) {
  return (k / 64) * (size_t)rows * 64 + (size_t)(row >> 3) * 512 + ((k & 63) >> 3) * 64 + (row & 7) * 8 + (k & 7);
}
inline int image_rows(int rows) { return (rows + 7) / 8 * 8; }

struct ImageOperand {
  const __nv_bfloat16* p;
  int rows;  // a multiple of 8
};

// KS: MMAs (16 of K) per block: 4, or 1 where only the first 16 of a 64-wide block are not zero.
template <int BN, int KS>
struct WsShape {
  static constexpr int REGION = BN <= 64 ? 64 : BN <= 128 ? 128 : 256;  // TMEM columns of a region
  static constexpr int A_BYTES = 128 * 128, B_BYTES = BN * 128, STAGE = A_BYTES + B_BYTES;
  static constexpr int STAGES = 196608 / STAGE < 8 ? 196608 / STAGE : 8;
  static constexpr int ROWS_BYTES = 2 * 128 * 16;  // the gathering warps' row tables (two per row)
  static constexpr size_t SMEM = (size_t)STAGES * STAGE + 1024 + 256 + ROWS_BYTES;
  static_assert(8 * (3 * STAGES + 4) + 8 <= 256, "barriers, TMEM slot, abort flag");
  static constexpr int HALF = BN / 2;  // columns of a promoting warp
  static constexpr int CH = HALF == 96 ? 16 : HALF % 32 == 0 ? 32 : HALF % 24 == 0 ? 24 : 8;  // columns read from TMEM at a time
  static_assert(BN % 16 == 0 && HALF % CH == 0 && BN <= 256 && STAGES >= 4, "tile");
};

__device__ __forceinline__ void tc_ld8_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
}
template <int CH>
__device__ __forceinline__ void tc_ld_add(uint32_t taddr, float* acc) {
  if constexpr (CH == 32) {
    float v[32];
    tc_ld32(taddr, v);
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] += v[j];
  } else {
    uint32_t r[CH];
#pragma unroll
    for (int j = 0; j < CH; j += 8) tc_ld8_nowait(taddr + j, r + j);
    tc_ld_wait(r);
#pragma unroll
    for (int j = 0; j < CH; ++j) acc[j] += __uint_as_float(r[j]);
  }
}
__device__ __forceinline__ void ws_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void ws_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void ws_bulk(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void ws_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool ws_wait(uint32_t bar, uint32_t parity, long limit, volatile int* abort) {
  for (long i = 0; i < limit; ++i) {
    if (tc_try_wait(bar, parity)) return true;
    if ((i & 63) == 63 && *abort) return false;
  }
  return false;
}

// Transpose of 8 x 8 16-bit values over eight consecutive lanes: lane p's r[i] holds values 2 i, 2 i + 1 of row p; afterwards
// of column p.
__device__ __forceinline__ void transpose8(uint32_t (&r)[4], int lane) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const uint32_t o = __shfl_xor_sync(0xffffffffu, r[i], 1);
    r[i] = (lane & 1) ? __byte_perm(o, r[i], 0x7632) : __byte_perm(r[i], o, 0x5410);
  }
#pragma unroll
  for (int i = 0; i < 4; i += 2) {
    const uint32_t o = __shfl_xor_sync(0xffffffffu, (lane & 2) ? r[i] : r[i + 1], 2);
    if (lane & 2) r[i] = o;
    else r[i + 1] = o;
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const uint32_t o = __shfl_xor_sync(0xffffffffu, (lane & 4) ? r[i] : r[i + 2], 4);
    if (lane & 4) r[i] = o;
    else r[i + 2] = o;
  }
}

// Warps that gather A (or, where A is an image, issue its copies).  A warp spends ~60 clocks a cp.async on addresses
// and masks one after the other; with two warps the MMAs of the narrow layers waited 2100 clocks a block for A
// (input gradients of 48 and 96 columns: 497 and 210 us with two warps, 264 and 122 with four).  At 256 columns the
// promoting warps' 128 sums leave no registers for two more warps (232 us with two, 480 with four and spills).
template <class LoadA, int BN>
__host__ __device__ constexpr int ws_gather_warps() {
  return !LoadA::kGather ? 1 : BN <= 192 ? 4 : 2;
}
template <class LoadA, int BN>
__host__ __device__ constexpr int ws_threads() {
  return WS_PROMOTE + 32 * ws_gather_warps<LoadA, BN>() + 32;
}

// Work of one launch: row tiles x column tiles x splits of K, columns fastest (CTAs side by side share A's rows).
struct WsWork {
  int row_tiles, col_tiles, splits, kb_all, kb_per;
};

// A row of a gathered operand: the address of its tap 0 (not necessarily inside the array) and, in bit t of m, whether
// its tap t lies inside (other bits are the loader's).
struct GatherRow {
  const __nv_bfloat16* p;
  unsigned m;
  unsigned pad;
};
// LoadA: gathered operands define kGather = true, GatherRow row(int m), int tile_class(int tile), K kpos(int k, int cls)
// with a member tap, int offset(row, K) in elements, and int kb_next(int cls, int kb): the first block >= kb with a
// nonzero element in row tiles of the class (skipped blocks would add exact zeros).  Image operands: kGather = false, member `op`.
// Epi: Row prep(int m) and epi(Row, col, v) with eight consecutive columns.
template <class LoadA, class Epi, int BN, int KS>
__global__ void __launch_bounds__(ws_threads<LoadA, BN>(), 1)
    k_gemm_ws(LoadA la, ImageOperand b, WsWork wk, Epi epi, int* status, long spin) {
  using S = WsShape<BN, KS>;
  constexpr int ST = S::STAGES, GW = ws_gather_warps<LoadA, BN>();
  extern __shared__ __align__(1024) unsigned char ws_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)ws_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + ST * S::STAGE);
  // barriers: [ST] A gathered, [ST] bulk copies landed, [ST] stage free, [2] region done, [2] region free
  const uint32_t fullA = tc_smem_u32(bars), fullB = fullA + 8 * ST, empty = fullB + 8 * ST, done = empty + 8 * ST,
                 rfree = done + 16;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 3 * ST + 4);
  volatile int* abort = reinterpret_cast<volatile int*>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(tslot)),
                 "r"(2 * S::REGION));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 0) {
    auto init = [](uint32_t bar, int n) { asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(n)); };
    for (int i = 0; i < ST; ++i) {
      init(fullA + 8 * i, 32 * GW);
      init(fullB + 8 * i, 1);
      init(empty + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      init(done + 8 * i, 1);
      init(rfree + 8 * i, WS_PROMOTE / 32);
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;

  const int items = wk.row_tiles * wk.col_tiles * wk.splits;
  struct Item {
    int tile, n0, kb0, kb1, cls;
  };
  auto item = [&](int w) {
    Item it;
    it.n0 = (w % wk.col_tiles) * BN;
    it.tile = w / wk.col_tiles % wk.row_tiles;
    const int z = w / wk.col_tiles / wk.row_tiles;
    it.kb0 = z * wk.kb_per;
    it.kb1 = min(it.kb0 + wk.kb_per, wk.kb_all);
    if constexpr (LoadA::kGather) it.cls = la.tile_class(it.tile);
    return it;
  };
  auto next = [&](const Item& it, int kb) {  // first block >= kb of the item with work, or kb1
    if constexpr (LoadA::kGather) return min(la.kb_next(it.cls, kb), it.kb1);
    else return kb;
  };
  auto fail = [&]() {
    *abort = 1;
    atomicOr(status, PTY_ETIMEOUT);
  };
  int q = 0;  // blocks of this CTA so far; block q uses stage q % ST, region q % 2

  if (warp < 8) {
    // ---- promote ----
    const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
    const int col0 = (warp >> 2) * S::HALF;
    bool ok = true;
    for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
      const Item it = item(w);
      float acc[S::HALF];
#pragma unroll
      for (int j = 0; j < S::HALF; ++j) acc[j] = 0.f;
      for (int kb = next(it, it.kb0); kb < it.kb1; kb = next(it, kb + 1), ++q) {
        const int r = q & 1;
        ok = __all_sync(0xffffffffu, ws_wait(done + 8 * r, (uint32_t)(q >> 1) & 1, spin, abort)) != 0;
        if (!ok) {
          if (lane == 0) fail();
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t region = tmem + (uint32_t)(r * S::REGION) + lane_base + col0;
#pragma unroll
        for (int c = 0; c < S::HALF; c += S::CH) tc_ld_add<S::CH>(region + c, acc + c);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) ws_arrive(rfree + 8 * r);
      }
      if (!ok) break;
      const typename Epi::Row row = epi.prep(it.tile * 128 + 32 * (warp & 3) + lane);
#pragma unroll
      for (int j = 0; j < S::HALF; j += 8) epi(row, it.n0 + col0 + j, acc + j);
    }
  } else if (warp < 8 + GW) {
    // ---- gather A; bulk copies ----
    const int t = tid - WS_PROMOTE;
    const bool copies = t == 0;
    [[maybe_unused]] int announced = 0;
    bool ok = true;
    for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
      const Item it = item(w);
      if constexpr (LoadA::kGather) {
        // warp pairs take 256 / GW rows each, the two warps of a pair four of the eight 16-byte chunks of K
        const int kg = (lane >> 3) + 4 * (warp & 1), row0 = ((warp - 8) >> 1) * (256 / GW);
        constexpr int ROWS = 32 / GW;
        GatherRow* table = reinterpret_cast<GatherRow*>(base + ST * S::STAGE + 256) + (256 / GW) * (warp - 8);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < ROWS / 4; ++j) table[lane + 32 * j] = la.row(it.tile * 128 + row0 + lane + 32 * j);
        __syncwarp();
        GatherRow row[ROWS];
#pragma unroll
        for (int j = 0; j < ROWS; ++j) row[j] = table[(lane & 7) + 8 * j];
        for (int kb = next(it, it.kb0); kb < it.kb1; kb = next(it, kb + 1), ++q) {
          const int s = q % ST;
          ok = q < ST || __all_sync(0xffffffffu, ws_wait(empty + 8 * s, (uint32_t)(q / ST - 1) & 1, spin, abort));
          if (!ok) {
            if (lane == 0) fail();
            break;
          }
          unsigned char* st = base + s * S::STAGE;
          if (copies) {
            ws_expect(fullB + 8 * s, S::B_BYTES);
            ws_bulk(tc_smem_u32(st + S::A_BYTES), b.p + (size_t)kb * b.rows * 64 + (size_t)it.n0 * 64, S::B_BYTES, fullB + 8 * s);
          }
          if (KS == 4 || kg < 2 * KS) {
            const typename LoadA::K k = la.kpos(kb * kWsBlock + 8 * kg, it.cls);
            const uint32_t d = tc_smem_u32(st) + row0 * 128 + (lane & 7) * 16 + kg * 128;
#pragma unroll
            for (int j = 0; j < ROWS; ++j) {
              const bool in = (row[j].m >> k.tap) & 1;
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d + j * 1024),
                           "l"(in ? row[j].p + la.offset(row[j], k) : la.any()), "r"(in ? 16 : 0)
                           : "memory");
            }
          }
          asm volatile("cp.async.commit_group;" ::: "memory");
          if (q - announced >= 2) {  // block q - 2 has landed
            asm volatile("cp.async.wait_group 2;" ::: "memory");
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            ws_arrive(fullA + 8 * (announced % ST));
            ++announced;
          }
        }
      } else if (copies) {
        for (int kb = it.kb0; kb < it.kb1; ++kb, ++q) {
          const int s = q % ST;
          if (q >= ST && !ws_wait(empty + 8 * s, (uint32_t)(q / ST - 1) & 1, spin, abort)) {
            fail();
            ok = false;
            break;
          }
          unsigned char* st = base + s * S::STAGE;
          const int m0 = it.tile * 128, ar = min(128, la.op.rows - m0), br = min(BN, b.rows - it.n0);
          ws_expect(fullB + 8 * s, (uint32_t)(ar + br) * 128);
          ws_bulk(tc_smem_u32(st), la.op.p + (size_t)kb * la.op.rows * 64 + (size_t)m0 * 64, (uint32_t)ar * 128, fullB + 8 * s);
          ws_bulk(tc_smem_u32(st + S::A_BYTES), b.p + (size_t)kb * b.rows * 64 + (size_t)it.n0 * 64, (uint32_t)br * 128, fullB + 8 * s);
        }
      }
    }
    if constexpr (LoadA::kGather) {
      asm volatile("cp.async.wait_all;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      for (; announced < q; ++announced) ws_arrive(fullA + 8 * (announced % ST));
    }
    if (copies) {  // every copy has landed before the CTA can end (only after an abort is there one to wait for)
      for (int i = q > ST ? q - ST : 0; i < q; ++i) tc_wait(fullB + 8 * (i % ST), (uint32_t)(i / ST) & 1);
    }
  } else if (lane == 0) {
    // ---- MMA ----
    constexpr uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | (8u << 24);
    bool ok = true;
    for (int w = blockIdx.x; w < items && ok; w += gridDim.x) {
      const Item it = item(w);
      for (int kb = next(it, it.kb0); kb < it.kb1; kb = next(it, kb + 1), ++q) {
        const int s = q % ST, r = q & 1;
        const uint32_t par = (uint32_t)(q / ST) & 1;
        ok = ws_wait(fullB + 8 * s, par, spin, abort) && (!LoadA::kGather || ws_wait(fullA + 8 * s, par, spin, abort)) &&
             (q < 2 || ws_wait(rfree + 8 * r, (uint32_t)((q >> 1) - 1) & 1, spin, abort));
        if (!ok) {
          fail();
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sa = tc_smem_u32(base + s * S::STAGE), sb = sa + S::A_BYTES, d = tmem + (uint32_t)(r * S::REGION);
#pragma unroll
        for (int k = 0; k < KS; ++k) {
          const uint64_t da = tc_desc(sa + k * 256), db = tc_desc(sb + k * 256);
          const uint32_t accum = k > 0 ? 1u : 0u;
          asm volatile(
              "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d),
              "l"(da), "l"(db), "r"(id), "r"(accum));
        }
        ws_commit(empty + 8 * s);
        ws_commit(done + 8 * r);
      }
    }
    // the last block's MMAs are complete before the tensor memory is released
    if (q > 0) tc_wait(done + 8 * ((q - 1) & 1), (uint32_t)((q - 1) >> 1) & 1);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * S::REGION));
}

template <int BN, int KS, class LA, class Epi>
cudaError_t launch_gemm_ws(const LA& la, const ImageOperand& b, WsWork wk, const Epi& epi, int* status, cudaStream_t st) {
  auto kern = k_gemm_ws<LA, Epi, BN, KS>;
  using S = WsShape<BN, KS>;
  static bool ready[256] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
  if (!__atomic_load_n(&ready[dev], __ATOMIC_ACQUIRE)) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    if (e != cudaSuccess) return e;
    __atomic_store_n(&ready[dev], true, __ATOMIC_RELEASE);
  }
  if (wk.splits > wk.kb_all) wk.splits = wk.kb_all;
  if (wk.splits < 1) wk.splits = 1;
  wk.kb_per = (wk.kb_all + wk.splits - 1) / wk.splits;
  wk.splits = (wk.kb_all + wk.kb_per - 1) / wk.kb_per;
  const long long items = (long long)wk.row_tiles * wk.col_tiles * wk.splits;
  kern<<<(unsigned)(items < 152 ? items : 152), ws_threads<LA, BN>(), S::SMEM, st>>>(la, b, wk, epi, status, stage_wait_limit());
  return cudaGetLastError();
}

}  // namespace pty
