// GEMMs of the MAR block: QKV, attention output, MLP up and down projections
// (Eq. 9's F(X[I_compute]) for the token subset, and the full-layer forms).
//
// bf16: a persistent, warp-specialised tcgen05 kernel, on single CTAs or on
// CTA pairs that share a 256-row tile (cta_group::2). Warp 0 streams A and W
// tiles with TMA (128B swizzle) into a ring of shared-memory stages, warp 1
// issues tcgen05.mma (128 x BN x 16, fp32 accumulators in tensor memory,
// double-buffered so the epilogue of one tile overlaps the main loop of the
// next) and 8 to 16 epilogue warps drain the accumulators with tcgen05.ld and
// apply the fused epilogue: bias, GELU, fp32 residual add, or the Q/K/V split
// with the K/V rows scattered into the token cache (row_map). Few rows take
// tiles of 64 rows.
//
// f32: CUDA-core kernels with the same epilogues (the tensor cores have no fp32
// kind; these serve the fp32 configuration): small tiles with K split over the
// warps, and for many rows a 64 x 64 register-tiled kernel.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <mutex>

#include <cstring>

#include "lazymar_internal.cuh"

namespace lm {

// ---------------------------------------------------------------------------
// Epilogue shared by both kernels: NC consecutive columns of one row.
// ---------------------------------------------------------------------------
template <typename T, int NC>
__device__ __forceinline__ void epilogue_apply(const GemmEpi& e, int row, int col0, float* v) {
  if (e.bias) {
    float bv[NC];
    Vec<T, NC>::load(static_cast<const T*>(e.bias) + col0, bv);
#pragma unroll
    for (int i = 0; i < NC; ++i) v[i] += bv[i];
  }
  switch (e.mode) {
    case LAZYMAR_EPI_GELU:
#pragma unroll
      for (int i = 0; i < NC; ++i) v[i] = gelu_erf(v[i]);
      Vec<T, NC>::store(static_cast<T*>(e.out) + (size_t)row * e.ldo + col0, v);
      break;
    case LAZYMAR_EPI_SILU:
#pragma unroll
      for (int i = 0; i < NC; ++i) v[i] = silu(v[i]);
      Vec<T, NC>::store(static_cast<T*>(e.out) + (size_t)row * e.ldo + col0, v);
      break;
    case LAZYMAR_EPI_RESIDUAL: {
      float* o = static_cast<float*>(e.out) + (size_t)row * e.ldo + col0;
      float r[NC];
      Vec<float, NC>::load(o, r);
      if (e.gate) {
        float g[NC];
        Vec<T, NC>::load(static_cast<const T*>(e.gate) + (size_t)row * e.ldg + col0, g);
#pragma unroll
        for (int i = 0; i < NC; ++i) v[i] *= g[i];
      }
#pragma unroll
      for (int i = 0; i < NC; ++i) r[i] += v[i];
      Vec<float, NC>::store(o, r);
      break;
    }
    case LAZYMAR_EPI_QKV: {
      const int part = col0 / e.D;
      const int c = col0 - part * e.D;
      T* dst;
      if (part == 0) {
        dst = static_cast<T*>(e.out) + (size_t)row * e.D + c;
      } else {
        const int drow = e.row_map ? e.row_map[row] : row;
        dst = static_cast<T*>(part == 1 ? e.k_out : e.v_out) + (size_t)drow * e.D + c;
      }
      Vec<T, NC>::store(dst, v);
      break;
    }
    default:
      Vec<T, NC>::store(static_cast<T*>(e.out) + (size_t)row * e.ldo + col0, v);
      break;
  }
}

// ---------------------------------------------------------------------------
// tcgen05 kernel
// ---------------------------------------------------------------------------
namespace tc {
constexpr int BM = 128;  // rows per tile = MMA M (one accumulator lane per row)

// Epilogue kinds: BF16OUT stores bf16 (bias / GELU / Q-K-V split); the two
// residual kinds add into the fp32 residual stream. RESID_WIDE stages whole
// 32-column fp32 chunks (for short K, where the epilogue bounds the kernel, at
// the cost of one pipeline stage); RESID_HALF stages 16-column halves and keeps
// every stage (for long K, where the main loop bounds it).
// RESID_WIDE_GATED is RESID_WIDE with a per-element gate on the product
// (out += gate * y, the adaptive-LayerNorm residual of the diffusion head),
// a separate instantiation so that the ungated kinds carry no gate code.
// BF16OUT_SILU is BF16OUT with the SiLU activation, likewise separate.
enum EpiKind { BF16OUT = 0, RESID_WIDE = 1, RESID_HALF = 2, RESID_WIDE_GATED = 3, BF16OUT_SILU = 4 };
template <int EK>
constexpr bool is_wide() { return EK == RESID_WIDE || EK == RESID_WIDE_GATED; }
template <int EK>
constexpr bool is_bf16out() { return EK == BF16OUT || EK == BF16OUT_SILU; }

// BK: K per pipeline stage (elements), one or two swizzle atoms. A 128-wide
// tile runs 128-deep stages (two atoms, eight MMAs per barrier round trip):
// its 128 x 128 x 16 MMAs are too short to hide the per-stage wait and commit
// at 64 (measured 13-19 % faster); wider tiles keep 64 for a deeper ring.
// F8: E4M3 operands (kind::f8f6f4): a 128-byte atom holds 128 elements and an
// MMA step is K = 32, still 32 bytes; BK = 128 is one atom, the bytes of a
// 64-deep bf16 stage.
// PAIR: two CTAs (a cluster of two on neighbouring SMs) share a 256 x BN tile.
// Each holds its own 128 rows of A and half of the tile's B rows, so an SM
// fills and reads 128 + BN / 2 instead of 128 + BN operand rows per K step; the
// even CTA issues the MMAs (cta_group::2) for both.
// ROWS: rows of a tile = M of its MMAs. 64-row tiles serve few-row GEMMs: an MMA
// takes as long as its operands' shared-memory reads, 64 cycles at M = 128 for
// any N up to 128 (measured 65 at N = 64) and half of that at M = 64.
template <int BN, int EK, int BK, int F8 = 0, int PAIR = 0, int ROWS = 128>
struct Cfg {
  static constexpr int EB = F8 ? 1 : 2;          // bytes per operand element
  static constexpr int ATOM_E = 128 / EB;        // elements per 128-byte swizzle atom
  static constexpr int ATOMS = BK / ATOM_E;
  // (64-wide tiles, with half the B tile per stage, afford one more stage)
  static constexpr int SINGLE_STAGES = ATOMS == 2 ? (is_wide<EK>() ? 2 : 3) + (BN == 64 ? 1 : 0)
                                          : is_wide<EK>() ? (BN == 256 ? 3 : BN == 192 ? 4 : 5)
                                                             : (BN == 256 ? 4 : BN == 192 ? 5 : 6);
  static constexpr uint32_t A_BYTES = ROWS * BK * EB;
  static constexpr int B_ROWS = PAIR ? BN / 2 : BN;  // rows of B in this CTA's shared memory
  static constexpr uint32_t B_BYTES = B_ROWS * BK * EB;
  static constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
  // two accumulator buffers (columns [0, BN) and [BN, 2 BN)); the allocation
  // is a power of two
  static constexpr uint32_t TMEM_COLS = 2 * BN <= 256 ? 256 : 512;
  // Per-warp staging of 32 rows (64 or 128 bytes each), rows padded by 16
  // bytes so that both the row-wise writes and the column-block reads are
  // bank-conflict-lean.
  // Epilogue warps: the bf16-output kinds use four (three for BN = 192) per
  // tensor-memory lane quarter, so more warps share a tile's conversion,
  // GELU and stores; the residual kinds, with more live registers, two.
  static constexpr int EPI_WARPS = !is_bf16out<EK>() ? 8 : (BN == 192 ? 12 : BN == 64 ? 8 : 16);
  static constexpr int THREADS = 64 + EPI_WARPS * 32;
  static constexpr int CHUNKS = BN / 32 / (EPI_WARPS / 4);  // 32-column chunks per warp and tile
  // Per-warp staging of 32 rows: bf16 rows of 64 bytes, 16-byte blocks
  // swizzled by row (conflict-free row-wise writes and column-block reads);
  // fp32 rows of 64 or 128 bytes padded by 16 bytes.
  static constexpr uint32_t ROW_BYTES = is_wide<EK>() ? 128 : 64;
  static constexpr uint32_t STG_PITCH = is_bf16out<EK>() ? 64 : ROW_BYTES + 16;
  static constexpr uint32_t STG_BYTES = 32 * STG_PITCH;
  // a pair's smaller stages: as many as shared memory holds, at most eight
  static constexpr int FIT_STAGES = (int)((232448 - 1024 - 256 - EPI_WARPS * STG_BYTES) / STAGE_BYTES);
  static constexpr int STAGES = !PAIR && ROWS == 128 ? SINGLE_STAGES : FIT_STAGES < 8 ? FIT_STAGES : 8;
  static constexpr size_t SMEM = 1024 + (size_t)STAGES * STAGE_BYTES + EPI_WARPS * STG_BYTES + 256;
  // Instruction descriptor: D fp32 (bit 4); kind::f16 with A and B bf16
  // (bits 7-9 and 10-12 = 1), or kind::f8f6f4 with A and B E4M3 (format 0);
  // both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
  static constexpr uint32_t IDESC = (1u << 4) | (F8 ? 0u : (1u << 7) | (1u << 10)) | ((uint32_t)(BN >> 3) << 17) |
                                    ((uint32_t)((PAIR ? 2 * BM : ROWS) >> 4) << 24);
  // Rows of a tile in each tensor-memory lane quarter: 32, or, at M = 64, 16 (in
  // its first 16 lanes).
  static constexpr int QROWS = ROWS / 4;
};

// Shared-memory matrix descriptor of a K-major tile written by TMA with
// SWIZZLE_128B: rows of 128 bytes, 8-row groups 1024 bytes apart (stride byte
// offset), descriptor version 1 (bit 46), layout SWIZZLE_128B (2 at bit 61).
// The leading byte offset is not used by this layout.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Four packed bf16 values as floats (the gates of four residual columns).
__device__ __forceinline__ float4 bf16x4_to_f4(uint2 u) {
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

// Destination row pointer of a bf16 epilogue for tile row `row`, column `col`
// (a 32-column chunk never straddles the Q/K/V parts).
__device__ __forceinline__ bf16* out_row(const GemmEpi& e, int row, int col) {
  if (e.mode != LAZYMAR_EPI_QKV) return static_cast<bf16*>(e.out) + (size_t)row * e.ldo + col;
  const int part = col / e.D;
  const int c = col - part * e.D;
  if (part == 0) return static_cast<bf16*>(e.out) + (size_t)row * e.D + c;
  const int drow = e.row_map ? e.row_map[row] : row;
  return static_cast<bf16*>(part == 1 ? e.k_out : e.v_out) + (size_t)drow * e.D + c;
}
}  // namespace tc

template <int BN, int EK, int BK, int F8 = 0, int PAIR = 0, int ROWS = 128, bool SPLIT = false>
__global__ void __launch_bounds__(tc::Cfg<BN, EK, BK, F8, PAIR, ROWS>::THREADS, 1)
    gemm_bf16_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmO0, const __grid_constant__ CUtensorMap tmO1,
                        const __grid_constant__ CUtensorMap tmO2, const __grid_constant__ CUtensorMap tmBt, int whole,
                        int split, int tma_out, int M, int N, int K, GemmEpi epi, unsigned* err) {
  using C = tc::Cfg<BN, EK, BK, F8, PAIR, ROWS>;
  static_assert(ROWS == 128 || (ROWS == 64 && !PAIR && !F8), "64-row tiles: single CTAs, bf16 operands");
  static_assert(!(F8 && PAIR), "pairs: bf16 operands only");
  static_assert(!F8 || EK == tc::BF16OUT, "E4M3 operands: bf16-output epilogue only");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::STAGES * C::A_BYTES;
  uint8_t* sStg = smem + C::STAGES * C::STAGE_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(sStg + C::EPI_WARPS * C::STG_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* acc_full = empty + C::STAGES;
  uint64_t* acc_empty = acc_full + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Tiles are numbered column-tile fastest: the CTAs running at the same time
  // cover a few row tiles completely, so each activation row tile is fetched
  // from memory once and shared through L2 by the CTAs that use it (the
  // weights, at most a few MB, stay in L2 throughout).
  constexpr int TM = PAIR ? 2 * tc::BM : ROWS;  // rows of a tile
  const int num_m = (M + TM - 1) / TM;
  const int num_n = N / BN;
  // `whole` tiles of the full width, then the others as `split` tiles of
  // BN / split columns each, which spread a short last round over all SMs.
  const int tiles = SPLIT ? whole + (num_m * num_n - whole) * split : num_m * num_n;
  struct Tile {
    int m, n, bn;  // first row and column of the CTA's or pair's tile, and its width
  };
  auto tile_at = [&](int t) {
    if (!SPLIT || t < whole) return Tile{(t / num_n) * TM, (t % num_n) * BN, BN};
    const int u = t - whole, base = whole + u / split, bw = BN / split;
    return Tile{(base / num_n) * TM, (base % num_n) * BN + (u % split) * bw, bw};
  };
  const int KB = K / BK;
  // a pair works on one tile: the even CTA (rank 0) on its first 128 rows and
  // the first half of its B rows, the odd one on the others
  const int rank = PAIR ? (int)cluster_ctarank() : 0;
  const int first = PAIR ? (int)blockIdx.x / 2 : (int)blockIdx.x, step = PAIR ? (int)gridDim.x / 2 : (int)gridDim.x;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], PAIR ? 2 * C::EPI_WARPS : C::EPI_WARPS);  // (of a pair: the even CTA's is used)
    }
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
    if (tma_out) {
      prefetch_tmap(&tmO0);
      if (epi.mode == LAZYMAR_EPI_QKV) {
        prefetch_tmap(&tmO1);
        prefetch_tmap(&tmO2);
      }
    }
  }
  if (warp == 1) {
    if (PAIR) {
      tmem_alloc_pair(tmem_slot, C::TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(tmem_slot, C::TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (PAIR) cluster_sync();  // the peer's barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Tile loads complete on the full barrier of the CTA that issues the MMAs.
  auto expect_stage = [&](int s, int bw) {
    const uint32_t b_bytes = (uint32_t)bw * BK * C::EB;
    if (rank == 0) mbar_arrive_expect_tx(&full[s], PAIR ? 2 * C::A_BYTES + b_bytes : C::A_BYTES + b_bytes);
  };
  auto load_a = [&](int s, int kb, int m0) {
#pragma unroll
    for (int a = 0; a < C::ATOMS; ++a) {
      uint8_t* dst = sA + s * C::A_BYTES + a * (C::A_BYTES / C::ATOMS);
      if (PAIR)
        tma_load_2d_pair(&tmA, cluster_map(smem_u32(&full[s]), 0), dst, kb * BK + a * C::ATOM_E, m0);
      else
        tma_load_2d(&tmA, &full[s], dst, kb * BK + a * C::ATOM_E, m0);
    }
  };
  auto load_b = [&](int s, int kb, int n0, int bw) {
#pragma unroll
    for (int a = 0; a < C::ATOMS; ++a) {
      uint8_t* dst = sB + s * C::B_BYTES + a * (C::B_BYTES / C::ATOMS);
      if (PAIR)
        tma_load_2d_pair(bw == BN ? &tmB : &tmBt, cluster_map(smem_u32(&full[s]), 0), dst, kb * BK + a * C::ATOM_E,
                         n0 + rank * (bw / 2));
      else
        tma_load_2d(bw == BN ? &tmB : &tmBt, &full[s], dst, kb * BK + a * C::ATOM_E, n0);
    }
  };
  // Weights are never written by any kernel, so the producer fetches the
  // weight tiles of its first stages before waiting for the predecessor grid;
  // every other access follows pdl_wait().
  int pre = 0;
  if (warp == 0 && lane == 0 && first < tiles) {
    const Tile t = tile_at(first);
    pre = KB < C::STAGES ? KB : C::STAGES;
    for (int s = 0; s < pre; ++s) {
      expect_stage(s, t.bn);
      load_b(s, s, t.n, t.bn);
    }
  }
  pdl_wait();
  pdl_trigger();

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int tile = first; tile < tiles && ok; tile += step) {
        const Tile t = tile_at(tile);
        const int m0 = t.m + rank * tc::BM, n0 = t.n;
        for (int kb = 0; kb < KB; ++kb) {
          if (tile == first && kb < pre) {
            // weight tile already in flight on this stage: add the activations
            load_a(stage, kb, m0);
          } else {
            if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, err)) { ok = false; break; }
            expect_stage(stage, t.bn);
            load_a(stage, kb, m0);
            load_b(stage, kb, n0, t.bn);
          }
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (of a pair: the even CTA's) ----------------
    // For the small tiles and the bf16-output pairs the warp runs converged and
    // one elected lane issues (few-row fc2, a stage of eight 128 x 64 x 16 MMAs:
    // 0.322 us against 0.347 with a single lane in the loop, 0.252 of it the
    // MMAs; full-layer Q/K/V 47.7 -> 45.0 us, fc1 65.2 -> 65.6); the other kinds
    // are up to 2 % faster with the single lane.
    constexpr bool CONVERGED = BN == 64 || ROWS == 64 || (PAIR && tc::is_bf16out<EK>());
    if (rank == 0 && (CONVERGED || lane == 0)) {
      const bool lead = CONVERGED ? elect_one() : true;
      auto wait = [&](uint64_t* bar, uint32_t parity) {
        const bool done = mbar_wait(bar, parity, abort_flag, err);
        return CONVERGED ? (bool)__all_sync(0xffffffffu, done) : done;
      };
      int stage = 0;
      uint32_t phase = 0;
      int it = 0;
      bool ok = true;
      for (int tile = first; tile < tiles && ok; tile += step, ++it) {
        const int buf = it & 1;
        const uint32_t use = (uint32_t)(it >> 1) & 1u;
        if (!wait(&acc_empty[buf], use ^ 1u)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(buf * BN);
        // N of the MMAs (bits 17 up of the instruction descriptor)
        const uint32_t idesc = C::IDESC - ((uint32_t)((BN - tile_at(tile).bn) >> 3) << 17);
        for (int kb = 0; kb < KB; ++kb) {
          ok = wait(&full[stage], phase);
          if (!ok) break;
          tc_fence_after();
          const uint64_t a0 = tc::sw128_desc(smem_u32(sA + stage * C::A_BYTES));
          const uint64_t b0 = tc::sw128_desc(smem_u32(sB + stage * C::B_BYTES));
          if (lead) {
#pragma unroll
            for (int k = 0; k < C::ATOMS * 4; ++k) {  // +32 bytes per MMA step inside an atom
              const int a = k / 4, ks = k % 4;
              const uint64_t ao = (uint64_t)((a * (C::A_BYTES / C::ATOMS)) >> 4) + 2 * ks;
              const uint64_t bo = (uint64_t)((a * (C::B_BYTES / C::ATOMS)) >> 4) + 2 * ks;
              if (PAIR)
                umma_bf16_pair(d_tmem, a0 + ao, b0 + bo, idesc, (kb | k) != 0 ? 1u : 0u);
              else if (F8)
                umma_e4m3(d_tmem, a0 + ao, b0 + bo, idesc, (kb | k) != 0 ? 1u : 0u);
              else
                umma_bf16(d_tmem, a0 + ao, b0 + bo, idesc, (kb | k) != 0 ? 1u : 0u);
            }
            if (PAIR)
              umma_commit_pair(&empty[stage]);
            else
              umma_commit(&empty[stage]);
          }
          if (CONVERGED) __syncwarp();
          if (++stage == C::STAGES) { stage = 0; phase ^= 1u; }
        }
        if (ok && lead) {
          if (PAIR)
            umma_commit_pair(&acc_full[buf]);
          else
            umma_commit(&acc_full[buf]);
        }
        if (CONVERGED) __syncwarp();
      }
    }
    __syncwarp();
  } else {
    // ---------------- epilogue warps ----------------
    // Each warp owns 32 accumulator rows (its TMEM lane quarter) and one of the
    // EPI_WARPS / 4 column ranges of the tile, processed as 32 x 32 chunks (16 x 32 in a 64-row tile)
    // (CHUNKS per tile). tcgen05.ld gives one row
    // per thread; each chunk is transposed through the warp's staging buffer
    // (32 rows x 64 bytes: 32 bf16 columns, or 16 fp32 columns at a time) so
    // that every global store and residual load covers 8 rows x 64 contiguous
    // bytes per warp instruction. The residual of the next chunk is loaded
    // while the current one is processed, and the first chunk's before the
    // accumulator is ready.
    const int ew = warp - 2;        // 0 .. EPI_WARPS - 1
    const int quarter = warp & 3;   // tensor-memory lanes this warp may read
    const int half = ew >> 2;       // which column range of the tile (of EPI_WARPS / 4)
    constexpr int CHUNKS = C::CHUNKS;
    uint8_t* stg = sStg + ew * C::STG_BYTES;
    const int cr = lane >> 2;       // row within an 8-row pass
    const int cq = lane & 3;        // 16-byte block within the 64-byte row segment
    float* const res_base = static_cast<float*>(epi.out);
    int it = 0;
    for (int tile = first; tile < tiles; tile += step, ++it) {
      const int buf = it & 1;
      const uint32_t use = (uint32_t)(it >> 1) & 1u;
      const Tile t = tile_at(tile);
      const int m0 = t.m + rank * tc::BM, n0 = t.n;
      const int rbase = m0 + quarter * C::QROWS;  // first of this warp's rows
      // this warp's chunks: a narrower tile gives each warp fewer, some none
      const int per = t.bn == BN ? CHUNKS : (t.bn / 32 + C::EPI_WARPS / 4 - 1) / (C::EPI_WARPS / 4);
      const int c0 = half * per;
      const int c1 = t.bn == BN ? c0 + CHUNKS : min(c0 + per, t.bn / 32);
      // residual of a 32-column chunk in the coalesced layout: [16-col half][pass]
      float4 res[2][4];
      uint2 rbias[2];  // the 4 bias values of this lane's columns in each 16-column half (bf16)
      auto load_res = [&](int col) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          rbias[h] = epi.bias ? *reinterpret_cast<const uint2*>(static_cast<const bf16*>(epi.bias) + col + h * 16 + cq * 4)
                              : make_uint2(0u, 0u);
#pragma unroll
          for (int p = 0; p < C::QROWS / 8; ++p) {
            const int row = rbase + p * 8 + cr;
            res[h][p] = row < M ? *reinterpret_cast<const float4*>(res_base + (size_t)row * epi.ldo + col + h * 16 + cq * 4)
                                : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
      };
      // RESID_WIDE layout: [pass] with 4 rows x 8 blocks of 16 bytes per pass
      // (gated kind: the gates of the same elements, prefetched alike)
      float4 resw[8];
      uint2 gatew[8];  // 4 bf16 gates each
      uint2 wbias;     // the 4 bias values of this lane's columns (bf16)
      auto load_resw = [&](int col) {
        const int wr = lane >> 3, wq = lane & 7;
        wbias = epi.bias ? *reinterpret_cast<const uint2*>(static_cast<const bf16*>(epi.bias) + col + wq * 4)
                         : make_uint2(0u, 0u);
#pragma unroll
        for (int p = 0; p < C::QROWS / 4; ++p) {
          const int row = rbase + p * 4 + wr;
          resw[p] = row < M ? *reinterpret_cast<const float4*>(res_base + (size_t)row * epi.ldo + col + wq * 4)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
          if (EK == tc::RESID_WIDE_GATED)
            gatew[p] = row < M ? *reinterpret_cast<const uint2*>(static_cast<const bf16*>(epi.gate) +
                                                                 (size_t)row * epi.ldg + col + wq * 4)
                               : make_uint2(0u, 0u);
        }
      };
      // bf16-output kinds: the bias of the next 32-column chunk (packed bf16),
      // loaded before it is needed, the first chunk's before the accumulator
      // is ready
      uint4 bpre[4];
      auto load_bias = [&](int col) {
        if (epi.bias) {
          const uint4* bp = reinterpret_cast<const uint4*>(static_cast<const bf16*>(epi.bias) + col);
#pragma unroll
          for (int j = 0; j < 4; ++j) bpre[j] = bp[j];
        }
      };
      const bool some = !SPLIT || c0 < c1;
      if (EK == tc::RESID_HALF && some) load_res(n0 + c0 * 32);
      if (tc::is_wide<EK>() && some) load_resw(n0 + c0 * 32);
      if (tc::is_bf16out<EK>() && !F8 && some) load_bias(n0 + c0 * 32);
      const bool ok = mbar_wait(&acc_full[buf], use, abort_flag, err);
      if (__any_sync(0xffffffffu, !ok)) break;
      tc_fence_after();
      // The tensor-memory load of chunk c + 1 is issued as soon as chunk c's
      // accumulator registers have been consumed, and waited for at the top
      // of the next iteration (the wait names the registers, so no use of
      // them moves above it).
      // (Only for the kinds where the extra live registers do not spill: the
      // residual kind over short K and the bf16-output kinds up to 192 wide.
      // The others load and wait at the top of each iteration.)
      constexpr bool PIPE = EK == tc::RESID_WIDE || (tc::is_bf16out<EK>() && BN <= 192);
      uint32_t r[32];
      auto tld = [&](int c) {
        tmem_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * BN + c * 32), r);
      };
      // The tile's accumulator buffer goes back to the MMA warp as soon as
      // this warp's last chunk is out of tensor memory, before its stores.
      auto release = [&] {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          if (PAIR)
            mbar_arrive_cluster(cluster_map(smem_u32(&acc_empty[buf]), 0));
          else
            mbar_arrive(&acc_empty[buf]);
        }
      };
      if (!some) {
        release();
        continue;
      }
      if (PIPE) tld(c0);
#pragma unroll 1
      for (int c = c0; c < c1; ++c) {
        const int col = n0 + c * 32;
        const bool more = c + 1 < c1;
        if (!PIPE) tld(c);
        tmem_wait_ld_regs(r);
        if (tc::is_wide<EK>()) {
          // whole 32-column fp32 chunk: 4 rows x 128 B per warp instruction
          float4* srow = reinterpret_cast<float4*>(stg + lane * C::STG_PITCH);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            srow[j] = make_float4(__uint_as_float(r[4 * j]), __uint_as_float(r[4 * j + 1]),
                                  __uint_as_float(r[4 * j + 2]), __uint_as_float(r[4 * j + 3]));
          if (PIPE && more) tld(c + 1);
          if (!more) release();  // the whole accumulator is out of tensor memory
          __syncwarp();
          const int wr = lane >> 3, wq = lane & 7;
          const float4 bq = tc::bf16x4_to_f4(wbias);  // prefetched with the residual
          float4 cur[8];
          uint2 curg[8];
#pragma unroll
          for (int p = 0; p < C::QROWS / 4; ++p) {
            cur[p] = resw[p];
            if (EK == tc::RESID_WIDE_GATED) curg[p] = gatew[p];
          }
          if (c + 1 < c1) load_resw(col + 32);  // prefetch the next chunk
#pragma unroll
          for (int p = 0; p < C::QROWS / 4; ++p) {
            const int lr = p * 4 + wr;
            const int row = rbase + lr;
            const float4 a = *reinterpret_cast<const float4*>(stg + lr * C::STG_PITCH + wq * 16);
            if (row < M) {
              float4 o;
              if (EK == tc::RESID_WIDE_GATED) {
                const float4 gg = tc::bf16x4_to_f4(curg[p]);
                o.x = fmaf(gg.x, a.x + bq.x, cur[p].x);
                o.y = fmaf(gg.y, a.y + bq.y, cur[p].y);
                o.z = fmaf(gg.z, a.z + bq.z, cur[p].z);
                o.w = fmaf(gg.w, a.w + bq.w, cur[p].w);
              } else {
                o.x = cur[p].x + (a.x + bq.x);
                o.y = cur[p].y + (a.y + bq.y);
                o.z = cur[p].z + (a.z + bq.z);
                o.w = cur[p].w + (a.w + bq.w);
              }
              *reinterpret_cast<float4*>(res_base + (size_t)row * epi.ldo + col + wq * 4) = o;
            }
          }
          __syncwarp();
        } else if (EK == tc::RESID_HALF) {
          float4 cur[2][4];
#pragma unroll
          for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int p = 0; p < C::QROWS / 8; ++p) cur[h][p] = res[h][p];
          const uint2 cbias[2] = {rbias[0], rbias[1]};  // prefetched with the residual
          if (c + 1 < c1) load_res(col + 32);  // prefetch the next chunk
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            // stage 16 raw fp32 accumulator columns of this thread's row
            float4* srow = reinterpret_cast<float4*>(stg + lane * C::STG_PITCH);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              srow[j] = make_float4(__uint_as_float(r[16 * h + 4 * j]), __uint_as_float(r[16 * h + 4 * j + 1]),
                                    __uint_as_float(r[16 * h + 4 * j + 2]), __uint_as_float(r[16 * h + 4 * j + 3]));
            if (h == 1 && !more) release();
            __syncwarp();
            const float4 bq = tc::bf16x4_to_f4(cbias[h]);
#pragma unroll
            for (int p = 0; p < C::QROWS / 8; ++p) {
              const int lr = p * 8 + cr;
              const int row = rbase + lr;
              const float4 a = *reinterpret_cast<const float4*>(stg + lr * C::STG_PITCH + cq * 16);
              if (row < M) {
                float4 o;
                o.x = cur[h][p].x + (a.x + bq.x);
                o.y = cur[h][p].y + (a.y + bq.y);
                o.z = cur[h][p].z + (a.z + bq.z);
                o.w = cur[h][p].w + (a.w + bq.w);
                *reinterpret_cast<float4*>(res_base + (size_t)row * epi.ldo + col + h * 16 + cq * 4) = o;
              }
            }
            __syncwarp();
          }
        } else {
          // bias (+ GELU) in the row layout, bf16 to the staging buffer, then
          // whole-row-segment stores
          float v[32];
          if (F8) {
            // E4M3 weights carry one scale per output column: 8 columns at a
            // time, so that scales and biases do not hold 64 registers
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              float sv[8], bb[8];
              Vec<float, 8>::load(epi.wscale + col + 8 * g, sv);
              if (epi.bias) {
                Vec<bf16, 8>::load(static_cast<const bf16*>(epi.bias) + col + 8 * g, bb);
              } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) bb[i] = 0.f;
              }
#pragma unroll
              for (int i = 0; i < 8; ++i) v[8 * g + i] = fmaf(__uint_as_float(r[8 * g + i]), sv[i], bb[i]);
            }
          } else {
            if (epi.bias) {
              const uint32_t* bw = reinterpret_cast<const uint32_t*>(bpre);
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const float2 b2 = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&bw[i]));
                f32x2_unpack(f32x2_add(f32x2_pack(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])),
                                       f32x2_pack(b2.x, b2.y)),
                             v[2 * i], v[2 * i + 1]);
              }
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
            }
            // the next chunk's bias loads while this chunk is converted and stored
            if (c + 1 < c1) load_bias(col + 32);
          }
          if (EK == tc::BF16OUT_SILU) {
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = silu(v[i]);
          } else if (epi.mode == LAZYMAR_EPI_GELU) {
#pragma unroll
            for (int i = 0; i < 16; ++i) gelu_erf_x2(v[2 * i], v[2 * i + 1]);
          }
          uint4 pk[4];
          {
            uint32_t* w = reinterpret_cast<uint32_t*>(pk);
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = pack_bf16(v[2 * i], v[2 * i + 1]);
          }
          if (PIPE && more) tld(c + 1);
          if (!more) release();
          if (tma_out) {
            // the previous chunk's store must have read the staging buffer
            if (lane == 0) bulk_wait_read();
            __syncwarp();
          }
          // row `lane`, 16-byte block j at block j ^ ((lane >> 1) & 3): the
          // TMA 64-byte swizzle of a 32 x 32 bf16 box
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint4*>(stg + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) = pk[j];
          if (tma_out) {
            // one TMA store of the 32 x 32 chunk; rows beyond M are clipped
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0 && rbase < M) {
              const int part = epi.mode == LAZYMAR_EPI_QKV ? col / epi.D : 0;
              const CUtensorMap* tm = part == 0 ? &tmO0 : part == 1 ? &tmO1 : &tmO2;
              tma_store_2d(tm, stg, col - part * epi.D, rbase);
              bulk_commit();
            }
          } else {
            __syncwarp();
#pragma unroll
            for (int p = 0; p < C::QROWS / 8; ++p) {
              const int lr = p * 8 + cr;
              const int row = rbase + lr;
              const uint4 val = *reinterpret_cast<const uint4*>(stg + lr * 64 + ((cq ^ ((lr >> 1) & 3)) << 4));
              if (row < M) *reinterpret_cast<uint4*>(tc::out_row(epi, row, col) + cq * 8) = val;
            }
            __syncwarp();
          }
        }
      }
    }
    if (tma_out && lane == 0) bulk_wait_all();  // stores complete before the CTA exits
  }
  __syncthreads();
  if (PAIR) cluster_sync();  // neither CTA leaves while the other may arrive on its barriers or use its operands
  if (warp == 1) {
    tc_fence_after();
    if (PAIR)
      tmem_dealloc_pair(tmem_base, C::TMEM_COLS);
    else
      tmem_dealloc(tmem_base, C::TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// fp32 CUDA-core kernel: 64 x 64 tile, 256 threads, 4 x 4 outputs per thread
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) gemm_f32_kernel(const float* __restrict__ A, const float* __restrict__ W, int M,
                                                       int N, int K, GemmEpi epi) {
  __shared__ float As[16][64 + 4];
  __shared__ float Ws[16][64 + 4];
  pdl_wait();
  pdl_trigger();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int idx = threadIdx.x + i * 256;
      const int r = idx >> 4, c = idx & 15;
      As[c][r] = (m0 + r < M && k0 + c < K) ? A[(size_t)(m0 + r) * K + k0 + c] : 0.f;
      Ws[c][r] = (n0 + r < N && k0 + c < K) ? W[(size_t)(n0 + r) * K + k0 + c] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = As[kk][ty * 4 + i];
        b[i] = Ws[kk][tx * 4 + i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  const int col = n0 + tx * 4;
  if (col >= N) return;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = m0 + ty * 4 + i;
    if (row < M) epilogue_apply<float, 4>(epi, row, col, acc[i]);
  }
}

// fp32, few tiles: the 64 x 64 tiles of the fp32 configuration's GEMMs leave
// most SMs idle and each runs its whole K in series (fc2 at M = 40: 4 CTAs, 64
// K steps of two barriers each). Here a CTA owns a TS x TS tile (16 or 32) and
// its NW warps split K; each warp computes the whole tile over its slice (TS /
// 8 rows x TS / 4 columns per lane, float4 along K from its own staged chunk, the next chunk's
// loads in flight meanwhile), and the partial tiles are summed in warp order
// through shared memory. Measured,
// against the 64 x 64 tiles (us): 40 x 768 x 256 13.0 -> 2.5, 40 x 256 x 1024
// 47.6 -> 5.3, 160 x 1024 x 256 13.2 -> 6.6, 640 x 256 x 1024 48.8 -> 21.2
constexpr int kF32Chunk = 32;               // K per staged chunk
constexpr int kF32Pitch = kF32Chunk + 4;    // floats: rows 16 bytes apart in banks
template <int NW, int TS>
constexpr int kF32Smem = NW * 2 * TS * kF32Pitch * (int)sizeof(float);

template <int NW, int TS>
__global__ void __launch_bounds__(NW * 32, NW == 8 || TS == 16 ? 2 : 1) gemm_f32_splitk_kernel(const float* __restrict__ A,
                                                                  const float* __restrict__ W, int M, int N, int K,
                                                                  GemmEpi epi) {
  extern __shared__ __align__(16) float f32_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.y * TS, n0 = blockIdx.x * TS;
  constexpr int P = TS / 4, RI = TS / 8, CJ = TS / 4;  // load passes; rows and columns of a lane
  float* sA = f32_smem + warp * (2 * TS * kF32Pitch);
  float* sW = sA + TS * kF32Pitch;
  const int slice = ((K / 4 + NW - 1) / NW) * 4;
  const int k0 = min(warp * slice, K), k1 = min(k0 + slice, K);
  // chunk loads: passes of 4 rows x 8 float4
  const int lr = lane >> 3, lk = (lane & 7) * 4;
  float4 ra[P], rw[P];
  auto fetch = [&](const float* src, int r0, int rows, int k, float4 (&r)[P]) {
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const int row = r0 + p * 4 + lr;
      r[p] = row < rows && k + lk < k1 ? *reinterpret_cast<const float4*>(src + (size_t)row * K + k + lk)
                                       : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  if (k0 < k1) fetch(W, n0, N, k0, rw);  // weights: no kernel writes them
  pdl_wait();
  pdl_trigger();
  if (k0 < k1) fetch(A, m0, M, k0, ra);
  float acc[RI][CJ] = {};
  const int ry = lane >> 2, cx = lane & 3;  // this lane's rows ry + 8 i and columns cx + 4 j: no bank conflicts
  for (int k = k0; k < k1; k += kF32Chunk) {
    __syncwarp();
#pragma unroll
    for (int p = 0; p < P; ++p) {
      *reinterpret_cast<float4*>(sA + (p * 4 + lr) * kF32Pitch + lk) = ra[p];
      *reinterpret_cast<float4*>(sW + (p * 4 + lr) * kF32Pitch + lk) = rw[p];
    }
    __syncwarp();
    if (k + kF32Chunk < k1) {
      fetch(W, n0, N, k + kF32Chunk, rw);
      fetch(A, m0, M, k + kF32Chunk, ra);
    }
#pragma unroll 2
    for (int kk = 0; kk < kF32Chunk; kk += 4) {
      float4 a[RI], w;
#pragma unroll
      for (int i = 0; i < RI; ++i) a[i] = *reinterpret_cast<const float4*>(sA + (ry + 8 * i) * kF32Pitch + kk);
#pragma unroll
      for (int j = 0; j < CJ; ++j) {
        w = *reinterpret_cast<const float4*>(sW + (cx + 4 * j) * kF32Pitch + kk);
#pragma unroll
        for (int i = 0; i < RI; ++i) {
          acc[i][j] = fmaf(a[i].x, w.x, acc[i][j]);
          acc[i][j] = fmaf(a[i].y, w.y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, w.z, acc[i][j]);
          acc[i][j] = fmaf(a[i].w, w.w, acc[i][j]);
        }
      }
    }
  }
  // partial tiles over the chunk buffers, then NW-term sums
  __syncthreads();
  float* part = f32_smem;
#pragma unroll
  for (int i = 0; i < RI; ++i)
#pragma unroll
    for (int j = 0; j < CJ; ++j) part[(warp * TS + ry + 8 * i) * kF32Pitch + cx + 4 * j] = acc[i][j];
  __syncthreads();
  const int row = threadIdx.x / (TS / 4), col = (threadIdx.x % (TS / 4)) * 4;
  if (threadIdx.x < TS * TS / 4 && m0 + row < M && n0 + col < N) {
    float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const float4 q = *reinterpret_cast<const float4*>(part + (w * TS + row) * kF32Pitch + col);
      v[0] += q.x; v[1] += q.y; v[2] += q.z; v[3] += q.w;
    }
    epilogue_apply<float, 4>(epi, m0 + row, n0 + col, v);
  }
}

template <int NW, int TS>
static cudaError_t launch_f32_splitk(const Ctx& c, const float* A, const float* W, int M, int N, int K,
                                     const GemmEpi& epi) {
  static int attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    const cudaError_t e = cudaFuncSetAttribute(gemm_f32_splitk_kernel<NW, TS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               kF32Smem<NW, TS>);
    if (e != cudaSuccess) return e;
    attr_set[dev] = 1;
  }
  return launch_pdl(gemm_f32_splitk_kernel<NW, TS>, dim3((N + TS - 1) / TS, (M + TS - 1) / TS), dim3(NW * 32),
                    (size_t)kF32Smem<NW, TS>, c.stream, A, W, M, N, K, epi);
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// 2-D tensor map over a row-major [outer, inner] matrix with the given row
// pitch, box [box_outer, box_inner], out-of-bounds elements read as zero.
static bool make_tmap_2d(CUtensorMapDataType dt, CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer,
                         uint64_t pitch_bytes, uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz) {
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {pitch_bytes};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t es[2] = {1, 1};
  return enc(m, dt, 2, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool make_tmap_bf16(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer, uint64_t pitch_bytes,
                    uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz) {
  return make_tmap_2d(CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, m, base, inner, outer, pitch_bytes, box_inner, box_outer, swz);
}

bool gemm_supported(int dtype, int M, int N, int K, const GemmEpi& epi, const char** why) {
  if (M < 0 || N <= 0 || K <= 0) { *why = "M >= 0, N > 0, K > 0 required"; return false; }
  if (epi.mode < LAZYMAR_EPI_BIAS || epi.mode > LAZYMAR_EPI_SILU) { *why = "unknown epilogue"; return false; }
  if (epi.mode == LAZYMAR_EPI_QKV && (epi.D <= 0 || N != 3 * epi.D)) { *why = "QKV epilogue needs N = 3D"; return false; }
  if (epi.gate && (epi.mode != LAZYMAR_EPI_RESIDUAL || epi.ldg < N || epi.ldg % 4 != 0)) {
    *why = "a gate needs the residual epilogue and ldg >= N, ldg % 4 == 0"; return false;
  }
  if (dtype == LAZYMAR_E4M3) {
    if (K % 128 != 0) { *why = "E4M3 GEMM needs K % 128 == 0"; return false; }
    if (N % 128 != 0) { *why = "E4M3 GEMM needs N % 128 == 0"; return false; }
    if (epi.mode == LAZYMAR_EPI_RESIDUAL || epi.mode == LAZYMAR_EPI_SILU) {
      *why = "E4M3 GEMM: bias, GELU or Q/K/V epilogue only"; return false;
    }
    if (!epi.wscale) { *why = "E4M3 GEMM needs the per-column weight scales"; return false; }
    if (epi.mode == LAZYMAR_EPI_QKV && epi.D % 32 != 0) { *why = "QKV epilogue needs D % 32 == 0"; return false; }
    if (epi.mode != LAZYMAR_EPI_QKV && epi.ldo % 8 != 0) { *why = "ldo % 8 == 0 required"; return false; }
  } else if (dtype == LAZYMAR_BF16) {
    if (K % 64 != 0) { *why = "bf16 GEMM needs K % 64 == 0"; return false; }
    if (N % 128 != 0) { *why = "bf16 GEMM needs N % 128 == 0"; return false; }
    if (epi.mode == LAZYMAR_EPI_QKV && epi.D % 32 != 0) { *why = "QKV epilogue needs D % 32 == 0"; return false; }
    if (epi.mode != LAZYMAR_EPI_QKV && epi.ldo % 8 != 0) { *why = "ldo % 8 == 0 required"; return false; }
  } else if (dtype == LAZYMAR_F32) {
    if (K % 4 != 0 || N % 4 != 0) { *why = "f32 GEMM needs K % 4 == 0 and N % 4 == 0"; return false; }
    if (epi.mode == LAZYMAR_EPI_QKV && epi.D % 4 != 0) { *why = "QKV epilogue needs D % 4 == 0"; return false; }
    if (epi.mode != LAZYMAR_EPI_QKV && epi.ldo % 4 != 0) { *why = "ldo % 4 == 0 required"; return false; }
  } else {
    *why = "unknown dtype";
    return false;
  }
  return true;
}

// How `base` tiles of width bn run on `slots` CTAs or pairs: `whole` of them at
// full width, the others, a last round that would leave slots idle, as `split`
// tiles each (equal parts of a multiple of 32 columns, at least 64). Returns
// the cost of all rounds, `time` being a full-width round's.
//
// A round of split tiles takes these parts of a full one, measured in per cent
// (half, third and quarter width): residual kinds 68, 56, 60 below K = 2048 and
// 50 above; bf16 outputs 80, -, 70 on pairs and 83, -, 75 on single CTAs.
// Measured, one launch of equal tiles -> with a split last round (us). Pairs: M
// = 20480, width 768: fc2 69.1 -> 65.3; width 1024: fc2 111.3 -> 104.7; M = 5440,
// width 1024: fc2 44.4 -> 38.4. Single CTAs: out at M = 20480,
// width 768 32.6 -> 29.6, M = 5440, width 1024 18.0 -> 14.6, M = 6400 19.1 -> 16.2;
// fc1 at M = 1600, width 768 12.5 -> 10.7, width 1024 15.2 -> 14.0. Not with bf16 outputs
// of single CTAs at K < 512 from four rounds on, where the kernel that can split
// costs more than the round it shortens (M = 40960, N = 1024, GELU: K = 64 27.0 -> 28.3, 192
// 28.7 -> 30.4, 320 30.7 -> 32.1; but 20480 x 1024 x 512 21.0 -> 20.1).
static long rounds_cost(long base, long slots, int bn, long time, bool pair, bool resid, int K, int* whole,
                        int* split) {
  const long rounds = base / slots, rem = base - rounds * slots;
  *whole = (int)base;
  *split = 1;
  if (rem == 0) return rounds * time;
  long best = time;
  if (rounds > 0 && !(!pair && !resid && K < 512 && rounds >= 4))
    for (int s = 2; s <= 4; ++s) {
      if (bn % (32 * s) != 0 || bn / s < 64) continue;
      const long pct = resid ? (s == 2 ? 68 : s == 3 ? 56 : K < 2048 ? 60 : 50)
                             : (s == 2 ? (pair ? 80 : 83) : (pair ? 70 : 75));
      const long t = (rem * s + slots - 1) / slots * (time * pct / 100);
      if (t < best) {
        best = t;
        *whole = (int)(rounds * slots);
        *split = s;
      }
    }
  return rounds * time + best;
}

// Whether the kernel of these tiles has a form that splits its last round. Single
// CTAs have a kernel of their own for it: a tile width known only at run time
// costs short launches 2 to 5 % (out at M = 1600, width 768: 5.6 against 5.8 us).
constexpr bool can_split(int bn, int ek, bool f8, bool pair) {
  return pair || (bn == 256 && !f8 && (ek == tc::BF16OUT || ek == tc::RESID_WIDE));
}

template <int BN, int EK, int BK, int F8 = 0, int PAIR = 0, int ROWS = 128>
static cudaError_t launch_tc(const Ctx& c, const void* A, const void* W, int M, int N, int K, const GemmEpi& epi) {
  using C = tc::Cfg<BN, EK, BK, F8, PAIR, ROWS>;
  const CUtensorMapDataType dt = F8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  CUtensorMap ta, tb;
  if (!make_tmap_2d(dt, &ta, A, (uint64_t)K, (uint64_t)M, (uint64_t)K * C::EB, C::ATOM_E, ROWS,
                    CU_TENSOR_MAP_SWIZZLE_128B) ||
      !make_tmap_2d(dt, &tb, W, (uint64_t)K, (uint64_t)N, (uint64_t)K * C::EB, C::ATOM_E, C::B_ROWS,
                    CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  constexpr bool CAN_SPLIT = can_split(BN, EK, F8 != 0, PAIR != 0);
  const auto kernel = gemm_bf16_tc_kernel<BN, EK, BK, F8, PAIR, ROWS, PAIR != 0>;
  const auto split_kernel = gemm_bf16_tc_kernel<BN, EK, BK, F8, PAIR, ROWS, CAN_SPLIT>;
  static int attr_set[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 0 && dev < 64 && !attr_set[dev]) {
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e == cudaSuccess && CAN_SPLIT)
      e = cudaFuncSetAttribute(split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
    if (e != cudaSuccess) return e;
    attr_set[dev] = 1;
  }
  // bf16 outputs leave through TMA stores of 32 x 32 boxes (64-byte swizzle),
  // except Q/K/V with a row map, whose K/V rows are scattered
  CUtensorMap to[3];
  std::memset(to, 0, sizeof to);
  int tma_out = 0;
  if (tc::is_bf16out<EK>() && !(epi.mode == LAZYMAR_EPI_QKV && epi.row_map)) {
    tma_out = 1;
    if (epi.mode == LAZYMAR_EPI_QKV) {
      const void* outs[3] = {epi.out, epi.k_out, epi.v_out};
      for (int i = 0; i < 3; ++i)
        if (!make_tmap_bf16(&to[i], outs[i], (uint64_t)epi.D, (uint64_t)M, (uint64_t)epi.D * 2, 32, C::QROWS,
                            CU_TENSOR_MAP_SWIZZLE_64B))
          return cudaErrorInvalidValue;
    } else if (!make_tmap_bf16(&to[0], epi.out, (uint64_t)N, (uint64_t)M, (uint64_t)epi.ldo * 2, 32, C::QROWS,
                               CU_TENSOR_MAP_SWIZZLE_64B)) {
      return cudaErrorInvalidValue;
    }
  }
  constexpr int TM = PAIR ? 2 * tc::BM : ROWS;
  const int base = ((M + TM - 1) / TM) * (N / BN), slots = PAIR ? c.num_sms / 2 : c.num_sms;
  int whole = base, split = 1;
  if (CAN_SPLIT) rounds_cost(base, slots, BN, 100, PAIR, !tc::is_bf16out<EK>(), K, &whole, &split);
  CUtensorMap tbt = tb;
  if (split > 1 && !make_tmap_2d(dt, &tbt, W, (uint64_t)K, (uint64_t)N, (uint64_t)K * C::EB, C::ATOM_E,
                                 C::B_ROWS / split, CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  const int tiles = whole + (base - whole) * split;
  const int grid = tiles < slots ? tiles : slots;
  if (PAIR)
    return launch_pdl_cluster(kernel, dim3(2 * grid), dim3(C::THREADS), C::SMEM, 2, c.stream, ta, tb, to[0], to[1], to[2],
                              tbt, whole, split, tma_out, M, N, K, epi, c.err);
  return launch_pdl(split > 1 ? split_kernel : kernel, dim3(grid), dim3(C::THREADS), C::SMEM, c.stream, ta, tb,
                    to[0], to[1], to[2], tbt, whole, split, tma_out, M, N, K, epi, c.err);
}

// Added to a tile width: tiles of 256 rows on CTA pairs; of 64 rows.
constexpr int kPair = 1000, kRows64 = 2000;

// Relative time of one round of tiles of width bn on single CTAs, measured: a
// narrower tile does proportionally less work per pipeline stage and runs well
// below the 256-wide rate, least so with the fp32-residual epilogue over long K
// (fc2), whose cost follows the width. 64-wide tiles win only where 128-wide
// ones fit in one round with SMs to spare. (M = 3200, width 768, two rounds of
// 192 or 256 wide Q/K/V tiles: 10.8 and 12.2 us; M = 40960, width 1024: 34, 51
// and 26 rounds of 192, 128 and 256 in 194, 237 and 176 us.)
enum { T_BF16, T_RESID, T_RESID_HALF, T_OTHER };  // bf16 out, residual below and from K = 2048, gated / SiLU / E4M3
static int tile_time(int bn, int kind) {
  static const int t[4][4] = {{256, 225, 180, 153}, {256, 224, 167, 153}, {256, 199, 153, 110}, {256, 243, 187, 153}};
  return t[kind][bn == 256 ? 0 : bn == 192 ? 1 : bn == 128 ? 2 : 3];
}

// Tile width with the fewest rounds of tiles over the SMs x the time of one
// tile; kPair + width for tiles of 256 rows on CTA pairs.
//
// A pair's round is shorter than a single CTA's of the same width, because an
// SM fills and reads 256 instead of 384 operand rows per K step (measured, us
// per round: Q/K/V at K = 768 4.7 against 5.5, fc2 at K = 3072 17.5 against
// 20.3, 14.8 against 16.3 at width 192), but a launch of pairs costs about 1.5 us
// more, which is 54000 / K of the unit (1 / 256 of a single CTA's 256-wide
// round). Whole GEMMs, one CTA -> pairs (us): M = 20480, width 768: Q/K/V 55.3 ->
// 46.8, fc1 68.9 -> 67.5, fc2 81.5 -> 70.2; M = 40960, width 1024: Q/K/V 169.8 ->
// 148.1, fc1 226.9 -> 201.0, fc2 228.8 -> 211.0. The out-projection, bound by its
// residual rows, stays on single CTAs (width 1024, with split last rounds: M =
// 17408 42.6 against 44.5, M = 40960 86.8 against 89.0; width 768 8.2 against 9.2 a
// round). Where the 256-row tiles need more rounds single CTAs win too (M = 3200,
// width 768: Q/K/V 11.9 against 13.5, fc2 15.1 against 19.1), and where 256-wide tiles
// of single CTAs fit in one round, which is the shorter the fewer SMs work in it
// (single against pairs, fc2: width 768, M = 5120 21.8 : 23.2, 6400 23.5 : 24.1; width
// 1024, M = 2560 25.6 : 26.6, 4500 27.9 : 28.1; width 1280, M = 2240 30.1 : 31.5, 3200 31.0 :
// 32.1; and 3 to 10 % with bf16 outputs), except for a nearly full round of long K (width
// 1024, M = 4864 30.0 : 28.8; width 1280, M = 3500 34.8 : 33.1, 3840 36.1 : 33.8).
static int choose_bn(const Ctx& c, int dtype, int M, int N, const GemmEpi& epi, int K) {
  const long mt = (M + tc::BM - 1) / tc::BM;
  const bool resid = epi.mode == LAZYMAR_EPI_RESIDUAL;
  const bool resid_half = resid && !epi.gate && K >= 2048;
  // kinds of tile_time; the first two have a kernel that splits the last round
  const bool plain = dtype == LAZYMAR_BF16 && epi.mode != LAZYMAR_EPI_SILU && !epi.gate;
  const int kind = resid_half ? T_RESID_HALF : !plain ? T_OTHER : resid ? T_RESID : T_BF16;
  const int widths[4] = {256, 192, 128, 64};
  int bn = 128;
  long best = -1;
  for (int i = 0; i < 4; ++i) {
    if (N % widths[i] != 0) continue;
    const long tiles = mt * (N / widths[i]), time = tile_time(widths[i], kind);
    int whole, split;
    const long t = widths[i] == 256 && (kind == T_BF16 || kind == T_RESID)
                       ? rounds_cost(tiles, c.num_sms, 256, time, false, resid, K, &whole, &split)
                       : (tiles + c.num_sms - 1) / c.num_sms * time;
    if (best < 0 || t < best) {
      best = t;
      bn = widths[i];
    }
  }
  const long single = N % 256 == 0 ? mt * (N / 256) : c.num_sms + 1L;  // 256-wide tiles of single CTAs
  if (plain && kind != T_RESID && (single > c.num_sms || (K >= 4096 && single * 12 >= 11L * c.num_sms))) {
    const long pt = (mt + 1) / 2, pairs = c.num_sms / 2;
    auto consider = [&](int width, int time) {
      if (pairs < 1 || N % width != 0) return;
      int whole, split;
      const long t = rounds_cost(pt * (N / width), pairs, width, time, true, resid, K, &whole, &split) + 54000 / K;
      if (t < best) {
        best = t;
        bn = kPair + width;
      }
    };
    // short K with GELU: the epilogue takes a larger part of a round (fc1 at width
    // 768, pairs against single CTAs (us): M = 5632 22.9 : 21.7, 6144 24.5 : 23.4,
    // 7680 29.0 : 28.2, but 12800 43.6 : 45.0)
    consider(256, resid_half ? 219 : epi.mode == LAZYMAR_EPI_GELU && K < 1024 ? 243 : 236);
    if (resid_half) consider(192, 186);
  }
  // Few rows: 64 x 64 tiles while they fit in one round. Measured, 128 x 64 tiles ->
  // 64 x 64 (us): M = 50, width 768: out 4.5 -> 3.9, fc2 10.6 -> 8.8; M = 320 fc2
  // 11.3 -> 9.0; M = 200, width 1024: out 5.2 -> 4.5, fc2 13.9 -> 11.2; the diffusion
  // head's sampling of 128 tokens 9.74 -> 8.64 ms
  if (dtype == LAZYMAR_BF16 && K % 128 == 0 && (long)((M + 63) / 64) * (N / 64) <= c.num_sms)
    bn = kRows64 + 64;
  // Residual kinds whose 128 x 128 tiles occupy at most half of the SMs: 64 x
  // 128 tiles (M = 1600, width 768: out 6.6 -> 5.6 us, fc2 13.3 -> 12.4)
  else if (bn == 128 && dtype == LAZYMAR_BF16 && resid && !epi.gate && K % 128 == 0 &&
           (long)((M + 63) / 64) * (N / 128) <= c.num_sms)
    bn = kRows64 + 128;
  return bn;
}

static int epi_kind(const GemmEpi& epi, int K) {
  return epi.mode == LAZYMAR_EPI_SILU       ? tc::BF16OUT_SILU
         : epi.mode != LAZYMAR_EPI_RESIDUAL ? tc::BF16OUT
         : epi.gate                          ? tc::RESID_WIDE_GATED
         : K < 2048                          ? tc::RESID_WIDE
                                             : tc::RESID_HALF;
}

// The bf16 tiles of launch_gemm's automatic choice: rows (256: on CTA pairs) and
// width of a tile, the tiles at full width, the parts of each of the others.
void gemm_tiles(int num_sms, int M, int N, int K, const GemmEpi& epi, int* rows, int* width, int* whole, int* split) {
  const Ctx c{nullptr, nullptr, num_sms};
  const int bn = choose_bn(c, LAZYMAR_BF16, M, N, epi, K);
  *rows = bn >= kRows64 ? 64 : bn >= kPair ? 256 : 128;
  *width = bn % kPair;
  const int base = (M + *rows - 1) / *rows * (N / *width);
  const bool pair = *rows == 256;
  *whole = base;
  *split = 1;
  if (*rows >= 128 && can_split(*width, epi_kind(epi, K), false, pair))
    rounds_cost(base, pair ? num_sms / 2 : num_sms, *width, 100, pair, epi.mode == LAZYMAR_EPI_RESIDUAL, K, whole, split);
}

static cudaError_t launch_bn(const Ctx& c, int dtype, const void* A, const void* W, int M, int N, int K,
                             const GemmEpi& epi, int bn) {
  if (dtype == LAZYMAR_E4M3) {
    // E4M3 operands (bf16-output kinds): a 128-element stage is one atom; the
    // tile width follows the bf16 choice
    if (bn == 256) return launch_tc<256, tc::BF16OUT, 128, 1>(c, A, W, M, N, K, epi);
    if (bn == 192) return launch_tc<192, tc::BF16OUT, 128, 1>(c, A, W, M, N, K, epi);
    return launch_tc<128, tc::BF16OUT, 128, 1>(c, A, W, M, N, K, epi);
  }
  const int ek = epi_kind(epi, K);
  if (bn == kRows64 + 128) {
    if (ek == tc::RESID_WIDE) return launch_tc<128, tc::RESID_WIDE, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
    return launch_tc<128, tc::RESID_HALF, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
  }
  if (bn == kRows64 + 64) {
    if (ek == tc::RESID_WIDE) return launch_tc<64, tc::RESID_WIDE, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_WIDE_GATED) return launch_tc<64, tc::RESID_WIDE_GATED, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_HALF) return launch_tc<64, tc::RESID_HALF, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::BF16OUT_SILU) return launch_tc<64, tc::BF16OUT_SILU, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
    return launch_tc<64, tc::BF16OUT, 128, 0, 0, 64>(c, A, W, M, N, K, epi);
  }
  if (bn == kPair + 192) return launch_tc<192, tc::RESID_HALF, 64, 0, 1>(c, A, W, M, N, K, epi);
  if (bn == kPair + 256) {
    if (ek == tc::RESID_HALF) return launch_tc<256, tc::RESID_HALF, 64, 0, 1>(c, A, W, M, N, K, epi);
    return launch_tc<256, tc::BF16OUT, 64, 0, 1>(c, A, W, M, N, K, epi);
  }
  if (bn == 192) {
    if (ek == tc::RESID_WIDE) return launch_tc<192, tc::RESID_WIDE, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_WIDE_GATED) return launch_tc<192, tc::RESID_WIDE_GATED, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_HALF) return launch_tc<192, tc::RESID_HALF, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::BF16OUT_SILU) return launch_tc<192, tc::BF16OUT_SILU, 64>(c, A, W, M, N, K, epi);
    return launch_tc<192, tc::BF16OUT, 64>(c, A, W, M, N, K, epi);
  }
  if (bn == 256) {
    if (ek == tc::RESID_WIDE) return launch_tc<256, tc::RESID_WIDE, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_WIDE_GATED) return launch_tc<256, tc::RESID_WIDE_GATED, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_HALF) return launch_tc<256, tc::RESID_HALF, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::BF16OUT_SILU) return launch_tc<256, tc::BF16OUT_SILU, 64>(c, A, W, M, N, K, epi);
    return launch_tc<256, tc::BF16OUT, 64>(c, A, W, M, N, K, epi);
  }
  if (bn == 64) {
    if (K % 128 == 0) {
      if (ek == tc::RESID_WIDE) return launch_tc<64, tc::RESID_WIDE, 128>(c, A, W, M, N, K, epi);
      if (ek == tc::RESID_WIDE_GATED) return launch_tc<64, tc::RESID_WIDE_GATED, 128>(c, A, W, M, N, K, epi);
      if (ek == tc::RESID_HALF) return launch_tc<64, tc::RESID_HALF, 128>(c, A, W, M, N, K, epi);
      if (ek == tc::BF16OUT_SILU) return launch_tc<64, tc::BF16OUT_SILU, 128>(c, A, W, M, N, K, epi);
      return launch_tc<64, tc::BF16OUT, 128>(c, A, W, M, N, K, epi);
    }
    if (ek == tc::RESID_WIDE) return launch_tc<64, tc::RESID_WIDE, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_WIDE_GATED) return launch_tc<64, tc::RESID_WIDE_GATED, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_HALF) return launch_tc<64, tc::RESID_HALF, 64>(c, A, W, M, N, K, epi);
    if (ek == tc::BF16OUT_SILU) return launch_tc<64, tc::BF16OUT_SILU, 64>(c, A, W, M, N, K, epi);
    return launch_tc<64, tc::BF16OUT, 64>(c, A, W, M, N, K, epi);
  }
  if (K % 128 == 0) {
    if (ek == tc::RESID_WIDE) return launch_tc<128, tc::RESID_WIDE, 128>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_WIDE_GATED) return launch_tc<128, tc::RESID_WIDE_GATED, 128>(c, A, W, M, N, K, epi);
    if (ek == tc::RESID_HALF) return launch_tc<128, tc::RESID_HALF, 128>(c, A, W, M, N, K, epi);
    if (ek == tc::BF16OUT_SILU) return launch_tc<128, tc::BF16OUT_SILU, 128>(c, A, W, M, N, K, epi);
    return launch_tc<128, tc::BF16OUT, 128>(c, A, W, M, N, K, epi);
  }
  if (ek == tc::RESID_WIDE) return launch_tc<128, tc::RESID_WIDE, 64>(c, A, W, M, N, K, epi);
  if (ek == tc::RESID_WIDE_GATED) return launch_tc<128, tc::RESID_WIDE_GATED, 64>(c, A, W, M, N, K, epi);
  if (ek == tc::RESID_HALF) return launch_tc<128, tc::RESID_HALF, 64>(c, A, W, M, N, K, epi);
  if (ek == tc::BF16OUT_SILU) return launch_tc<128, tc::BF16OUT_SILU, 64>(c, A, W, M, N, K, epi);
  return launch_tc<128, tc::BF16OUT, 64>(c, A, W, M, N, K, epi);
}

// fp32: tile width, and the warps that split K of the narrower tiles.
//
// 16 x 16 tiles while 32 x 32 ones would leave half of the SMs idle (40 x 256 x 1024:
// 5.3 against 11.7 us); 16 warps rather than 8 for K > 512 while the tiles leave SMs
// idle too (160 x 768 x 1024 12.3 against 14.2 us, but 160 x 1024 x 1024 23.3 : 21.2 and
// 640 x 768 x 768 44.6 : 31.2); 64 x 64 tiles from four per SM on, and before that where
// they take less time by the estimates below, in ns, fitted to M = 1..10000, N = 64..20000
// and K = 4..2048. A splitting warp works on chunks of 32, so a slice of K shorter
// than that saves nothing: 1280 x 768 x 64 21.2 against 9.0 us in 64 x 64 tiles, 2400 x
// 768 x 768 90 : 82, but 2560 x 768 x 256 38.3 : 48.3.
enum { F32_64, F32_32_8, F32_32_16, F32_16_8, F32_16_16 };
static int choose_f32(const Ctx& c, int M, int N, int K) {
  const long sms = c.num_sms;
  const long t64 = (long)((M + 63) / 64) * ((N + 63) / 64), t32 = (long)((M + 31) / 32) * ((N + 31) / 32);
  if (t64 > 4 * sms) return F32_64;
  if (t32 * 2 <= sms) return K > 512 ? F32_16_16 : F32_16_8;
  const bool w16 = K > 512 && t32 <= sms;
  const long k = K, slices = w16 ? 512 : 256;  // K of one chunk in every warp
  const double split = 2500 + t32 * 152.0 / sms * (3.7 + 0.0625 * ((k + slices - 1) / slices * slices));
  const double wide = t64 <= sms           ? 2000 + 45.0 * k
                      : t64 * 3 <= sms * 4 ? 3000 + 77.0 * k
                      : t64 <= 3 * sms     ? 3000 + 103.0 * k
                                           : 4000 + 175.0 * k;
  if (wide < 0.9375 * split) return F32_64;
  return w16 ? F32_32_16 : F32_32_8;
}

cudaError_t launch_gemm(const Ctx& c, int dtype, const void* A, const void* W, int M, int N, int K,
                        const GemmEpi& epi, int flags) {
  if (M == 0) return cudaSuccess;
  if (dtype == LAZYMAR_F32) {
    const float *a = static_cast<const float*>(A), *w = static_cast<const float*>(W);
    switch (choose_f32(c, M, N, K)) {
      case F32_64:
        return launch_pdl(gemm_f32_kernel, dim3((N + 63) / 64, (M + 63) / 64), dim3(256), 0, c.stream, a, w, M, N, K,
                          epi);
      case F32_32_8: return launch_f32_splitk<8, 32>(c, a, w, M, N, K, epi);
      case F32_32_16: return launch_f32_splitk<16, 32>(c, a, w, M, N, K, epi);
      case F32_16_8: return launch_f32_splitk<8, 16>(c, a, w, M, N, K, epi);
      default: return launch_f32_splitk<16, 16>(c, a, w, M, N, K, epi);
    }
  }
  if (flags == 2 && N % 256 == 0) return launch_bn(c, dtype, A, W, M, N, K, epi, 256);
  if (flags == 3 && N % 192 == 0) return launch_bn(c, dtype, A, W, M, N, K, epi, 192);
  if (flags == 4) return launch_bn(c, dtype, A, W, M, N, K, epi, 64);
  if (flags != 0) return launch_bn(c, dtype, A, W, M, N, K, epi, 128);
  return launch_bn(c, dtype, A, W, M, N, K, epi, choose_bn(c, dtype, M, N, epi, K));
}

}  // namespace lm
