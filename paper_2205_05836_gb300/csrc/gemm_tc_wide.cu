// Tensor-core contraction for Eq. 1 over more than 256 cut terms, on pairs of
// SMs (tcgen05 cta_group::2).
//
// Same split operands and products as the other tensor-core GEMMs (FP16 hi/lo,
// three products, power-of-two scales).  Every 64 values of k accumulate in a
// fresh TMEM accumulator (a "chunk", as in tc_gemm_kernel), cross products
// first and hi x hi last, so that only the last four MMAs of a chunk are cut
// off at the chunk's full size; the chunks are added in registers with
// round-to-nearest.  Chunks of 128 values took 3% less time (129 us against
// 133, below) but lost more than tc_gemm_kernel on terms of one sign: 4.6e-7
// of the outputs on uniform operands over 1024 terms where that kernel loses
// 3.5e-7 and this order 1.8e-7 (attributed tensors: 2.8e-7, 4.1e-7, 1.8e-7).
//
// With more than four 64-wide k-blocks an SM cannot keep its rows of A, so
// both operands stream, and what bounds a tile is how many operand bytes an
// SM takes in per multiply-add: a 128 x 128 tile of one SM (tc_gemm_kernel)
// needs 64 KB per k-block of 12 MMAs of 64 cycles, 85 bytes per cycle, more
// than the L2 delivers to every SM at once.  Here a pair computes 256 x 256
// (M = 256, N = 256 per instruction): each CTA loads its 128 rows of A and
// its 128 rows of B, 64 KB per 12 MMAs of 128 cycles.
//
// Shared memory: rings of 32 KB slots (A and B of one k-block, one plane).
// A k-block's cross products come before its hi x hi products, so its lo
// plane is free again before its hi plane: four hi slots and three lo slots
// use the shared memory that three whole stages of 64 KB would leave.
// Tensor memory: two accumulators of 256 columns (all 512).
//
// Roles (both CTAs): warp 8 lane 0 loads; warp 9 lane 0 of CTA 0 issues the
// MMAs; warps 0-7 drain: warp w takes rows 32 (w % 4) .. +31 of its CTA and
// columns 128 (w / 4) .. +127 of the tile, 128 float32 totals per thread.
// Register stores as in tc_pair_gemm_kernel: the launcher takes this kernel
// only for outputs whose low three column bits are the low three output bits.
// Barriers and bounded waits as in tc_pair_gemm_kernel.
// 2^12 x 2^13 outputs of 1024 terms (GB300): 133 us (1.55 PFLOP/s of executed
// products, 0.82 of the bf16 burst rate), tc_gemm_kernel 186; 2^13 x 2^14 495
// against 649; 2^12 x 2^12 of 4096 terms 252 against 524.
#include "internal.cuh"
#include "contract.cuh"
#include "tc_ptx.cuh"

#include <algorithm>
#include <mutex>
#include <set>

namespace cutqc {

namespace {

using namespace tc;

constexpr int BM = 128, BN = 256, BNH = 128, BK = 64;    // rows of A, columns (both CTAs), rows of B per CTA, k per block
constexpr int HI_SLOTS = 4, LO_SLOTS = 3;
constexpr int OPERAND_BYTES = 128 * BK * 2;              // 16 KiB: one operand's plane of a k-block
constexpr int SLOT_BYTES = 2 * OPERAND_BYTES;            // A and B
constexpr int NBUF = 2;
constexpr int TMEM_COLS = NBUF * BN;                     // 512
constexpr int NUM_THREADS = 320, EPI_WARPS = 8, EPI_COLS = 128;

struct WideMaps {
  CUtensorMap a_hi, a_lo, b_hi, b_lo;   // [rows][Kp] fp16, box 64 x 128, 128B swizzle
};

struct WideArgs {
  const float* sa;
  const float* sb;
  int64_t M, N;
  int num_kb;
  const int* num_kb_dev;   // nullable: k-blocks in use, read on the device (<= num_kb)
  int64_t num_mb, num_tiles;
  float alpha;
  uint64_t mask_m, mask_n;
  float* out;
  double* sum;
  int* status;
};

struct Tail {
  uint64_t hi_full[HI_SLOTS], lo_full[LO_SLOTS];     // CTA 0: both CTAs' loads of a slot landed
  uint64_t hi_empty[HI_SLOTS], lo_empty[LO_SLOTS];   // each CTA: its slot may be refilled
  uint64_t cfull[NBUF];      // each CTA: accumulator holds a finished chunk
  uint64_t cempty[NBUF];     // CTA 0: both CTAs' epilogues read the accumulator
  uint64_t fin;              // CTA 0: every MMA finished
  uint32_t tmem_slot;
  int abort_flag;
};

constexpr size_t kSmemBytes = 1024 + (size_t)(HI_SLOTS + LO_SLOTS) * SLOT_BYTES + sizeof(Tail);
static_assert(kSmemBytes <= 232448, "shared memory budget");

// kind::f16, A = B = F16, D = F32, both K-major, N = 256, M = 256.
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);

// kDirect64: 64 consecutive columns are 64 consecutive floats (else 8)
template <bool kDirect64>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
tc_wide_gemm_kernel(const __grid_constant__ WideMaps maps, const __grid_constant__ WideArgs args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* hi_smem = smem;
  uint8_t* lo_smem = smem + HI_SLOTS * SLOT_BYTES;
  Tail* tail = reinterpret_cast<Tail*>(smem + (HI_SLOTS + LO_SLOTS) * SLOT_BYTES);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int64_t pair = blockIdx.x >> 1, num_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < HI_SLOTS; ++s) {
      mbar_init(smem_u32(&tail->hi_full[s]), 1);
      mbar_init(smem_u32(&tail->hi_empty[s]), 1);
    }
    for (int s = 0; s < LO_SLOTS; ++s) {
      mbar_init(smem_u32(&tail->lo_full[s]), 1);
      mbar_init(smem_u32(&tail->lo_empty[s]), 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(smem_u32(&tail->cfull[b]), 1);
      mbar_init(smem_u32(&tail->cempty[b]), 2 * EPI_WARPS);
    }
    mbar_init(smem_u32(&tail->fin), 1);
    tail->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tail->tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();           // both CTAs' barriers are initialised before any remote use
  tc_fence_after();
  grid_dependency_wait();   // the operands' preparation
  const int num_kb = args.num_kb_dev ? max(1, min(args.num_kb, __ldg(args.num_kb_dev))) : args.num_kb;
  const uint32_t tmem_base = tail->tmem_slot;
  volatile int* abort_flag = &tail->abort_flag;
  auto fail = [&]() {
    *abort_flag = 1;
    record_status(args.status, CUTQC_ETIMEOUT);
  };

  if (warp == 8) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      bool hi_used[HI_SLOTS] = {}, lo_used[LO_SLOTS] = {};
      uint32_t hi_par[HI_SLOTS] = {}, lo_par[LO_SLOTS] = {};
      int hs = 0, ls = 0;
      uint32_t hp = 0, lp = 0;
      bool ok = true;
      for (int64_t tile = pair; tile < args.num_tiles && ok && !*abort_flag; tile += num_pairs) {
        int arow = (int)((tile % args.num_mb) * 2 * BM) + (int)rank * BM;
        int brow = (int)((tile / args.num_mb) * BN) + (int)rank * BNH;
        if (arow >= args.M) arow = 0;     // rows and columns beyond the output are never stored
        if (brow >= args.N) brow = 0;
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait(smem_u32(&tail->hi_empty[hs]), hp ^ 1u, abort_flag)) { fail(); ok = false; break; }
          {
            uint8_t* st = hi_smem + hs * SLOT_BYTES;
            const uint32_t full = map_to_rank(smem_u32(&tail->hi_full[hs]), 0);
            if (rank == 0) mbar_expect_tx(smem_u32(&tail->hi_full[hs]), 2 * SLOT_BYTES);
            tma_load_pair(smem_u32(st), &maps.a_hi, kb * BK, arow, full);
            tma_load_pair(smem_u32(st + OPERAND_BYTES), &maps.b_hi, kb * BK, brow, full);
            hi_used[hs] = true;
            hi_par[hs] = hp;
            if (++hs == HI_SLOTS) { hs = 0; hp ^= 1u; }
          }
          if (!mbar_wait(smem_u32(&tail->lo_empty[ls]), lp ^ 1u, abort_flag)) { fail(); ok = false; break; }
          {
            uint8_t* st = lo_smem + ls * SLOT_BYTES;
            const uint32_t full = map_to_rank(smem_u32(&tail->lo_full[ls]), 0);
            if (rank == 0) mbar_expect_tx(smem_u32(&tail->lo_full[ls]), 2 * SLOT_BYTES);
            tma_load_pair(smem_u32(st), &maps.a_lo, kb * BK, arow, full);
            tma_load_pair(smem_u32(st + OPERAND_BYTES), &maps.b_lo, kb * BK, brow, full);
            lo_used[ls] = true;
            lo_par[ls] = lp;
            if (++ls == LO_SLOTS) { ls = 0; lp ^= 1u; }
          }
        }
      }
      // every copy this CTA started has landed, and been read, before it
      // exits (the loads complete on CTA 0's barriers, which this thread
      // cannot wait on)
      for (int s = 0; s < HI_SLOTS; ++s)
        if (hi_used[s] && !mbar_wait(smem_u32(&tail->hi_empty[s]), hi_par[s], nullptr))
          record_status(args.status, CUTQC_ETIMEOUT);
      for (int s = 0; s < LO_SLOTS; ++s)
        if (lo_used[s] && !mbar_wait(smem_u32(&tail->lo_empty[s]), lo_par[s], nullptr))
          record_status(args.status, CUTQC_ETIMEOUT);
    }
  } else if (warp == 9) {
    // ----------------------------------------------------------- MMA issue
    if (lane == 0 && rank == 0) {
      const uint64_t hi_desc0 = sw128_desc(smem_u32(hi_smem)), lo_desc0 = sw128_desc(smem_u32(lo_smem));
      constexpr uint64_t kSlotStep = SLOT_BYTES >> 4, kBStep = OPERAND_BYTES >> 4;   // in the descriptors' 16-byte units
      int hs = 0, ls = 0, buf = 0;
      uint32_t hp = 0, lp = 0, bp = 0;
      bool ok = true, any = false;
      for (int64_t tile = pair; tile < args.num_tiles && ok && !*abort_flag; tile += num_pairs) {
        for (int kb = 0; kb < num_kb; ++kb) {
          if (!mbar_wait(smem_u32(&tail->cempty[buf]), bp ^ 1u, abort_flag) ||
              !mbar_wait(smem_u32(&tail->hi_full[hs]), hp, abort_flag) ||
              !mbar_wait(smem_u32(&tail->lo_full[ls]), lp, abort_flag)) { fail(); ok = false; break; }
          tc_fence_after();
          const uint32_t d = tmem_base + (uint32_t)(buf * BN);
          const uint64_t ah = hi_desc0 + (uint64_t)hs * kSlotStep, al = lo_desc0 + (uint64_t)ls * kSlotStep;
          // the cross products free the lo slot, then hi x hi the hi slot
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            // 16 values of k: 32 bytes inside the swizzle rows
            const uint64_t o = (uint64_t)(kk * 2);
            umma_pair_ss(d, ah + o, al + kBStep + o, kIdesc, kk ? 1u : 0u);
            umma_pair_ss(d, al + o, ah + kBStep + o, kIdesc, 1u);
          }
          any = true;
          umma_commit_mc(smem_u32(&tail->lo_empty[ls]), 0x3);
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint64_t o = (uint64_t)(kk * 2);
            umma_pair_ss(d, ah + o, ah + kBStep + o, kIdesc, 1u);
          }
          umma_commit_mc(smem_u32(&tail->hi_empty[hs]), 0x3);
          if (++hs == HI_SLOTS) { hs = 0; hp ^= 1u; }
          if (++ls == LO_SLOTS) { ls = 0; lp ^= 1u; }
          umma_commit_mc(smem_u32(&tail->cfull[buf]), 0x3);
          if (++buf == NBUF) { buf = 0; bp ^= 1u; }
        }
      }
      // all MMAs this thread issued complete before tensor memory is freed
      if (any) {
        umma_commit_mc(smem_u32(&tail->fin), 0x1);
        if (!mbar_wait(smem_u32(&tail->fin), 0, nullptr)) record_status(args.status, CUTQC_ETIMEOUT);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    const int g = warp & 3, h = warp >> 2;
    int buf = 0;
    uint32_t bp = 0;
    double local = 0.0;
    const float sbg = __ldg(args.sb);
    // a warp's deposit of a value all its lanes share (see tc_pair_gemm_kernel)
    const uint64_t mplace = pdep64((uint64_t)1 << lane, args.mask_m);
    const uint64_t nplace = pdep64((uint64_t)1 << lane, args.mask_n);
    const uint64_t rlane = pdep64((uint64_t)(lane >> 2), args.mask_m);
    auto deposit = [&](uint64_t v, uint64_t place) -> uint64_t {
      const uint64_t mine = ((v >> lane) & 1) ? place : 0;
      return ((uint64_t)__reduce_or_sync(0xffffffffu, (unsigned)(mine >> 32)) << 32) |
             __reduce_or_sync(0xffffffffu, (unsigned)mine);
    };
    const uint64_t m3 = __shfl_sync(0xffffffffu, mplace, 3), m4 = __shfl_sync(0xffffffffu, mplace, 4);
    // output offsets of column bits 3 .. 6
    int64_t gofs[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) gofs[i] = (int64_t)__shfl_sync(0xffffffffu, nplace, 3 + i);
    // totals: [64-column half][16-row half][pair]; pair 2 q + r: row
    // 16 h2 + lane / 4 + 8 r, columns 64 c + 8 q + 2 (lane % 4) + {0, 1}
    unsigned long long tot[2][2][16];
    bool ok = true;
    for (int64_t tile = pair; tile < args.num_tiles && ok && !*abort_flag; tile += num_pairs) {
#pragma unroll
      for (int i = 0; i < 64; ++i) tot[i >> 5][(i >> 4) & 1][i & 15] = 0ull;
#pragma unroll 1
      for (int kb = 0; kb < num_kb; ++kb) {
        if (!mbar_wait(smem_u32(&tail->cfull[buf]), bp, abort_flag)) { fail(); ok = false; break; }
        tc_fence_after();
        __syncwarp();
        const uint32_t taddr = tmem_base + ((uint32_t)(g * 32) << 16) + (uint32_t)(buf * BN + h * EPI_COLS);
        // 32 columns of 16 rows at a time: 16 registers beside the totals
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              uint32_t r[16];
              tmem_ld16x256_x4(taddr + (uint32_t)(64 * c + 32 * e) + ((uint32_t)(16 * h2) << 16), r);
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int i = 0; i < 8; ++i)
                tot[c][h2][8 * e + i] = fadd2(tot[c][h2][8 * e + i], pack2(r[2 * i], r[2 * i + 1]));
            }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) remote_arrive(map_to_rank(smem_u32(&tail->cempty[buf]), 0));
        if (++buf == NBUF) { buf = 0; bp ^= 1u; }
      }
      if (!ok) break;
      const int64_t mrow0 = (tile % args.num_mb) * 2 * BM + (int64_t)rank * BM + g * 32;
      const int64_t n0 = (tile / args.num_mb) * BN + h * EPI_COLS;
      const uint64_t rbase = deposit((uint64_t)mrow0, mplace) | rlane;
      float* obase = args.out + (rbase | deposit((uint64_t)n0, nplace)) + 2 * (lane & 3);
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int64_t m = mrow0 + (lane >> 2) + 16 * h2 + 8 * r;
          if (m >= args.M) continue;
          const unsigned long long rs = pair2(args.alpha * __ldg(args.sa + m) * sbg);
          float* orow = obase + ((r ? m3 : 0) | (h2 ? m4 : 0));
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            if (n0 + 64 * c >= args.N) break;
            float* grp[8];
            grp[0] = orow + (c ? gofs[3] : 0);
#pragma unroll
            for (int q = 1; q < 8; ++q)
              grp[q] = kDirect64 ? grp[0] + 8 * q : grp[q & (q - 1)] + (q & 1 ? gofs[0] : q & 2 ? gofs[1] : gofs[2]);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              if (n0 + 64 * c + 8 * q < args.N) {
                unsigned long long& v = tot[c][h2][2 * q + r];
                v = fmul2(v, rs);
                __stcs(reinterpret_cast<float2*>(grp[q]), unpack2(v));
              }
            }
          }
          // the total: the row's 32 outputs in float32 in a tree (N is a
          // multiple of 64 when a thread's columns end inside the tile),
          // float64 across rows and tiles; one float32 sum over the four rows
          // was up to 3e-6 off
          if (args.sum) {
            unsigned long long part[2] = {0ull, 0ull};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
              if (n0 + 64 * c >= args.N) break;
#pragma unroll
              for (int w = 4; w > 0; w /= 2)
#pragma unroll
                for (int q = 0; q < w; ++q)
                  tot[c][h2][2 * q + r] = fadd2(tot[c][h2][2 * q + r], tot[c][h2][2 * (q + w) + r]);
              part[c] = tot[c][h2][r];
            }
            const float2 f = unpack2(fadd2(part[0], part[1]));
            local += (double)(f.x + f.y);
          }
        }
    }
    __syncwarp();
    if (args.sum) {
      for (int off = 16; off; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
      if (lane == 0) atomicAdd(args.sum, local);
    }
  }

  // Both CTAs reach this point only after their roles ended: CTA 0's MMAs
  // have completed, every chunk was read, every copy landed.
  tc_fence_before();
  __syncthreads();
  cluster_sync();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

int make_map(CUtensorMap* map, const __half* base, int64_t rows, int64_t Kp) {
  auto enc = get_encode();
  if (!enc) return set_error(CUTQC_ECUDA, "cuTensorMapEncodeTiled unavailable");
  if (((uintptr_t)base & 15) != 0) return set_error(CUTQC_EINVAL, "operand not 16-byte aligned");
  cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)Kp * sizeof(__half)};
  cuuint32_t box[2] = {(cuuint32_t)BK, 128};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(CUTQC_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return CUTQC_OK;
}

}  // namespace

bool tc_wide_supported(int64_t M, int64_t N, int64_t Kp, uint64_t mask_m, uint64_t mask_n, const float* out) {
  return Kp > 256 && Kp % BK == 0 && Kp / BK <= kWideMaxKb && M >= kWideMinSide && N >= kWideMinSide &&
         ((M + 127) / 128) * ((N + 127) / 128) > sm_count() && M < ((int64_t)1 << 30) && N < ((int64_t)1 << 30) &&
         (mask_n & 7) == 7 && (mask_m & mask_n) == 0 && ((uintptr_t)out & 7) == 0;
}

int launch_tc_wide_gemm(const TcOperand& a, const TcOperand& b, int64_t Kp, float alpha, uint64_t mask_m,
                        uint64_t mask_n, float* out, double* sum, cudaStream_t st, const int* num_kb_dev) {
  WideMaps maps;
  int rc;
  if ((rc = make_map(&maps.a_hi, a.hi, a.rows, Kp))) return rc;
  if ((rc = make_map(&maps.a_lo, a.lo, a.rows, Kp))) return rc;
  if ((rc = make_map(&maps.b_hi, b.hi, b.rows, Kp))) return rc;
  if ((rc = make_map(&maps.b_lo, b.lo, b.rows, Kp))) return rc;
  WideArgs args{};
  args.sa = a.scale;
  args.sb = b.scale;
  args.M = a.rows;
  args.N = b.rows;
  args.num_kb = (int)(Kp / BK);
  args.num_kb_dev = num_kb_dev;
  args.num_mb = (a.rows + 2 * BM - 1) / (2 * BM);
  args.num_tiles = args.num_mb * ((b.rows + BN - 1) / BN);
  args.alpha = alpha;
  args.mask_m = mask_m;
  args.mask_n = mask_n;
  args.out = out;
  args.sum = sum;
  args.status = device_status_ptr();
  {
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      CUTQC_CUDA_TRY(cudaFuncSetAttribute(tc_wide_gemm_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kSmemBytes));
      CUTQC_CUDA_TRY(cudaFuncSetAttribute(tc_wide_gemm_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)kSmemBytes));
      done.insert(dev);
    }
  }
  const int grid = (int)(2 * std::min<int64_t>(args.num_tiles, std::max(1, sm_count() / 2)));
  const auto kernel = (mask_n & 63) == 63 ? tc_wide_gemm_kernel<true> : tc_wide_gemm_kernel<false>;
  CUTQC_CUDA_TRY(launch_dependent(kernel, dim3(grid), dim3(NUM_THREADS), kSmemBytes, st, maps, args));
  CUTQC_LAUNCH_CHECK("tc_wide_gemm_kernel");
  return CUTQC_OK;
}

}  // namespace cutqc
