// Tensor-core contraction for Eq. 1 on pairs of SMs (tcgen05 cta_group::2).
//
// Same products as tc_gemm_kernel (FP16 hi/lo split operands, three
// products, power-of-two row / operand scales), for K <= 256 (four 64-wide
// k-blocks).  Each 128 values of k accumulate in a fresh TMEM accumulator
// ("chunk", 24 MMAs), cross products (hi x lo, lo x hi) first and hi x hi
// last: the tensor core rounds its FP32 accumulator toward zero, and only
// the last MMAs of a chunk do so at the chunk's full magnitude.  Chunks are
// added in registers with round-to-nearest.  (Modelled on the 30-qubit
// workload, this order with 128-wide chunks leaves a third of the bias of
// 64-wide chunks in product order: sum p error -3.6e-7 against -5.4e-7.)
// The kernel is organised to move fewer operand bytes per output:
//
// * a cluster of two CTAs on two SMs computes 256 x 128 output tiles with
//   one MMA stream (M = 256, N = 128, K = 16 per instruction): CTA r holds
//   A rows r*128 .. +127 and B rows r*64 .. +63 of the tile, the tensor core
//   reads both halves of B from both shared memories, and each CTA's tensor
//   memory receives its own 128 rows x 128 columns;
// * A stays resident: a pair takes a work item (one 256-row block of A and a
//   run of consecutive 128-column tiles) and keeps the CTA's A rows for all
//   k: A hi in tensor memory (written by the epilogue warps, read by two of
//   the three products), A lo in shared memory (one TMA load per item).
//   Only B streams (16 KiB per CTA per k-block, 5 stages), so a CTA moves 1
//   byte of operands per byte of output (4 for a 128 x 128 tile that streams
//   both operands).
// * one thread cannot issue N = 128 pair MMAs as fast as the tensor core
//   runs them, so two threads issue alternate chunks;
// * three 128-column accumulator buffers let the MMAs run two chunks (256
//   values of k) ahead of the epilogue.
//
// Tensor memory per CTA (512 columns): A hi [0, 128) (two fp16 values of k
// per 32-bit column), chunk accumulators at 128, 256, 384.
//
// Roles (both CTAs): warp 8 lane 0 loads B per k-block; lane 0 of warps 9
// and 10 of CTA 0 issue the MMAs (alternate chunks); warps 0-7 write A hi to
// tensor memory and load A lo at the start of an item, then drain the
// chunks, scale and store their CTA's rows.  Row-major outputs (out[m * N +
// n]) go straight from registers (16 x 256-bit tensor-memory loads give each
// quad of lanes 8 consecutive columns of a row: whole 32-byte sectors per
// store) -- staging them through shared memory would add 128 KiB of shared
// memory traffic per tile on top of the MMAs' operand reads and the B
// stream, more than the SM's shared memory bandwidth allows at the tensor
// rate.  Bit-deposit layouts whose low three column bits are the
// low three output bits store the same way (each quad's 8 columns are one
// 32-byte sector); the others go through a staged transpose that writes whole
// 128-byte lines.  The loads of both CTAs complete on CTA 0's
// barriers (it waits for both halves); MMA completion is multicast to the
// barriers of both CTAs; epilogue warps of both CTAs report A written and
// chunk buffers read on CTA 0's barriers.  Every wait is bounded; on expiry
// a CTA records CUTQC_ETIMEOUT, raises its abort flag and falls through to
// the common exit (a cluster barrier, then tensor memory is freed).
#include "internal.cuh"
#include "contract.cuh"
#include "tc_ptx.cuh"
#include "line_stores.cuh"

#include <algorithm>
#include <atomic>
#include <mutex>
#include <set>
#include <type_traits>

namespace cutqc {

namespace {

using namespace tc;

constexpr int BM = 128;                                  // A rows per CTA (256 per pair)
constexpr int BN = 128;                                  // output columns per tile
constexpr int BNH = BN / 2;                              // B rows per CTA
constexpr int BK = 64;                                   // k per block (128-byte rows)
constexpr int MAX_KB = 4;                                // resident A: k <= 256
constexpr int STAGES_MAX = 10;
constexpr int NBUF = 3;                                  // chunk buffers in TMEM
constexpr int KB_PER_CHUNK = 2;                          // 128 values of k per accumulator
constexpr int A_COLS = MAX_KB * BK / 2;                  // 128 TMEM columns of A hi
constexpr int ACC_COL0 = A_COLS;                         // first accumulator column
constexpr int A_KB_BYTES = BM * BK * 2;                  // 16 KiB: A lo, one k-block
constexpr int ALO_BYTES = MAX_KB * A_KB_BYTES;           // 64 KiB
constexpr int B_HALF = BNH * BK * 2;                     // 8 KiB
constexpr int STAGE_BYTES = 2 * B_HALF;                  // 16 KiB: B hi + lo, one k-block
constexpr int TMEM_COLS = 512;
static_assert(ACC_COL0 + NBUF * BN <= TMEM_COLS, "tensor memory budget");
constexpr int NUM_THREADS = 352;
constexpr int EPI_WARPS = 8;
constexpr int EPI_COLS = 64;                             // columns per epilogue warp
constexpr int kStaged = 0, kDirect64 = 1, kDirect8 = 2;  // store layouts (tc_pair_gemm_kernel)
constexpr int kStatBlockMax = 1, kStatAbsMax = 2;        // epilogue statistics (tc_pair_gemm_kernel)
constexpr int BLK_FLOATS = 32 * 32;                      // one 32 x 32 staging block
constexpr int EPI_STG_BYTES = EPI_WARPS * (EPI_COLS / 32) * BLK_FLOATS * 4;   // 64 KiB
// Direct stores need no staging block: its 64 KiB go to five more B stages,
// which keeps the B stream ahead of the MMAs while the output stream loads
// the memory system (4.27 -> 4.05 ms on the 32-qubit chain's last step).
template <bool kDirect> struct Cfg {
  static constexpr int STAGES = kDirect ? 10 : 5;
  static constexpr int STG = kDirect ? 0 : EPI_STG_BYTES;
};

struct PairMaps {
  CUtensorMap a_lo;         // [rows][Kp] fp16, box 64 x 128
  CUtensorMap b_hi, b_lo;   // [rows][Kp] fp16, box 64 x 64
};

struct PairArgs {
  const __half* a_hi;   // [M][Kp]
  int64_t Kp;
  const float* sa;
  const float* sb;
  int64_t M, N;
  int num_kb;
  const int* num_kb_dev;  // nullable: k-blocks in use, read on the device (<= num_kb)
  int num_mp;           // 256-row blocks of A
  int64_t num_nt;       // 128-column tiles
  int64_t tiles_per_item;   // 0: each pair takes one contiguous share of all tiles (Items)
  int64_t num_items;
  float alpha;
  uint64_t mask_m, mask_n;
  int n_contig;
  int m_low5;           // mask_m holds address bits 0..4 (rows 32-aligned are consecutive)
  uint64_t coff_lo[64]; // pdep(c, mask_n) for c < 64: column offsets inside a 64-aligned group
  uint64_t tile_step;   // pdep(BN, mask_n): one column tile further in the output offset
  LineStores lines;     // staged layouts: the walk of a 32 x 32 block in whole output lines
  float* out;
  double* sum;
  float* cmax;          // nullable: largest value of each 32-row x 64-column block of the output
  unsigned int* amax;   // nullable: largest |output| of the launch (float bits, atomicMax)
  int64_t cmax_cols;    // blocks per 32-row stripe: ceil(N / 64)
  int streaming;
  int* status;
};

struct Tail {
  uint64_t full[STAGES_MAX];     // CTA 0: both CTAs' B halves of a stage landed
  uint64_t empty[STAGES_MAX];    // each CTA: its stage may be refilled
  uint64_t cfull[NBUF];      // each CTA: chunk buffer holds a finished chunk
  uint64_t cempty[NBUF];     // CTA 0: both CTAs' epilogues read the buffer
  uint64_t afull;            // CTA 0: both CTAs wrote A hi to TMEM and their A lo landed
  uint64_t aempty;           // each CTA: both issuers are done with A
  uint64_t fin[2];           // CTA 0: every MMA of issuer j finished
  uint32_t tmem_slot;
  int abort_flag;
};

template <bool kDirect>
constexpr size_t smem_bytes() {
  return 1024 + ALO_BYTES + Cfg<kDirect>::STAGES * STAGE_BYTES + Cfg<kDirect>::STG + sizeof(Tail);
}
static_assert(smem_bytes<true>() <= 232448 && smem_bytes<false>() <= 232448, "shared memory budget");

// kind::f16, A = B = F16, D = F32, both K-major, N = 128, M = 256.
constexpr uint32_t kIdescPair = (1u << 4) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);

// D (TMEM) (+)= A (TMEM, both CTAs' rows) x B (shared memory, both CTAs' halves)
__device__ __forceinline__ void umma_pair_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(kIdescPair), "r"(accum)
      : "memory");
}
// 32 lanes x 32 columns of 32 bits from registers (lane = thread)
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// Arrive on CTA 0's barrier after writing tensor memory that CTA 0's MMAs
// read: cluster-scope release (once per work item).
__device__ __forceinline__ void remote_arrive_release_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// The work items of one pair: a 256-row block mp and its tiles [t0, t1).
// With tiles_per_item t, items are dealt out in turn, row blocks fastest, so
// that the pairs read the same B tiles at about the same time (through L2).
// With t = 0 the tiles (row block major) are cut into one contiguous share
// per pair: an exact balance and the fewest changes of A, for B operands that
// L2 holds whichever part of it a pair reads.
struct Items {
  int64_t cur, end, step;
  int mp;
  int64_t t0, t1;
  __device__ __forceinline__ Items(const PairArgs& a, int64_t pair, int64_t pairs) {
    if (a.tiles_per_item) {
      cur = pair;
      end = a.num_items;
      step = pairs;
    } else {
      const int64_t total = (int64_t)a.num_mp * a.num_nt;
      cur = total * pair / pairs;
      end = total * (pair + 1) / pairs;
      step = 0;
    }
  }
  __device__ __forceinline__ bool next(const PairArgs& a) {
    if (cur >= end) return false;
    if (step) {
      mp = (int)(cur % a.num_mp);
      t0 = (cur / a.num_mp) * a.tiles_per_item;
      t1 = t0 + a.tiles_per_item < a.num_nt ? t0 + a.tiles_per_item : a.num_nt;
      cur += step;
    } else {
      mp = (int)(cur / a.num_nt);
      t0 = cur - (int64_t)mp * a.num_nt;
      t1 = t0 + (end - cur) < a.num_nt ? t0 + (end - cur) : a.num_nt;
      cur += t1 - t0;
    }
    return true;
  }
};

// kLayout: how a tile is stored.  kDirect64: from registers, 64 consecutive
// columns are 64 consecutive floats; kDirect8: from registers, 8 consecutive
// columns are 8 consecutive floats (a 32-byte sector; the offsets of the
// eight groups come from coff_lo); kStaged: through shared memory.
// The 2^12 x 2^16 contraction over 256 terms in a qubit order whose low bits
// come in runs of three from either operand takes 300 us as kDirect8; through
// the staging with one 4-byte store per lane scattered over 32 sectors it
// took 906.
// kStat: 0 nothing more; kStatBlockMax: each epilogue warp's 32 x 64 block
// maximum per tile into args.cmax; kStatAbsMax: the largest |output| of the
// launch into *args.amax (float bits; the values are non-negative, so the
// integer max orders them).
template <int kLayout, int kStat>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
tc_pair_gemm_kernel(const __grid_constant__ PairMaps maps, const PairArgs args) {
  constexpr bool kRowMajor = kLayout != kStaged;
  constexpr int STAGES = Cfg<kRowMajor>::STAGES;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* alo_smem = smem;
  uint8_t* b_smem = smem + ALO_BYTES;
  float* stg_all = reinterpret_cast<float*>(smem + ALO_BYTES + STAGES * STAGE_BYTES);
  Tail* tail = reinterpret_cast<Tail*>(smem + ALO_BYTES + STAGES * STAGE_BYTES + Cfg<kRowMajor>::STG);
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cta_rank();
  const int64_t pair = blockIdx.x >> 1;
  const int64_t num_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&tail->full[s]), 1);
      mbar_init(smem_u32(&tail->empty[s]), 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(smem_u32(&tail->cfull[b]), 1);
      mbar_init(smem_u32(&tail->cempty[b]), 2 * EPI_WARPS);
    }
    mbar_init(smem_u32(&tail->afull), 2 * EPI_WARPS);
    mbar_init(smem_u32(&tail->aempty), 2);
    mbar_init(smem_u32(&tail->fin[0]), 1);
    mbar_init(smem_u32(&tail->fin[1]), 1);
    tail->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    // one warp of each CTA of the pair allocates, collectively
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
  // k-blocks in use: a count chosen on the device (cut-term pruning) when
  // given, never more than the operands hold
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
      bool issued[STAGES] = {};
      uint32_t issued_par[STAGES] = {};
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (Items it(args, pair, num_pairs); ok && !*abort_flag && it.next(args);) {
        const int64_t t0 = it.t0, t1 = it.t1;
        for (int64_t nt = t0; nt < t1 && ok; ++nt) {
          int brow = (int)(nt * BN) + (int)rank * BNH;
          if (brow >= args.N) brow = 0;     // columns beyond N are never stored
          for (int kb = 0; kb < num_kb; ++kb) {
            if (!mbar_wait(smem_u32(&tail->empty[stage]), phase ^ 1u, abort_flag)) { fail(); ok = false; break; }
            uint8_t* st = b_smem + stage * STAGE_BYTES;
            const uint32_t lead_full = map_to_rank(smem_u32(&tail->full[stage]), 0);
            if (rank == 0) mbar_expect_tx(smem_u32(&tail->full[stage]), 2 * STAGE_BYTES);
            tma_load_pair(smem_u32(st), &maps.b_hi, kb * BK, brow, lead_full);
            tma_load_pair(smem_u32(st + B_HALF), &maps.b_lo, kb * BK, brow, lead_full);
            issued[stage] = true;
            issued_par[stage] = phase;
            if (++stage == STAGES) { stage = 0; phase ^= 1u; }
          }
        }
      }
      // Every copy this CTA started completes on CTA 0's barriers, which
      // this thread cannot wait on; wait instead until the MMAs that read
      // them have finished (each stage's last use) before exiting.
      for (int s = 0; s < STAGES; ++s)
        if (issued[s] && !mbar_wait(smem_u32(&tail->empty[s]), issued_par[s], nullptr))
          record_status(args.status, CUTQC_ETIMEOUT);
    }
  } else if (warp == 9 || warp == 10) {
    // ----------------------------------------------------------- MMA issue
    // Two issuing threads: chunk c (KB_PER_CHUNK k-blocks of one tile,
    // counted over the whole kernel) is issued by thread c % 2 into
    // accumulator buffer c % NBUF; k-block g (counted over the whole kernel)
    // sits in stage g % STAGES.  Within a chunk the hi x lo and lo x hi
    // products go first and the hi x hi products last, so that only the
    // last MMAs truncate (round toward zero) at the chunk's full magnitude.
    const int j = warp - 9;
    if (lane == 0 && rank == 0) {
      uint32_t aphase = 0;
      int64_t c = 0, g = 0;
      bool ok = true;
      for (Items it(args, pair, num_pairs); ok && !*abort_flag && it.next(args);) {
        const int64_t t0 = it.t0, t1 = it.t1;
        if (!mbar_wait(smem_u32(&tail->afull), aphase, abort_flag)) { fail(); ok = false; break; }
        aphase ^= 1u;
        tc_fence_after();
        for (int64_t nt = t0; nt < t1 && ok; ++nt) {
          for (int kb0 = 0; kb0 < num_kb; kb0 += KB_PER_CHUNK, ++c) {
            const int nkb = num_kb - kb0 < KB_PER_CHUNK ? num_kb - kb0 : KB_PER_CHUNK;
            if ((int)(c & 1) != j) { g += nkb; continue; }
            const int buf = (int)(c % NBUF);
            const uint32_t buf_phase = (uint32_t)((c / NBUF) & 1);
            if (!mbar_wait(smem_u32(&tail->cempty[buf]), buf_phase ^ 1u, abort_flag)) { fail(); ok = false; break; }
            tc_fence_after();
            int stage[KB_PER_CHUNK];
            for (int q = 0; q < nkb && ok; ++q) {
              stage[q] = (int)((g + q) % STAGES);
              const uint32_t phase = (uint32_t)(((g + q) / STAGES) & 1);
              if (!mbar_wait(smem_u32(&tail->full[stage[q]]), phase, abort_flag)) { fail(); ok = false; }
            }
            if (!ok) break;
            tc_fence_after();
            const uint32_t d = tmem_base + (uint32_t)(ACC_COL0 + buf * BN);
            uint32_t accum = 0;
            for (int pass = 0; pass < 2; ++pass) {        // 0: cross products, 1: hi x hi
              for (int q = 0; q < nkb; ++q) {
                const int kb = kb0 + q;
                const uint32_t ah = tmem_base + (uint32_t)(kb * (BK / 2));
                const uint32_t al = smem_u32(alo_smem + kb * A_KB_BYTES);
                const uint32_t bh = smem_u32(b_smem + stage[q] * STAGE_BYTES), bl = bh + B_HALF;
#pragma unroll
                for (int kk = 0; kk < BK / 16; ++kk) {
                  // 16 values of k: 8 TMEM columns of A hi, 32 bytes inside the
                  // swizzle rows of A lo and B
                  const uint32_t ta = kk * 8, off = kk * 32;
                  const uint64_t dbh = sw128_desc(bh + off);
                  if (pass == 0) {
                    umma_pair_ts(d, ah + ta, sw128_desc(bl + off), accum);
                    umma_pair_ss(d, sw128_desc(al + off), dbh, kIdescPair, 1u);
                    accum = 1u;
                  } else {
                    umma_pair_ts(d, ah + ta, dbh, 1u);
                  }
                }
              }
            }
            for (int q = 0; q < nkb; ++q) umma_commit_mc(smem_u32(&tail->empty[stage[q]]), 0x3);
            umma_commit_mc(smem_u32(&tail->cfull[buf]), 0x3);
            g += nkb;
          }
        }
        if (ok) umma_commit_mc(smem_u32(&tail->aempty), 0x3);   // this issuer is done with A
      }
      // all MMAs this thread issued complete before tensor memory is freed
      umma_commit_mc(smem_u32(&tail->fin[j]), 0x1);
      if (!mbar_wait(smem_u32(&tail->fin[j]), 0, nullptr)) record_status(args.status, CUTQC_ETIMEOUT);
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // warp w: TMEM lanes 32*(w%4).. = tile rows, columns 64*(w/4) .. +63
    // At the start of an item, warp w also writes A hi rows 32*(w%4) .. +31
    // of the CTA's block, k-blocks kb with kb % 2 == w / 4, to tensor memory;
    // warp 0 lane 0 loads the CTA's A lo rows by TMA.
    const int g = warp & 3, h = warp >> 2;
    int buf = 0;
    uint32_t buf_phase = 0;
    uint32_t aphase = 0;
    double local = 0.0;
    [[maybe_unused]] float amx = 0.f;    // kStatAbsMax: this thread's largest |output|
    const float sbg = __ldg(args.sb);
    float* stg0 = stg_all + warp * (EPI_COLS / 32) * BLK_FLOATS;
    const uint32_t lead_afull = map_to_rank(smem_u32(&tail->afull), 0);
    // this thread's 64 outputs of a tile as packed pairs: the chunk sums, the
    // scaling and the total's partial sums are half the instructions (the
    // first chunk is taken as it is, not added to zeros); fewer issued
    // instructions are also less power for the MMAs, which the kernel shares
    // the card's limit with
    unsigned long long tot[EPI_COLS / 2];
    bool ok = true;
    static_assert(EPI_COLS == 64, "block maxima cover one warp's 32 rows x 64 columns");
    // the warp's block of a tile (rows row0 .. +31, columns col0 .. +63):
    // its largest value, for the top-T selection of the caller
    auto put_cmax = [&](float mx, int64_t row0, int64_t col0) {
      for (int off = 16; off; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      if (lane == 0 && row0 < args.M && col0 < args.N) args.cmax[(row0 >> 5) * args.cmax_cols + (col0 >> 6)] = mx;
    };
    // a warp's deposit of a value all its lanes share: lane j holds the place
    // of bit j (once per launch), the set bits' places are OR-reduced (the
    // bit-by-bit loop per item cost several thousand cycles at its start)
    const uint64_t mplace = pdep64((uint64_t)1 << lane, args.mask_m);
    const uint64_t nplace = pdep64((uint64_t)1 << lane, args.mask_n);
    const uint64_t rlane = kRowMajor ? pdep64((uint64_t)(lane >> 2), args.mask_m) : 0;   // row bits 0..2
    auto deposit = [&](uint64_t v, uint64_t place) -> uint64_t {      // v < 2^32
      const uint64_t mine = ((v >> lane) & 1) ? place : 0;
      return ((uint64_t)__reduce_or_sync(0xffffffffu, (unsigned)(mine >> 32)) << 32) |
             __reduce_or_sync(0xffffffffu, (unsigned)mine);
    };
    [[maybe_unused]] int64_t gofs[3] = {(int64_t)args.coff_lo[8], (int64_t)args.coff_lo[16], (int64_t)args.coff_lo[32]};
    if constexpr (kLayout == kDirect8) asm volatile("" : "+l"(gofs[0]), "+l"(gofs[1]), "+l"(gofs[2]));
    const uint64_t mplace3 = __shfl_sync(0xffffffffu, mplace, 3), mplace4 = __shfl_sync(0xffffffffu, mplace, 4);
    for (Items it(args, pair, num_pairs); ok && !*abort_flag && it.next(args);) {
      const int mp = it.mp;
      const int64_t t0 = it.t0, t1 = it.t1;
      const int64_t mrow0 = (int64_t)mp * 2 * BM + (int64_t)rank * BM + g * 32;
      const int64_t m = mrow0 + lane;
      const bool mvalid = m < args.M;
      // direct-store layout: this thread's rows mrow0 + lane/4 + 16 h2 + 8 rsel,
      // each with its scale and its output offset (the row bits deposited)
      const int64_t rtile0 = mrow0 + (lane >> 2);
      float rsv[4];
      int64_t rowoff[4];
      const uint64_t rbase = deposit((uint64_t)mrow0, mplace) | rlane;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int64_t mm = rtile0 + 16 * (i >> 1) + 8 * (i & 1);
        const bool v = kRowMajor && mm < args.M;
        rsv[i] = v ? args.alpha * __ldg(args.sa + mm) * sbg : 0.f;
        rowoff[i] = !v ? 0 : (int64_t)(rbase | ((i & 1) ? mplace3 : 0) | ((i >> 1) ? mplace4 : 0));
      }
      // ---- A rows of this item into tensor memory, once the previous
      // item's MMAs are done with the old ones
      if (!mbar_wait(smem_u32(&tail->aempty), aphase ^ 1u, abort_flag)) { fail(); ok = false; break; }
      aphase ^= 1u;
      tc_fence_after();
      if (warp == 0 && lane == 0) {
        // A lo rows of this CTA (CTA 1's rows may lie wholly beyond M: it then
        // loads rows from 0, which are never stored)
        int arow = mp * 2 * BM + (int)rank * BM;
        if (arow >= args.M) arow = 0;
        for (int kb = 0; kb < num_kb; ++kb)
          tma_load_pair(smem_u32(alo_smem + kb * A_KB_BYTES), &maps.a_lo, kb * BK, arow, lead_afull);
      }
      {
        const uint4* row = reinterpret_cast<const uint4*>(args.a_hi + (mvalid ? m : 0) * args.Kp);
        const uint32_t tbase = tmem_base + ((uint32_t)(g * 32) << 16);
        for (int kb = h; kb < num_kb; kb += 2) {
          uint32_t r[32];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            uint4 v = mvalid ? __ldg(row + kb * 8 + q) : make_uint4(0, 0, 0, 0);
            r[4 * q] = v.x;
            r[4 * q + 1] = v.y;
            r[4 * q + 2] = v.z;
            r[4 * q + 3] = v.w;
          }
          tmem_st32(tbase + (uint32_t)(kb * (BK / 2)), r);
        }
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        // CTA 0's warp 0 arrives with the byte count of both CTAs' A lo loads
        if (rank == 0 && warp == 0)
          mbar_expect_tx(smem_u32(&tail->afull), (uint32_t)(2 * num_kb * A_KB_BYTES));
        else
          remote_arrive_release_cluster(lead_afull);
      }
      // output offset of this warp's first column of a tile: deposited once
      // per item, then stepped in the deposited domain (adding pdep(BN) with
      // the bits between the mask's filled); depositing it per tile took 54
      // of 408 us at 2^28 outputs of 256 terms
      uint64_t cbase, cnext = args.n_contig ? 0 : deposit((uint64_t)(t0 * BN + h * EPI_COLS), nplace);
      for (int64_t nt = t0; nt < t1 && ok; ++nt) {
        if (args.n_contig) {
          cbase = (uint64_t)(nt * BN + h * EPI_COLS);
        } else {
          cbase = cnext;
          cnext = ((cbase | ~args.mask_n) + args.tile_step) & args.mask_n;
        }
        const int num_ch = (num_kb + KB_PER_CHUNK - 1) / KB_PER_CHUNK;
        // one chunk's accumulators into r0 (tile rows 0 .. 15 of the warp, or
        // columns 0 .. 31) and r1
        auto drain = [&](uint32_t (&r0)[32], uint32_t (&r1)[32]) -> bool {
          if (!mbar_wait(smem_u32(&tail->cfull[buf]), buf_phase, abort_flag)) { fail(); return false; }
          tc_fence_after();
          __syncwarp();
          const uint32_t taddr =
              tmem_base + ((uint32_t)(g * 32) << 16) + (uint32_t)(ACC_COL0 + buf * BN + h * EPI_COLS);
          if constexpr (kRowMajor) {
            // two 16-lane halves, 64 columns each: value 4 q + e of half h2 is
            // row g*32 + 16 h2 + lane/4 + 8 (e/2), column 8 q + 2 (lane%4) + e%2
            tmem_ld16x256_x8(taddr, r0);
            tmem_ld16x256_x8(taddr + (16u << 16), r1);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          } else {
            // thread = row: r0 holds columns 0 .. 31, r1 32 .. 63
            tmem_ld32(taddr, r0);
            tmem_ld32(taddr + 32, r1);
          }
          return true;
        };
        auto release = [&]() {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) remote_arrive(map_to_rank(smem_u32(&tail->cempty[buf]), 0));
          if (++buf == NBUF) { buf = 0; buf_phase ^= 1u; }
        };
        {
          uint32_t r0[32], r1[32];
          if (!drain(r0, r1)) { ok = false; break; }
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            tot[i] = pack2(r0[2 * i], r0[2 * i + 1]);
            tot[16 + i] = pack2(r1[2 * i], r1[2 * i + 1]);
          }
          release();
        }
#pragma unroll 1
        for (int ch = 1; ch < num_ch; ++ch) {
          uint32_t r0[32], r1[32];
          if (!drain(r0, r1)) { ok = false; break; }
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            tot[i] = fadd2(tot[i], pack2(r0[2 * i], r0[2 * i + 1]));
            tot[16 + i] = fadd2(tot[16 + i], pack2(r1[2 * i], r1[2 * i + 1]));
          }
          release();
        }
        if (!ok) break;
        const float rs = mvalid ? args.alpha * __ldg(args.sa + m) * sbg : 0.f;
        const int64_t nbase = nt * BN + h * EPI_COLS;
        if (kRowMajor) {
          // straight from registers: the column bits 0..5 (kDirect8: 0..2) are
          // address bits 0..5 (0..2), so the warp's 64 (8) columns of a row
          // are consecutive floats; per instruction the warp writes 8 rows x
          // 32 bytes (4 lanes per row), whole sectors; no staging through
          // shared memory, whose bandwidth the MMAs' operand reads and the B
          // stream already use
          const int64_t nb0 = nbase + 2 * (lane & 3);
          const int64_t cb = (int64_t)cbase + 2 * (lane & 3);
          unsigned long long part = 0ull;     // this thread's 64 outputs of the tile (two sums); float64 across tiles
          [[maybe_unused]] float mx = -INFINITY;
#pragma unroll
          for (int h2 = 0; h2 < 2; ++h2)
#pragma unroll
            for (int rsel = 0; rsel < 2; ++rsel) {
              const int64_t mm = rtile0 + 16 * h2 + 8 * rsel;
              const unsigned long long rsm = pair2(rsv[2 * h2 + rsel]);
              float* orow = args.out + rowoff[2 * h2 + rsel] + cb;
              // the row's eight groups of 8 columns: consecutive, or (kDirect8)
              // at sums of the three group bits' offsets, which stay in
              // registers (read from the parameters per store they cost 70 us
              // of 257 at 2^28 outputs of 64 terms)
              float* grp[EPI_COLS / 8];
              grp[0] = orow;
#pragma unroll
              for (int q = 1; q < EPI_COLS / 8; ++q)
                grp[q] = kLayout == kDirect64 ? orow + 8 * q
                                              : grp[q & (q - 1)] + (q & 1 ? gofs[0] : q & 2 ? gofs[1] : gofs[2]);
#pragma unroll
              for (int q = 0; q < EPI_COLS / 8; ++q) {
                const unsigned long long v = fmul2(tot[16 * h2 + 2 * q + rsel], rsm);
                if (mm < args.M && nb0 + 8 * q < args.N) {
                  const float2 f = unpack2(v);
                  __stcs(reinterpret_cast<float2*>(grp[q]), f);
                  part = fadd2(part, v);
                  if constexpr (kStat == kStatBlockMax) mx = fmaxf(mx, fmaxf(f.x, f.y));
                  if constexpr (kStat == kStatAbsMax) amx = fmaxf(amx, fmaxf(fabsf(f.x), fabsf(f.y)));
                }
              }
            }
          if (args.sum) {
            const float2 f = unpack2(part);
            local += (double)(f.x + f.y);
          }
          if constexpr (kStat == kStatBlockMax) put_cmax(mx, mrow0, nbase);
        } else {
          if (args.m_low5) {
            // the low 5 bits of the row index are the low 5 address bits:
            // for each column the warp's 32 rows are 32 consecutive floats
            // (thread = row), stored column by column without staging.
            // nbase is a multiple of 64, so pdep(nbase + c) = pdep(nbase) |
            // pdep(c), the second term a constant of the launch.
            float* const obase = args.out + (mvalid ? rbase | (uint64_t)lane : 0);
            float part = 0.f;
            [[maybe_unused]] float mx = -INFINITY;
#pragma unroll
            for (int c = 0; c < EPI_COLS; ++c) {
              if (nbase + c >= args.N) break;
              const float2 pr = unpack2(tot[c >> 1]);
              const float val = ((c & 1) ? pr.y : pr.x) * rs;
              if (mvalid) {
                float* ptr = obase + (cbase | args.coff_lo[c]);
                if (args.streaming) __stcs(ptr, val); else *ptr = val;
                part += val;
                if constexpr (kStat == kStatBlockMax) mx = fmaxf(mx, val);
                if constexpr (kStat == kStatAbsMax) amx = fmaxf(amx, fabsf(val));
              }
            }
            if (args.sum) local += (double)part;
            if constexpr (kStat == kStatBlockMax) put_cmax(mx, mrow0, nbase);
            continue;
          }
          // general bit deposit through the staging block: every store
          // instruction writes one whole 128-byte line (LineStores)
          [[maybe_unused]] float mx = -INFINITY;
#pragma unroll
          for (int q = 0; q < EPI_COLS / 32; ++q) {
            const int64_t n0 = nbase + q * 32;
            if (n0 >= args.N) break;
            float v[32];
#pragma unroll
            for (int c = 0; c < 32; c += 2) {
              const float2 pr = unpack2(tot[(q * 32 + c) >> 1]);
              v[c] = pr.x * rs;
              v[c + 1] = pr.y * rs;
            }
            float part = 0.f;
            store_block_lines(v, stg0 + q * BLK_FLOATS, args.lines, lane, mrow0, n0, args.M, args.N, args.mask_m,
                              args.mask_n, rbase | cbase | args.coff_lo[32 * q], args.out, args.streaming, [&](float val) {
                                part += val;
                                if constexpr (kStat == kStatBlockMax) mx = fmaxf(mx, val);
                                if constexpr (kStat == kStatAbsMax) amx = fmaxf(amx, fabsf(val));
                              });
            if (args.sum) local += (double)part;
          }
          if constexpr (kStat == kStatBlockMax) put_cmax(mx, mrow0, nbase);
        }
      }
    }
    __syncwarp();
    if (args.sum) {
      for (int off = 16; off; off >>= 1) local += __shfl_xor_sync(0xffffffffu, local, off);
      if (lane == 0) atomicAdd(args.sum, local);
    }
    if constexpr (kStat == kStatAbsMax) {
      for (int off = 16; off; off >>= 1) amx = fmaxf(amx, __shfl_xor_sync(0xffffffffu, amx, off));
      if (lane == 0) atomicMax(args.amax, __float_as_uint(amx));
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

int make_map(CUtensorMap* map, const __half* base, int64_t rows, int64_t Kp, int box_rows) {
  auto enc = get_encode();
  if (!enc) return set_error(CUTQC_ECUDA, "cuTensorMapEncodeTiled unavailable");
  if (((uintptr_t)base & 15) != 0) return set_error(CUTQC_EINVAL, "operand not 16-byte aligned");
  cuuint64_t dims[2] = {(cuuint64_t)Kp, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)Kp * sizeof(__half)};
  cuuint32_t box[2] = {(cuuint32_t)BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(CUTQC_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return CUTQC_OK;
}

// Column operands (hi and lo) up to this size are read from L2 wherever a
// pair's share of the tiles lies (129 MB of L2, the output streaming past):
// contiguous shares instead of dealt-out items, from four tiles per pair on.
// (With fewer a share that crosses a row block doubles the pair's A loads: 2^14 x
// 2^8 outputs of 256 terms 31 us with shares, 27 with items of two tiles; 2^16 x
// 2^8 79 and 82.)
constexpr int64_t kFlatMaxB = (int64_t)64 << 20;

// Tiles per work item set by cutqc_fd_set_tiles_per_item (0: chosen below).
std::atomic<int> g_tiles_per_item{0};

// Tiles per work item: the fewest tile slots on the busiest pair, counting
// an A load (the pipe drains, the new A block lands) as about two tiles of
// time.  (One tile undercounted it where tiles are short: the dense DD
// recursion's one-k-block GEMM, 1024 row blocks x 32 column tiles, ran 3%
// faster with whole-row-block items than with the 16-tile items that
// weight picked; the FD picks are the same under both.)  Items of one to three
// tiles only where a pair has fewer than four.
int64_t pick_tiles_per_item(int64_t num_mp, int64_t num_nt, int64_t pairs) {
  int64_t best_t = 1;
  double best = 1e300;
  for (int64_t t = num_mp * num_nt < 4 * pairs ? 1 : 4; t <= 64; ++t) {
    const int64_t items = num_mp * ((num_nt + t - 1) / t);
    const int64_t per_pair = (items + pairs - 1) / pairs;
    const double cost = (double)per_pair * ((double)std::min(t, num_nt) + 2.0);
    if (cost < best) { best = cost; best_t = t; }
  }
  return std::min(best_t, num_nt);
}

}  // namespace

bool tc_pair_supported(int64_t Kp) { return Kp > 0 && Kp % BK == 0 && Kp / BK <= MAX_KB; }

int set_pair_tiles_per_item(int t) {
  if (t < 0 || t > 4096) return set_error(CUTQC_EINVAL, "tiles per item must be in 0..4096");
  g_tiles_per_item.store(t, std::memory_order_relaxed);
  return CUTQC_OK;
}

int launch_tc_pair_gemm(const TcOperand& a, const TcOperand& b, int64_t Kp, float alpha, uint64_t mask_m,
                        uint64_t mask_n, float* out, double* sum, int streaming, cudaStream_t st,
                        const int* num_kb_dev, float* cmax, unsigned int* amax) {
  if (a.rows <= 0 || b.rows <= 0) return CUTQC_OK;
  if (!tc_pair_supported(Kp)) return set_error(CUTQC_EINVAL, "paired tensor-core K must be 64..256, a multiple of 64");
  if (a.rows >= ((int64_t)1 << 30) || b.rows >= ((int64_t)1 << 30)) return set_error(CUTQC_EUNSUPPORTED, "too many rows");
  PairMaps maps;
  int rc;
  if (((uintptr_t)a.hi & 15) != 0) return set_error(CUTQC_EINVAL, "operand not 16-byte aligned");
  if ((rc = make_map(&maps.a_lo, a.lo, a.rows, Kp, BM))) return rc;
  if ((rc = make_map(&maps.b_hi, b.hi, b.rows, Kp, BNH))) return rc;
  if ((rc = make_map(&maps.b_lo, b.lo, b.rows, Kp, BNH))) return rc;
  PairArgs args{};
  args.a_hi = a.hi;
  args.Kp = Kp;
  args.sa = a.scale;
  args.sb = b.scale;
  args.M = a.rows;
  args.N = b.rows;
  args.num_kb = (int)(Kp / BK);
  args.num_kb_dev = num_kb_dev;
  const int64_t num_mp = (a.rows + 2 * BM - 1) / (2 * BM);
  args.num_mp = (int)num_mp;
  args.num_nt = (b.rows + BN - 1) / BN;
  const int64_t pairs_avail = std::max(1, sm_count() / 2);
  const int forced = g_tiles_per_item.load(std::memory_order_relaxed);
  if (forced <= 0 && b.rows * Kp * 4 <= kFlatMaxB && num_mp * args.num_nt >= 4 * pairs_avail) {
    args.tiles_per_item = 0;
    args.num_items = num_mp * args.num_nt;
  } else {
    args.tiles_per_item = forced > 0 ? std::min<int64_t>(forced, args.num_nt)
                                     : pick_tiles_per_item(num_mp, args.num_nt, pairs_avail);
    args.num_items = num_mp * ((args.num_nt + args.tiles_per_item - 1) / args.tiles_per_item);
  }
  args.alpha = alpha;
  args.mask_m = mask_m;
  args.mask_n = mask_n;
  args.n_contig = mask_is_low(mask_n) ? 1 : 0;
  args.m_low5 = (mask_m & 31) == 31 ? 1 : 0;
  for (int c = 0; c < 64; ++c) args.coff_lo[c] = pdep64((uint64_t)c, mask_n);
  args.tile_step = pdep64((uint64_t)BN, mask_n);
  args.lines = line_stores(mask_m, mask_n);
  args.out = out;
  args.sum = sum;
  if (cmax && amax) return set_error(CUTQC_EINVAL, "internal: one epilogue statistic per launch");
  args.cmax = cmax;
  args.amax = amax;
  args.cmax_cols = (b.rows + 63) / 64;
  args.streaming = streaming;
  args.status = device_status_ptr();
  // direct 8-byte stores from registers when column bits 0..5 are output
  // address bits 0..5 (e.g. out[m * N + n] with N a multiple of 64, or an
  // intermediate whose lowest open digits come from the column operand), or
  // bits 0..2 are (whole 32-byte sectors per quad of lanes), and the base is
  // 8-byte aligned; fewer low column bits would split sectors between lanes
  const bool direct = (mask_n & 7) == 7 && (mask_m & mask_n) == 0 && ((uintptr_t)out & 7) == 0;
  const int layout = !direct ? kStaged : (mask_n & 63) == 63 ? kDirect64 : kDirect8;
  if (args.n_contig && ((uintptr_t)out & 15) != 0) return set_error(CUTQC_EINVAL, "output not 16-byte aligned");
  {
    static std::mutex mu;
    static std::set<int> done;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    if (!done.count(dev)) {
      const void* fns[9] = {
          (const void*)tc_pair_gemm_kernel<kStaged, 0>,   (const void*)tc_pair_gemm_kernel<kStaged, 1>,
          (const void*)tc_pair_gemm_kernel<kStaged, 2>,   (const void*)tc_pair_gemm_kernel<kDirect64, 0>,
          (const void*)tc_pair_gemm_kernel<kDirect64, 1>, (const void*)tc_pair_gemm_kernel<kDirect64, 2>,
          (const void*)tc_pair_gemm_kernel<kDirect8, 0>,  (const void*)tc_pair_gemm_kernel<kDirect8, 1>,
          (const void*)tc_pair_gemm_kernel<kDirect8, 2>};
      for (int i = 0; i < 9; ++i)
        CUTQC_CUDA_TRY(cudaFuncSetAttribute(fns[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)(i < 3 ? smem_bytes<false>() : smem_bytes<true>())));
      done.insert(dev);
    }
  }
  const int64_t pairs = std::min<int64_t>(args.num_items, pairs_avail);
  const int grid = (int)(2 * pairs);
  const int stat = cmax ? kStatBlockMax : amax ? kStatAbsMax : 0;
  auto launch = [&](auto l) -> cudaError_t {
    constexpr int L = decltype(l)::value;
    const auto kernel = stat == kStatBlockMax ? tc_pair_gemm_kernel<L, kStatBlockMax>
                        : stat == kStatAbsMax ? tc_pair_gemm_kernel<L, kStatAbsMax>
                                              : tc_pair_gemm_kernel<L, 0>;
    return launch_dependent(kernel, dim3(grid), dim3(NUM_THREADS), smem_bytes<L != kStaged>(), st, maps, args);
  };
  CUTQC_CUDA_TRY(layout == kDirect64  ? launch(std::integral_constant<int, kDirect64>{})
                 : layout == kDirect8 ? launch(std::integral_constant<int, kDirect8>{})
                                      : launch(std::integral_constant<int, kStaged>{}));
  CUTQC_LAUNCH_CHECK("tc_pair_gemm_kernel");
  return CUTQC_OK;
}

}  // namespace cutqc

extern "C" int cutqc_fd_set_tiles_per_item(int tiles_per_item) {
  return cutqc::set_pair_tiles_per_item(tiles_per_item);
}
