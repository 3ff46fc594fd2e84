// FP64 block GEMM on the tensor cores by operand slicing (the splitting scheme
// of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with the
// products on matrix units as in Mukunoki et al., ISC 2020):
//
//   C[m, n] = sum_k A[m, k] B[n, k] (+ C[m, n]),  FP64 in and out.
//
// Every row of A and B is scaled by its own power of two and written as seven
// 8-bit signed digits (hs_bits.cuh: slice_fixed), each digit plane a BF16
// matrix. Digit products of equal weight ("level" l = i + j) are summed by
// tcgen05.mma in one FP32 accumulator; integers up to 2^24 are exact there,
//   (l - 1) pairs x 192 columns x 2^14 <= 5 * 192 * 2^14 < 2^24,
// so the levels 2..6 are drained into 64-bit integers every 192 columns and
// carry no rounding at all. Levels 7, 8 and 9 weigh 2^-40 and less of the
// leading one and share one accumulator; the 15 pairs beyond level 9 are left
// out, below the digits' own 2^-56 of the row's scale. (Leaving out level 9 as
// well is 18% faster, but on rows that fall off by six decades its 2^-52 per
// term was 1.7 times the error of an FP64 chain.) The roundings left are the
// operands' own, the truncated FP32 sums of levels 7..9 and that of the final
// 64-bit integer to FP64.
//
// Bound: the FP64 pipe of GB300 runs at 1.1 TF/s, BF16 tensor products at 1936
// (measured); 34 pairs per product leave 57 TF/s. One CTA per SM:
//   warp 0 lane 0   bulk copies: the split kernel writes each (row block, K step)
//                   as one contiguous, already swizzled piece of all seven planes
//                   (57 KB of A, 35 KB of B, two stages). A tensor map with
//                   64-byte rows took 4200 cycles a stage against the 2912 of its
//                   products;
//   warp 1 lane 0   tcgen05.mma 128 x 80 x 16 into six accumulators of 80 columns
//                   (480 of the 512 TMEM columns; with N = 80 an instruction
//                   reads 6.5 KB of shared memory in the 40 cycles it computes,
//                   so shared memory bounds it at 79%; N = 64 would give 67%, and
//                   N = 96 leaves no columns for the sixth accumulator);
//   warps 2..17     drain: TMEM -> 64-bit sums in registers (four quarters of 20
//                   columns), at the end FP64 through shared memory to C, while the
//                   next tile's products run. The drain is a chain of latencies, so
//                   it takes four warps per SM sub-partition: with two, 130
//                   instructions an entry took 50 thousand cycles a tile.
// All operand digits of a K step stay in shared memory for its 34 pair
// products, so each is read from L2 once per tile and step.
//
// The digits' errors are relative to the rows' largest entries, an FMA chain's to the
// terms it adds, so an entry whose large factors meet small ones (operands graded in
// opposite directions along k) would lose digits. First, gradings that a power of two a
// column takes out are taken out (slice_scale_kernel). Then every entry also gets S =
// sum |a||b|, from magnitudes in E5M2 (slice_mag8: one more byte an entry; mag_kernel,
// one MMA a K step), and an entry whose error bound
//   2^-56 2^(ea + eb) (sum |a| / 2^ea + sum |b| / 2^eb)      (operands' rounding)
//   + the truncation of levels 7..9
// exceeds 2 sqrt(K) 2^-53 S (kBoundEntry) is listed, and fma_kernel sums it by FP64 FMAs. (A chain's
// own worst case is K 2^-53 S, its error on random terms 0.5 2^-53 S, the slices' at the
// bound 1 to 2 2^-53 S; operands whose halves of the index hold rows in turn, 100 times
// larger: 0.59 as a chain, 3.2 with a bound of 4 sqrt(K), 0.59 with this one.) Entries of rows or columns that hold an infinity or NaN, or whose
// scale leaves [2^-400, 2^500], are listed too, so non-finite values propagate as in a
// chain. The chains of the library, whose operands carry errors of 2^-53 of their
// largest entries already, hold theirs to K 2^-53 S or to the rows' scale (SliceBound, where
// it is chosen). Root mean square of error / S in units of 2^-53, 10368 x 666 x 666, A falling
// and B rising by d decades along k; without scales and lists, with them, library DGEMM:
//   d = 0: 0.05, 0.05, 0.47   2: 3.6, 0.10, 0.48   4: 285, 0.12, 0.49   8: 2e6, 0.10, 0.47
// in 276 us before, 290 now. Of the CTMRG and HOTRG chains' entries some 1e-3 are listed
// in products over a boundary bond, fewer in the others.
#include <algorithm>
#include <climits>
#include <cmath>
#include <type_traits>

#include "hs_bits.cuh"
#include "hs_internal.cuh"
#include "hs_tc.cuh"

namespace hs {

namespace {

constexpr int BM = 128, BN = 80, KC = 32, NS = 7;
constexpr int ROW_BYTES = KC * 2;
constexpr int A_SLICE = BM * ROW_BYTES, B_SLICE = BN * ROW_BYTES;
constexpr int STAGE_BYTES = NS * (A_SLICE + B_SLICE);
constexpr int STAGES = 2;
constexpr int CHUNK = 6;  // K steps between drains
constexpr int NACC = 6;   // levels 2..6, and 7 to LMAX
constexpr int LMAX = 9;
constexpr uint32_t TMEM_COLS = 512;
constexpr int kEpiWarps = 16;
constexpr int NT = 32 * (2 + kEpiWarps);
constexpr int PART = BN / (kEpiWarps / 4);  // columns per epilogue warp
constexpr int STG_LD = 6;                   // staging row stride in doubles (four columns, 16-byte rows)
constexpr int STG_BYTES = kEpiWarps * 32 * STG_LD * 8;
constexpr int SMEM = STAGES * STAGE_BYTES + STG_BYTES + 256 + 1024;
static_assert(STAGE_BYTES % 1024 == 0 && A_SLICE % 1024 == 0 && B_SLICE % 1024 == 0, "swizzle atom alignment");
static_assert(SMEM <= 232448, "shared memory per CTA");
static_assert(NACC * BN <= (int)TMEM_COLS, "TMEM columns");
static_assert(5LL * CHUNK * KC * (1 << 14) < (1 << 24), "exact sums of level 6");
constexpr int kSpecial = INT_MIN;

// What the split leaves of a row beside its scale's exponent (kSpecial: marked): the
// sum of its magnitudes over the scale and the number of its nonzeros.
struct SlRow {
  float sum, count;
};

struct SlUnit {
  int M, N, K, ldc;
  int tile_start, tiles_n;
  int frac;  // extra fraction bits of the 64-bit sums
  // an entry is left to fma_kernel where its S (in units 2^-30 2^(ea + eb)) is below
  // g_round (rounding sums) + g_low, or |levels 7..9| above low_max
  float g_round, g_low, low_max;
  double* c;
  const unsigned char* pa;  // digit planes
  const unsigned char* pb;
  const unsigned char* ga;  // magnitudes
  const unsigned char* gb;
  const int* ea;
  const int* eb;
  const SlRow* ra;
  const SlRow* rb;
  SlMat a, b;  // FP64 sources
};

struct SlGroup {
  int n;
  SlUnit u[kMaxProblems];
};

// Bulk copy of contiguous bytes to shared memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// Shared-memory descriptor of a 64-byte-swizzled K-major operand (8-row groups
// 512 bytes apart): its upper word is a constant, the lower one holds the
// address in 16-byte units.
constexpr uint32_t kDescHi = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr & 0x3FFFF) >> 4) | (1u << 16); }

// kind::f16: FP32 accumulators, BF16 operands, both K-major, 128 x 80.
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t leader, uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n setp.ne.b32 q, %6, 0;\n"
      " mov.b64 da, {%1, %3};\n mov.b64 db, {%2, %3};\n"
      " @q tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n}\n" ::"r"(d_tmem),
      "r"(a_lo), "r"(b_lo), "r"(kDescHi), "r"(kIdesc), "r"(acc), "r"(leader));
}

// kind::f8f6f4 with both operands E5M2: the same descriptor bits (format 1).
__device__ __forceinline__ void mma_mag8(uint32_t leader, uint32_t d_tmem, uint32_t a_lo, uint32_t b_lo, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p, q;\n .reg .b64 da, db;\n setp.ne.b32 p, %5, 0;\n setp.ne.b32 q, %6, 0;\n"
      " mov.b64 da, {%1, %3};\n mov.b64 db, {%2, %3};\n"
      " @q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], da, db, %4, p;\n}\n" ::"r"(d_tmem),
      "r"(a_lo), "r"(b_lo), "r"(kDescHi), "r"(kIdesc), "r"(acc), "r"(leader));
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}

// The pair products of one K step (two instructions of 16 columns each) that
// go to accumulators [A0, A1).
template <int A0, int A1>
__device__ __forceinline__ void step_mmas(uint32_t leader, uint32_t tmem, uint32_t da, uint32_t db, bool first) {
#pragma unroll
  for (int kk = 0; kk < KC / 16; ++kk) {
#pragma unroll
    for (int i = 1; i <= NS; ++i) {
      const uint32_t a = da + ((i - 1) * A_SLICE + kk * 32) / 16;
#pragma unroll
      for (int j = 1; j <= NS; ++j) {
        const int acc = i + j - 2 < NACC - 1 ? i + j - 2 : NACC - 1;
        if (i + j > LMAX || acc < A0 || acc >= A1) continue;
        const uint32_t b = db + ((j - 1) * B_SLICE + kk * 32) / 16;
        // i = 1, j = acc + 1 is the first product of each accumulator
        const uint32_t keep = (kk == 0 && i == 1 && j <= NACC) ? (first ? 0u : 1u) : 1u;
        mma_bf16(leader, tmem + (uint32_t)(acc * BN), a, b, keep);
      }
    }
  }
}

// Entries left to fma_kernel: masks of them, one per row of PART columns, and a list of
// the rows with a mask. Row i of tile t and part p of its columns stand at
// (t * BM + i) * (BN / PART) + p.
constexpr int kTileRows = BM * (BN / PART);
static_assert(BN / PART == kEpiWarps / 4, "a warp per quarter of the rows and part of the columns");
struct SlList {
  int count, pad;
  unsigned long long work;  // FMAs of the entries that mag_kernel listed
  long long at[1];          // of kTileRows a tile
};

// Appends the rows of this warp with `on`.
__device__ __forceinline__ void list_rows(SlList* list, bool on, long long at) {
  const uint32_t rows = __ballot_sync(0xffffffffu, on);
  if (rows == 0u) return;
  const int lane = threadIdx.x % 32;
  int slot = 0;
  if (lane == 0) slot = atomicAdd(&list->count, __popc(rows));
  slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(rows & ((1u << lane) - 1u));
  if (on) list->at[slot] = at;
}

// The columns of a part of which `left` are in the matrix.
__device__ __forceinline__ uint32_t part_columns(int left) {
  return left <= 0 ? 0u : left < PART ? (1u << left) - 1u : (1u << PART) - 1u;
}

struct SlTile {
  int u, m0, n0;
};

__device__ __forceinline__ SlTile tile_at(const SlGroup& g, int t) {
  int u = 0;
  while (u + 1 < g.n && t >= g.u[u + 1].tile_start) ++u;
  t -= g.u[u].tile_start;
  return {u, (t / g.u[u].tiles_n) * BM, (t % g.u[u].tiles_n) * BN};
}

template <bool ACC>
__global__ void __launch_bounds__(NT, 1) gemm_sl_kernel(const __grid_constant__ SlGroup g, int total_tiles,
                                                        unsigned long long limit, uint32_t* __restrict__ masks,
                                                        SlList* __restrict__ list, int* __restrict__ err) {
  hs_pdl_enter();
  if (list->work > limit) return;  // fma_kernel computes the whole product
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  double* stage_c = reinterpret_cast<double*>(smem + STAGES * STAGE_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES + STG_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;  // [2]: accumulators 0..2, 3..5
  uint64_t* tempty = tfull + 2;      // [2]
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;  // warp: uniform
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(smem_u32(&tfull[h]), 1);
      mbar_init(smem_u32(&tempty[h]), kEpiWarps);
    }
    mbar_init(smem_u32(drain), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- copies ----
    long long it = 0;
    for (int t = blockIdx.x; t < total_tiles && !*abort_flag; t += gridDim.x) {
      const SlTile r = tile_at(g, t);
      const SlUnit& U = g.u[r.u];
      const int steps = (U.K + KC - 1) / KC;
      const unsigned char* pa = U.pa + (size_t)(r.m0 / BM) * steps * (NS * A_SLICE);
      const unsigned char* pb = U.pb + (size_t)(r.n0 / BN) * steps * (NS * B_SLICE);
      for (int k = 0; k < steps; ++k) {
        const int s = (int)(it % STAGES);
        const long long n = it / STAGES;
        if (n > 0 && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((n - 1) & 1), abort_flag, err, 11)) break;
        if (*abort_flag) break;
        const uint32_t fb = smem_u32(&full[s]);
        mbar_expect_tx(fb, STAGE_BYTES);
        const uint32_t st = smem_u32(smem + s * STAGE_BYTES);
        bulk_load(st, pa + (size_t)k * (NS * A_SLICE), NS * A_SLICE, fb);
        bulk_load(st + NS * A_SLICE, pb + (size_t)k * (NS * B_SLICE), NS * B_SLICE, fb);
        ++it;
      }
    }
    if (*abort_flag)
      for (long long j = it > STAGES ? it - STAGES : 0; j < it; ++j)
        mbar_drain(smem_u32(&full[j % STAGES]), (uint32_t)((j / STAGES) & 1));
  } else if (warp == 1) {
    // ---- MMA issuer: the whole warp, one elected lane's instructions ----
    const uint32_t leader = elect_one();
    // the stages' descriptors as loop constants (a descriptor that depends on
    // the step's stage cost 20 cycles more per instruction)
    static_assert(STAGES == 2, "two copies of the products");
    const uint32_t da0 = desc_lo(smem_u32(smem)), db0 = desc_lo(smem_u32(smem + NS * A_SLICE));
    const uint32_t da1 = desc_lo(smem_u32(smem + STAGE_BYTES)), db1 = desc_lo(smem_u32(smem + STAGE_BYTES + NS * A_SLICE));
    auto wait = [&](uint64_t* bar, long long n, int code) {
      return (bool)__all_sync(0xffffffffu, mbar_wait(smem_u32(bar), (uint32_t)(n & 1), abort_flag, err, code));
    };
    long long it = 0, use0 = 0, use1 = 0;  // steps; fills of the two halves of the accumulators
    bool any = false, ok = true, ready = false;
    for (int t = blockIdx.x; ok && t < total_tiles; t += gridDim.x) {
      const SlTile r = tile_at(g, t);
      const int steps = (g.u[r.u].K + KC - 1) / KC;
      for (int k0 = 0; ok && k0 < steps; k0 += CHUNK) {
        const int k1 = k0 + CHUNK < steps ? k0 + CHUNK : steps;
        for (int k = k0; k < k1; ++k) {
          const int s = (int)(it % STAGES);
          ok = ready || wait(&full[s], it / STAGES, 12);
          // the first half of the accumulators, then the second: a chunk's last
          // step hands the first half to the epilogue while the second still
          // multiplies, and its first step needs the second half later
          if (ok && k == k0 && use0 > 0)
            ok = wait(&tempty[0], use0 - 1, 14);
          if (!ok) break;
          fence_after();
          if (s == 0)
            step_mmas<0, 3>(leader, tmem, da0, db0, k == k0);
          else
            step_mmas<0, 3>(leader, tmem, da1, db1, k == k0);
          any = true;
          if (k == k1 - 1) {
            mma_commit_by(leader, smem_u32(&tfull[0]));
            ++use0;
          }
          if (k == k0 && use1 > 0) {
            ok = wait(&tempty[1], use1 - 1, 15);
            if (!ok) break;
            fence_after();
          }
          if (s == 0)
            step_mmas<NACC - 1, NACC>(leader, tmem, da0, db0, k == k0);
          else
            step_mmas<NACC - 1, NACC>(leader, tmem, da1, db1, k == k0);
          // the next step's barrier is tested before the last products are issued:
          // the test's shared-memory latency (250 cycles while the products hold
          // the port) is then hidden behind them
          ready = __all_sync(0xffffffffu, mbar_test(smem_u32(&full[1 - s]), (uint32_t)(((it + 1) / STAGES) & 1)));
          if (s == 0)
            step_mmas<3, NACC - 1>(leader, tmem, da0, db0, k == k0);
          else
            step_mmas<3, NACC - 1>(leader, tmem, da1, db1, k == k0);
          if (k == k1 - 1) {
            mma_commit_by(leader, smem_u32(&tfull[1]));
            ++use1;
          }
          mma_commit_by(leader, smem_u32(&empty[s]));
          ++it;
        }
      }
    }
    if (!ok && any) {
      mma_commit_by(leader, smem_u32(drain));
      mbar_drain(smem_u32(drain), 0);
    }
  } else if (warp >= 2) {
    // ---- drain and epilogue ----
    const int q = warp & 3, part = (warp - 2) / 4;
    double* stg = stage_c + (warp - 2) * 32 * STG_LD;
    const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(part * PART);
    uint32_t use0 = 0, use1 = 0;
    for (int t = blockIdx.x; t < total_tiles; t += gridDim.x) {
      const SlTile r = tile_at(g, t);
      const SlUnit& U = g.u[r.u];
      const int steps = (U.K + KC - 1) / KC;
      long long sum[PART];
      float low[PART];
#pragma unroll
      for (int j = 0; j < PART; ++j) {
        sum[j] = 0;
        low[j] = 0.f;
      }
      bool ok = true;
      const int row0 = r.m0 + q * 32, row = row0 + lane;
      const int colp = r.n0 + part * PART;  // this warp's first column
      // exponents of the scales (of marked rows: any, their entries are replaced)
      const int ea = row < U.M ? __ldg(U.ea + row) : 0;
      const int ebl = (lane < PART && colp + lane < U.N) ? __ldg(U.eb + colp + lane) : 0;
      // one lane polls: 512 polling threads slowed the products they wait for
      auto filled = [&](int h, uint32_t use) {
        int got = 1;
        if (lane == 0) got = mbar_wait(smem_u32(&tfull[h]), use & 1, abort_flag, err, 13);
        return (bool)__shfl_sync(0xffffffffu, got, 0);
      };
      for (int k0 = 0; k0 < steps; k0 += CHUNK) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          ok = ok && filled(h, h ? use1 : use0);
          if (!ok) break;
          fence_after();
#pragma unroll
          for (int c = 0; c < PART; c += 4) {
            uint32_t v[3][4];
#pragma unroll
            for (int l = 0; l < 3; ++l) tmem_ld4(base + (uint32_t)((3 * h + l) * BN + c), v[l]);
            tmem_wait_ld();
            // level l + 2 holds integers times 2^(-8 l); summed in units of level 6
#pragma unroll
            for (int j = 0; j < 4; ++j) {
#pragma unroll
              for (int l = 3 * h; l < 3 * h + 3; ++l) {
                const float f = __uint_as_float(v[l - 3 * h][j]);
                if (l == NACC - 1)
                  low[c + j] += f;
                else
                  sum[c + j] += (long long)__float2int_rn(f * (float)(1ull << (8 * l))) * (1ll << (8 * (4 - l)));
              }
            }
          }
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&tempty[h]));
          if (h)
            ++use1;
          else
            ++use0;
        }
        if (!ok) break;
      }
      if (!ok) break;
      // low digits that are not random (their truncated sums may be off by more than
      // mag_kernel assumes): these entries are left to fma_kernel too
      uint32_t late = 0u;
      const long long at = ((long long)t * BM + q * 32 + lane) * (BN / PART) + part;
      const uint32_t listed = ACC ? masks[at] : 0u;  // entries that fma_kernel adds to
      // to FP64: (sum + low 2^32) 2^(ea + eb - 46), with U.frac more bits
      const float lscale = __uint_as_float((uint32_t)(127 + 32 + U.frac) << 23);
      const bool vec = (U.ldc % 2 == 0) && ((reinterpret_cast<uintptr_t>(U.c) & 15) == 0);
#pragma unroll
      for (int c = 0; c < PART; c += 4) {
        if (colp + c >= U.N) break;
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
          double o[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int e = __shfl_sync(0xffffffffu, ebl, c + j + u) + ea - 46 - U.frac;
            if (fabsf(low[c + j + u]) > U.low_max) late |= 1u << (c + j + u);
            const long long J = (sum[c + j + u] << U.frac) + (long long)__float2int_rn(low[c + j + u] * lscale);
            o[u] = f64_from_bits(fixed_to_f64(J, e));
          }
          *reinterpret_cast<double2*>(&stg[lane * STG_LD + j]) = make_double2(o[0], o[1]);
        }
        __syncwarp();
        // two lanes per row, two columns each: sixteen rows (32-byte sectors) per warp store
        const int col = colp + c + 2 * (lane & 1);
#pragma unroll
        for (int i0 = 0; i0 < 32; i0 += 16) {
          const int i = i0 + (lane >> 1);
          const uint32_t skip = ACC ? __shfl_sync(0xffffffffu, listed | late, i) >> (c + 2 * (lane & 1)) : 0u;
          if (row0 + i < U.M && col < U.N) {
            double2 x = *reinterpret_cast<const double2*>(&stg[i * STG_LD + 2 * (lane & 1)]);
            double* dst = U.c + (long long)(row0 + i) * U.ldc + col;
            if (ACC && (skip & 3u)) {
              if (!(skip & 1u)) dst[0] += x.x;
              if (!(skip & 2u) && col + 1 < U.N) dst[1] += x.y;
            } else if (vec && col + 1 < U.N) {
              if (ACC) {
                const double2 y = *reinterpret_cast<const double2*>(dst);
                x.x += y.x;
                x.y += y.y;
              }
              *reinterpret_cast<double2*>(dst) = x;
            } else {
              dst[0] = ACC ? dst[0] + x.x : x.x;
              if (col + 1 < U.N) dst[1] = ACC ? dst[1] + x.y : x.y;
            }
          }
        }
        __syncwarp();
      }
      if (row >= U.M) late = 0u;
      late &= part_columns(U.N - colp);
      if (__any_sync(0xffffffffu, late != 0u)) {
        const uint32_t before = masks[at];
        list_rows(list, late != 0u && before == 0u, at);
        if (late != 0u) masks[at] = before | late;
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---- the entries that keep too few digits ------------------------------------------

// Entries (row, col0 + j), j a bit of m, by FP64 FMAs, of one warp (T = 32) or the whole
// CTA (T = 256). Bound by the FP64 pipe (19 cycles a warp's FMA) or by latency where
// they are few: threads over k with four columns at a time (K / 32 FMAs and 1.5 adds an
// entry), or a lane a column, the chain itself, where the row has enough of them that
// its K FMAs are fewer.
template <int T>
__device__ __forceinline__ void fma_row(const SlUnit& U, int row, int col0, uint32_t m, bool accumulate,
                                        double (*red)[4]) {
  const int lane = threadIdx.x % 32;
  double* dst = U.c + (long long)row * U.ldc + col0;
  if (T == 32 && (float)__popc(m) * ((float)((U.K + 31) / 32) + 1.5f) > (float)U.K) {
    if (!(m >> lane & 1)) return;
    double v = 0.0;
    for (int s = 0; s < U.a.nseg; ++s) {
      const double* pa = U.a.p[s] + (long long)row * U.a.ld;
      const double* pb = U.b.p[s] + (long long)(col0 + lane) * U.b.ld;
      const bool neg = U.a.neg[s] != U.b.neg[s];
#pragma unroll 4
      for (int k = 0; k < U.a.kseg; ++k) v = fma(neg ? -pa[k] : pa[k], pb[k], v);
    }
    dst[lane] = accumulate ? dst[lane] + v : v;
    return;
  }
  while (m != 0) {  // the same in every thread
    int col[4], n = 0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (m != 0) {
        col[t] = __ffs(m) - 1;
        m &= m - 1;
        n = t + 1;
      } else {
        col[t] = col[0];
      }
    }
    double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
    for (int kk = threadIdx.x % T; kk < U.K; kk += T) {
      const int s = kk >= U.a.kseg, k = s ? kk - U.a.kseg : kk;
      double x = (s ? U.a.p[1] : U.a.p[0])[(long long)row * U.a.ld + k];
      if (U.a.neg[s] != U.b.neg[s]) x = -x;
      const double* pb = (s ? U.b.p[1] : U.b.p[0]) + (long long)col0 * U.b.ld + k;
#pragma unroll
      for (int t = 0; t < 4; ++t)
        if (t < n) v[t] = fma(x, pb[col[t] * U.b.ld], v[t]);
    }
    // the four sums folded into quarters of the warp: lanes 8 t .. 8 t + 7 end with column t's
    const bool h = lane & 16, q = lane & 8;
    const double a0 = (h ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h ? v[0] : v[2], 16);
    const double a1 = (h ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h ? v[1] : v[3], 16);
    double r = (q ? a1 : a0) + __shfl_xor_sync(0xffffffffu, q ? a0 : a1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    const int t = lane >> 3;
    if (T > 32) {
      if ((lane & 7) == 0) red[threadIdx.x / 32][t] = r;
      __syncthreads();
      if (threadIdx.x < 32 && (lane & 7) == 0) {
        r = 0.0;
        for (int w = 0; w < T / 32; ++w) r += red[w][t];
      }
      __syncthreads();
    }
    if (threadIdx.x % T < 32 && (lane & 7) == 0 && t < n) {
      const int c = t == 0 ? col[0] : t == 1 ? col[1] : t == 2 ? col[2] : col[3];
      dst[c] = accumulate ? dst[c] + r : r;
    }
  }
}

// A 64 x 64 tile of a product, every entry a chain of FMAs over k, as gemm_f64_nt_kernel
// computes it.
constexpr int FT = 64, FK = 16;
__device__ __forceinline__ void fma_tile(const SlUnit& U, int m0, int n0, bool accumulate, double (*As)[FT + 2],
                                         double (*Bs)[FT + 2]) {
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  for (int k0 = 0; k0 < U.K; k0 += FK) {
    const int k = k0 + tx, s = k >= U.a.kseg, ks = s ? k - U.a.kseg : k;
    const bool in = k < U.K, flip = in && U.a.neg[s] != U.b.neg[s];
    const double* pa = (s ? U.a.p[1] : U.a.p[0]) + ks;
    const double* pb = (s ? U.b.p[1] : U.b.p[0]) + ks;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 16 * i;
      const double x = in && m0 + r < U.M ? pa[(long long)(m0 + r) * U.a.ld] : 0.0;
      As[tx][r] = flip ? -x : x;
      Bs[tx][r] = in && n0 + r < U.N ? pb[(long long)(n0 + r) * U.b.ld] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < FK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = As[kk][ty + 16 * i];
        b[i] = Bs[kk][tx + 16 * i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m < U.M && n < U.N) {
        double* o = U.c + (long long)m * U.ldc + n;
        *o = accumulate ? *o + acc[i][j] : acc[i][j];
      }
    }
}

// A listed row at a time: one warp's where the contraction is short, else one CTA's. Where
// the listed entries are more than a third of the work (limit), which the rows' FMAs take
// as long for as the whole product takes on shared tiles, the whole product is computed
// that way and gemm_sl_kernel is left out: 10368 x 666 x 666 with every entry listed
// 8.4 ms (23.2 row by row, 19.1 as serial dot products in the epilogue; the FP64 kernel alone
// 8.0), one column of NaN 0.49 ms (1.66).
constexpr int kWarpK = 512;
__global__ void __launch_bounds__(256, 3) fma_kernel(const __grid_constant__ SlGroup g, bool accumulate,
                                                     unsigned long long limit, const uint32_t* __restrict__ masks,
                                                     const SlList* __restrict__ list) {
  hs_pdl_enter();
  __shared__ double red[8][4];
  __shared__ double As[FK][FT + 2], Bs[FK][FT + 2];
  if (list->work > limit) {
    int t = blockIdx.x;
    for (int u = 0; u < g.n; ++u) {
      const SlUnit& U = g.u[u];
      const int tn = (U.N + FT - 1) / FT, tiles = (U.M + FT - 1) / FT * tn;
      for (; t < tiles; t += gridDim.x) fma_tile(U, t / tn * FT, t % tn * FT, accumulate, As, Bs);
      t -= tiles;
    }
    return;
  }
  const int n = list->count;
  bool longer = false, shorter = false;
  for (int u = 0; u < g.n; ++u) (g.u[u].K > kWarpK ? longer : shorter) = true;
  auto each = [&](int i, auto width) {
    const long long at = list->at[i];
    const int part = (int)(at % (BN / PART)), row = (int)(at / (BN / PART) % BM);
    const SlTile r = tile_at(g, (int)(at / kTileRows));
    const SlUnit& U = g.u[r.u];
    if ((U.K > kWarpK) == (width.value > 32))
      fma_row<width.value>(U, r.m0 + row, r.n0 + part * PART, masks[at], accumulate, red);
  };
  if (shorter)
    for (int i = blockIdx.x * 8 + threadIdx.x / 32; i < n; i += gridDim.x * 8) each(i, std::integral_constant<int, 32>());
  if (longer)
    for (int i = blockIdx.x; i < n; i += gridDim.x) each(i, std::integral_constant<int, 256>());
}

// ---- S = sum |a||b| of every entry ---------------------------------------------------
//
// Magnitudes in E5M2, 64 bytes a row and piece of two K steps. Bound by the bulk copies
// where K is long (13 KB a piece) and by the drain's latency where it is short: two CTAs
// an SM, accumulators in turn. As a last chunk of gemm_sl_kernel itself it took twice as
// long: its products waited there for a drain, and the drain for them.
constexpr int MSTAGES = 4, MPIECES = 2;
constexpr int A_PIECE = BM * 64, B_PIECE = BN * 64, M_STAGE = MPIECES * (A_PIECE + B_PIECE);
constexpr int kMagWarps = 8, MNT = 32 * (2 + kMagWarps);
constexpr int MCOLS = BN / (kMagWarps / 4);  // columns per warp: two parts
constexpr int MSMEM = MSTAGES * M_STAGE + 256 + 1024;
constexpr uint32_t M_TMEM = 256;
static_assert(MCOLS == 2 * PART && 2 * MSMEM <= 232448, "two parts a warp, two CTAs an SM");

__global__ void __launch_bounds__(MNT, 2) mag_kernel(const __grid_constant__ SlGroup g, int total_tiles,
                                                     uint32_t* __restrict__ masks, SlList* __restrict__ list,
                                                     int* __restrict__ err) {
  hs_pdl_enter();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + MSTAGES * M_STAGE);
  uint64_t* empty = full + MSTAGES;
  uint64_t* tfull = empty + MSTAGES;  // [2]
  uint64_t* tempty = tfull + 2;       // [2]
  uint64_t* drain = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;  // warp: uniform
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(M_TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < MSTAGES; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int h = 0; h < 2; ++h) {
      mbar_init(smem_u32(&tfull[h]), 1);
      mbar_init(smem_u32(&tempty[h]), kMagWarps);
    }
    mbar_init(smem_u32(drain), 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- copies ----
    long long it = 0;
    for (int t = blockIdx.x; t < total_tiles && !*abort_flag; t += gridDim.x) {
      const SlTile r = tile_at(g, t);
      const SlUnit& U = g.u[r.u];
      const int pieces = ((U.K + KC - 1) / KC + 1) / 2;
      const unsigned char* ga = U.ga + (size_t)(r.m0 / BM) * pieces * A_PIECE;
      const unsigned char* gb = U.gb + (size_t)(r.n0 / BN) * pieces * B_PIECE;
      for (int p = 0; p < pieces; p += MPIECES, ++it) {
        const uint32_t np = (uint32_t)(pieces - p < MPIECES ? pieces - p : MPIECES);
        const int s = (int)(it % MSTAGES);
        const long long n = it / MSTAGES;
        if (n > 0 && !mbar_wait(smem_u32(&empty[s]), (uint32_t)((n - 1) & 1), abort_flag, err, 16)) break;
        if (*abort_flag) break;
        const uint32_t fb = smem_u32(&full[s]), st = smem_u32(smem + s * M_STAGE);
        mbar_expect_tx(fb, np * (A_PIECE + B_PIECE));
        bulk_load(st, ga + (size_t)p * A_PIECE, np * A_PIECE, fb);
        bulk_load(st + MPIECES * A_PIECE, gb + (size_t)p * B_PIECE, np * B_PIECE, fb);
      }
    }
    if (*abort_flag)
      for (long long j = it > MSTAGES ? it - MSTAGES : 0; j < it; ++j)
        mbar_drain(smem_u32(&full[j % MSTAGES]), (uint32_t)((j / MSTAGES) & 1));
  } else if (warp == 1) {
    // ---- MMA issuer ----
    const uint32_t leader = elect_one();
    auto wait = [&](uint64_t* bar, long long n, int code) {
      return (bool)__all_sync(0xffffffffu, mbar_wait(smem_u32(bar), (uint32_t)(n & 1), abort_flag, err, code));
    };
    long long it = 0;
    int local = 0;
    bool any = false, ok = true;
    for (int t = blockIdx.x; ok && t < total_tiles; t += gridDim.x, ++local) {
      const SlTile r = tile_at(g, t);
      const int steps = (g.u[r.u].K + KC - 1) / KC, buf = local & 1, use = local >> 1;
      if (use > 0) ok = wait(&tempty[buf], use - 1, 18);
      if (!ok) break;
      fence_after();
      const uint32_t d = tmem + (uint32_t)buf * (M_TMEM / 2);
      for (int k0 = 0; k0 < steps; k0 += 2 * MPIECES, ++it) {
        const int s = (int)(it % MSTAGES);
        ok = wait(&full[s], it / MSTAGES, 17);
        if (!ok) break;
        fence_after();
        const uint32_t da = desc_lo(smem_u32(smem + s * M_STAGE)), db = desc_lo(smem_u32(smem + s * M_STAGE + MPIECES * A_PIECE));
#pragma unroll
        for (int i = 0; i < 2 * MPIECES; ++i)
          if (k0 + i < steps)
            mma_mag8(leader, d, da + (uint32_t)((i / 2 * A_PIECE + (i & 1) * 32) / 16),
                     db + (uint32_t)((i / 2 * B_PIECE + (i & 1) * 32) / 16), k0 + i > 0 ? 1u : 0u);
        any = true;
        mma_commit_by(leader, smem_u32(&empty[s]));
      }
      if (!ok) break;
      mma_commit_by(leader, smem_u32(&tfull[buf]));
    }
    if (!ok && any) {
      mma_commit_by(leader, smem_u32(drain));
      mbar_drain(smem_u32(drain), 0);
    }
  } else if (warp >= 2) {
    // ---- the entries whose S is too small ----
    const int q = warp & 3, half = (warp - 2) / 4;
    int local = 0;
    for (int t = blockIdx.x; t < total_tiles; t += gridDim.x, ++local) {
      const SlTile r = tile_at(g, t);
      const SlUnit& U = g.u[r.u];
      const int buf = local & 1, row = r.m0 + q * 32 + lane, col0 = r.n0 + half * MCOLS;
      const SlRow none = {0.f, 0.f};
      const SlRow ra = row < U.M ? U.ra[row] : none;
      const SlRow b0 = col0 + lane < U.N ? U.rb[col0 + lane] : none;
      const SlRow b1 = lane < MCOLS - 32 && col0 + 32 + lane < U.N ? U.rb[col0 + 32 + lane] : none;
      // bit j: column col0 + j
      const int e0 = col0 + lane < U.N ? U.eb[col0 + lane] : 0;
      const int e1 = lane < MCOLS - 32 && col0 + 32 + lane < U.N ? U.eb[col0 + 32 + lane] : 0;
      unsigned long long again = __ballot_sync(0xffffffffu, e0 == kSpecial) |
                                 (unsigned long long)__ballot_sync(0xffffffffu, e1 == kSpecial) << 32;
      if (row < U.M && U.ea[row] == kSpecial) again = ~0ull;
      int got = 1;
      if (lane == 0) got = mbar_wait(smem_u32(&tfull[buf]), (uint32_t)((local >> 1) & 1), abort_flag, err, 19);
      if (!__shfl_sync(0xffffffffu, got, 0)) break;
      fence_after();
      uint32_t v[MCOLS / 4][4];
      const uint32_t base = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * (M_TMEM / 2) + half * MCOLS);
#pragma unroll
      for (int c = 0; c < MCOLS / 4; ++c) tmem_ld4(base + (uint32_t)(4 * c), v[c]);
      tmem_wait_ld();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&tempty[buf]));
      // a rounded entry meets only the other row's nonzeros: the smaller of a row's sum and
      // the other's count, which only sparse rows make the count
      const bool dense = __all_sync(0xffffffffu, row >= U.M || ra.count == (float)U.K) &&
                         __all_sync(0xffffffffu, (col0 + lane >= U.N || b0.count == (float)U.K) &&
                                                     (lane >= MCOLS - 32 || col0 + 32 + lane >= U.N || b1.count == (float)U.K));
      const float inv_k = 1.f / (float)U.K;
      if (dense) {
        const float mine = U.g_round * ra.sum + U.g_low, s0 = U.g_round * b0.sum, s1 = U.g_round * b1.sum;
#pragma unroll
        for (int j = 0; j < MCOLS; ++j) {
          const float S = __uint_as_float(v[j / 4][j & 3]);
          const float need = mine + __shfl_sync(0xffffffffu, j < 32 ? s0 : s1, j & 31);  // by every lane
          if (S > 0.f && S < need) again |= 1ull << j;
        }
      } else
#pragma unroll
      for (int j = 0; j < MCOLS; ++j) {
        const float sb = __shfl_sync(0xffffffffu, j < 32 ? b0.sum : b1.sum, j & 31);
        const float nb = __shfl_sync(0xffffffffu, j < 32 ? b0.count : b1.count, j & 31);
        const float S = __uint_as_float(v[j / 4][j & 3]);
        // and so are the terms of the low levels no more than the smaller count
        const float low = U.g_low * sqrtf(fminf(ra.count, nb) * inv_k);
        if (S > 0.f && S < U.g_round * (fminf(ra.sum, nb) + fminf(sb, ra.count)) + low) again |= 1ull << j;
      }
      unsigned entries = 0u;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const uint32_t m = row < U.M ? (uint32_t)(again >> (p * PART)) & part_columns(U.N - col0 - p * PART) : 0u;
        const long long at = ((long long)t * BM + q * 32 + lane) * (BN / PART) + 2 * half + p;
        masks[at] = m;
        list_rows(list, m != 0u, at);
        entries += __popc(m);
      }
      entries = __reduce_add_sync(0xffffffffu, entries);
      if (lane == 0 && entries != 0u) atomicAdd(&list->work, (unsigned long long)entries * U.K);
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(M_TMEM) : "memory");
  }
}

// ---- the digit planes -------------------------------------------------------------

// Row block rb (of `block` rows), K step ks: [NS][block][32] BF16 at
// ((rb * steps) + ks) * NS * block * 64 bytes, the 16-byte quarters of row r
// exchanged by the 64-byte swizzle (q ^ (r / 2) % 4). The columns past K are zero; rows past the
// end are left as they are (they only reach entries that are not stored).
// Magnitudes of two K steps: [block][64] bytes at ((rb * pieces) + ks / 2) * block *
// 64, with the same swizzle.
struct SplitOp {
  SlMat m;
  int K, steps, block;
  unsigned char* planes;
  unsigned char* mags;
  int* exps;           // [rows]
  SlRow* row;          // [rows]
  const short* scale;  // [steps * 32]: column k times 2^scale[k] (A) or 2^-scale[k] (B), 0 past K
};
constexpr int kMaxSplit = 2 * kMaxProblems;
struct SplitOps {
  SplitOp op[kMaxSplit];
  SlList* list;  // its count is set to zero here
};

// Bits of entry k of a row, its sign flipped where the source is negated (as an
// integer: negating a double takes the FP64 pipe).
__device__ __forceinline__ unsigned long long sl_at(const SlMat& m, long long roff, int k) {
  const int s = k >= m.kseg;
  const double* p = s ? m.p[1] + roff - m.kseg : m.p[0] + roff;
  return f64_bits(p[k]) ^ ((unsigned long long)m.neg[s] << 63);
}

// ---- scales of the contraction index ---------------------------------------------------

// A power of two a column, A[:, k] 2^s and B[:, k] 2^-s, changes no product and no
// bit, and takes out what grading the operands have against each other. An operand's
// profile: over 32 of its rows, the upper quartile of an entry's exponent against the
// largest of the row's first 32 (rows of any scale, zeros and noise in most of a column
// do not disturb it; any s is right: what a sample does not show, S does). s is half of
// what the difference of the profiles of B and A differs from its mean over the first
// eight columns, towards zero, so that operands without such a grading keep their bits.
// Problems that share an operand share their scales. One CTA per 32 columns and set of
// problems, all its loads in flight at once. Bound by latency and, on its one SM, by
// the bisections: 5 us (64 rows, 13 steps and 32 reference columns: 9.5).
struct ScaleSet {
  SlMat m[2];  // an A operand and a B operand of the set
  short* scale;
};
struct ScaleSets {
  ScaleSet set[kMaxProblems];
};

__global__ void __launch_bounds__(1024) slice_scale_kernel(const __grid_constant__ ScaleSets sets) {
  hs_pdl_enter();
  const ScaleSet& S = sets.set[blockIdx.y];
  const int K = S.m[0].kseg * S.m[0].nseg, tx = threadIdx.x % 32, ty = threadIdx.x / 32, k0 = blockIdx.x * 32;
  if (k0 >= K) return;
  constexpr int kRef = 8, kLow = -256;  // profiles from kLow + 1; kLow: less, or a column of zeros
  constexpr short kNone = -32768, kZero = -20000;
  // exponent fields of row ty of A and B in the first columns and in this block's
  int e[2][2];
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const SlMat& m = S.m[w];
    // rows in no order, so that no leg's period is met (multiples of the golden ratio)
    const long long r =
        m.rows <= 32 ? ty : (long long)(((unsigned long long)((unsigned)ty * 2654435769u) * (unsigned)m.rows) >> 32);
#pragma unroll
    for (int own = 0; own < 2; ++own) {
      const int k = (own ? k0 : 0) + tx;
      e[w][own] = r < m.rows && k < K ? (int)(sl_at(m, r * m.ld, k) >> 52) & 0x7FF : -1;
    }
  }
  __shared__ short val[2][2][32][34];
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const int ref = __reduce_max_sync(0xffffffffu, e[w][0] == 0x7FF ? 0 : e[w][0]);
#pragma unroll
    for (int own = 0; own < 2; ++own) {
      const int x = e[w][own];
      val[w][own][ty][tx] = (short)(ref <= 0 || x < 0 ? kNone : x == 0 || x == 0x7FF ? kZero : x - ref);
    }
  }
  __syncthreads();
  // warp ty: column ty; the quartiles by bisection, of this block's and of the first columns
  __shared__ int dd[2][32];
  constexpr int kNo = 1 << 20;
#pragma unroll
  for (int own = 0; own < 2; ++own) {
    if (own == 0 && ty >= kRef) continue;
    const short a = val[0][own][tx][ty], b = val[1][own][tx][ty];
    const int wa = __popc(__ballot_sync(0xffffffffu, a != kNone)) / 4 + 1;
    const int wb = __popc(__ballot_sync(0xffffffffu, b != kNone)) / 4 + 1;
    int la = kLow, ha = 256, lb = kLow, hb = 256;
#pragma unroll
    for (int step = 0; step < 9; ++step) {
      const int ma = (la + ha) >> 1, mb = (lb + hb) >> 1;
      const bool ga = __popc(__ballot_sync(0xffffffffu, a >= ma)) >= wa, gb = __popc(__ballot_sync(0xffffffffu, b >= mb)) >= wb;
      la = ga ? ma : la;
      ha = ga ? ha : ma;
      lb = gb ? mb : lb;
      hb = gb ? hb : mb;
    }
    if (tx == 0) dd[own][ty] = la == kLow || lb == kLow ? kNo : lb - la;
  }
  __syncthreads();
  if (ty != 0) return;
  const int d0 = tx < kRef ? dd[0][tx] : kNo, d1 = dd[1][tx];
  const int n = __popc(__ballot_sync(0xffffffffu, d0 != kNo));
  const int sum = __reduce_add_sync(0xffffffffu, d0 != kNo ? d0 : 0);
  const int mean = n > 0 ? (sum >= 0 ? sum + n / 2 : sum - n / 2) / n : 0;
  S.scale[k0 + tx] = (short)(k0 + tx < K && d1 != kNo ? (d1 - mean) / 2 : 0);
}

// Float of digit i times 2^(-8 (i - 1)) from the biased value (exact, its upper
// 16 bits are the BF16): a byte b becomes the float 2^23 + b by its bit pattern,
// and one FMA takes 2^23 + 128 off and scales, so no conversion unit is used.
__device__ __forceinline__ uint32_t digit_bits(unsigned lo, unsigned hi, int i) {
  const float s = __uint_as_float((uint32_t)(127 - 8 * (i - 1)) << 23);
  if (i == 1) return __float_as_uint((float)((int)hi >> 16));
  const unsigned sel = i >= 4 ? (unsigned)(7 - i) : (unsigned)(3 - i);  // byte of lo (i >= 4) or hi
  const float m = __uint_as_float(__byte_perm(i >= 4 ? lo : hi, 0x4B000000u, 0x7440u | sel));
  return __float_as_uint(fmaf(m, s, -(8388608.f + 128.f) * s));
}

// The digits of 8 consecutive columns are 16 bytes of a plane's row, one thread's
// work: 64 bytes read, seven 16-byte stores. T threads share a row (T a power of
// two up to 32, or the whole block of 256), each with NR pieces held in registers
// between the row's largest exponent and its digits, so a row is read once; NR =
// 0 reads it twice, for rows too long for the registers. Bound by memory (8
// bytes read and 14 written per entry): 10368 x 666 takes 31 us (4-byte stores
// and a warp per row: 67), 20736 x 5184 0.43 ms (1.6).
__device__ __forceinline__ void sl_load(const SplitOp& P, bool vec, long long roff, int k,
                                        unsigned long long (&x)[8]) {
  if (vec) {
    const int s = k >= P.m.kseg;
    const double* p = (s ? P.m.p[1] + roff - P.m.kseg : P.m.p[0] + roff) + k;
    const unsigned long long flip = (unsigned long long)P.m.neg[s] << 63;
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      const ulonglong2 d =
          k + j < P.K ? *reinterpret_cast<const ulonglong2*>(p + j) : make_ulonglong2(0ull, 0ull);
      x[j] = d.x ^ flip;
      x[j + 1] = d.y ^ flip;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = k + j < P.K ? sl_at(P.m, roff, k + j) : 0ull;
  }
  const uint4 w = *reinterpret_cast<const uint4*>(P.scale + k);
  if ((w.x | w.y | w.z | w.w) == 0u) return;
  const unsigned sc[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int a = (int)(short)(sc[j / 2] >> (16 * (j & 1)));
    x[j] = slice_scaled(x[j], P.m.is_b ? -a : a);
  }
}

__device__ __forceinline__ unsigned long long sl_mag(const unsigned long long (&x)[8], unsigned long long mag) {
#pragma unroll
  for (int j = 0; j < 8; ++j) mag = max(mag, x[j] & 0x7FFFFFFFFFFFFFFFull);
  return mag;
}

__device__ __forceinline__ void sl_put(const SplitOp& P, unsigned char* row, unsigned char* mag, int rr, int k, int emax,
                                       const unsigned long long (&x)[8], float& sum, int& count) {
  const size_t plane = (size_t)P.block * ROW_BYTES;
  unsigned char* o = row + (size_t)(k / KC) * NS * plane + (((k % KC) / 8) ^ ((rr >> 1) & 3)) * 16;
  uint2* om = reinterpret_cast<uint2*>(mag + (size_t)(k / 64) * P.block * 64 + (((k % 64) / 16) ^ ((rr >> 1) & 3)) * 16 + (k & 8));
  if (k >= P.K) {  // padding
#pragma unroll
    for (int i = 0; i < NS; ++i) *reinterpret_cast<uint4*>(o + i * plane) = make_uint4(0u, 0u, 0u, 0u);
    *om = make_uint2(0u, 0u);
    return;
  }
  unsigned lo[8], hi[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const long long y = slice_bias(slice_fixed(x[j], emax));
    lo[j] = (unsigned)y;
    hi[j] = (unsigned)((unsigned long long)y >> 32);
  }
#pragma unroll
  for (int i = 1; i <= NS; ++i) {
    uint4 w;
    w.x = __byte_perm(digit_bits(lo[0], hi[0], i), digit_bits(lo[1], hi[1], i), 0x7632);
    w.y = __byte_perm(digit_bits(lo[2], hi[2], i), digit_bits(lo[3], hi[3], i), 0x7632);
    w.z = __byte_perm(digit_bits(lo[4], hi[4], i), digit_bits(lo[5], hi[5], i), 0x7632);
    w.w = __byte_perm(digit_bits(lo[6], hi[6], i), digit_bits(lo[7], hi[7], i), 0x7632);
    *reinterpret_cast<uint4*>(o + (i - 1) * plane) = w;
  }
  uint32_t g[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    g[j] = slice_mag8(x[j], emax);
    sum += slice_magf(x[j], emax);
    count += g[j] != 0u;
  }
  *om = make_uint2(g[0] | g[1] << 8 | g[2] << 16 | g[3] << 24, g[4] | g[5] << 8 | g[6] << 16 | g[7] << 24);
}

template <int NR>
__global__ void __launch_bounds__(256) slice_split_kernel(const __grid_constant__ SplitOps ops, int T) {
  hs_pdl_enter();
  const SplitOp& P = ops.op[blockIdx.y];
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) {
    ops.list->count = 0;
    ops.list->work = 0ull;
  }
  const int Kp = P.steps * KC;
  // 16-byte loads: even strides and lengths, sources aligned and changing between pieces
  const bool vec = P.K % 2 == 0 && P.m.ld % 2 == 0 && (reinterpret_cast<uintptr_t>(P.m.p[0]) & 15) == 0 &&
                   (P.m.nseg == 1 || (P.m.kseg % 8 == 0 && (reinterpret_cast<uintptr_t>(P.m.p[1]) & 15) == 0));
  __shared__ unsigned long long red[8];
  __shared__ float rsum[8];
  __shared__ int rcount[8];
  const int per = 256 / T, t = threadIdx.x % T;  // rows of the block at a time, thread within the row
  // the whole block runs the same number of turns (its barriers)
  for (int r0 = blockIdx.x * per; r0 < P.m.rows; r0 += gridDim.x * per) {
    const int r = r0 + threadIdx.x / T;
    const bool in = r < P.m.rows;
    const long long roff = (long long)(in ? r : 0) * P.m.ld;
    unsigned long long x[NR > 0 ? NR : 1][8];
    unsigned long long mag = 0;  // largest |bits|: its exponent field is the row's
    if (NR > 0) {
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        const int k = 8 * (t + i * T);
        if (in && k < P.K) {
          sl_load(P, vec, roff, k, x[i]);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) x[i][j] = 0ull;
        }
      }
#pragma unroll
      for (int i = 0; i < NR; ++i) mag = sl_mag(x[i], mag);
    } else {
      for (int k = 8 * t; k < P.K; k += 8 * T) {
        sl_load(P, vec, roff, k, x[0]);
        mag = sl_mag(x[0], mag);
      }
    }
    for (int o = (T < 32 ? T : 32) / 2; o > 0; o >>= 1) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    if (T > 32) {
      __syncthreads();
      if (threadIdx.x % 32 == 0) red[threadIdx.x / 32] = mag;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < 8; ++w) mag = max(mag, red[w]);
    }
    // zero rows and rows of the smallest scales (marked) get zero digits
    const int ef = (int)(mag >> 52), emax = ef >= 100 ? ef : 0x7FF;
    float sum = 0.f;
    int count = 0;
    if (in) {
      const int rb = r / P.block, rr = r - rb * P.block;
      unsigned char* row = P.planes + (size_t)rb * P.steps * NS * P.block * ROW_BYTES + rr * ROW_BYTES;
      unsigned char* mags = P.mags + (size_t)rb * ((P.steps + 1) / 2) * P.block * 64 + rr * 64;
      if (NR > 0) {
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          const int k = 8 * (t + i * T);
          if (k < Kp) sl_put(P, row, mags, rr, k, emax, x[i], sum, count);
        }
      } else {
        for (int k = 8 * t; k < Kp; k += 8 * T) {
          if (k < P.K) {
            sl_load(P, vec, roff, k, x[0]);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[0][j] = 0ull;
          }
          sl_put(P, row, mags, rr, k, emax, x[0], sum, count);
        }
      }
    }
    for (int o = (T < 32 ? T : 32) / 2; o > 0; o >>= 1) {
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
      count += __shfl_xor_sync(0xffffffffu, count, o);
    }
    if (T > 32) {
      if (threadIdx.x % 32 == 0) {
        rsum[threadIdx.x / 32] = sum;
        rcount[threadIdx.x / 32] = count;
      }
      __syncthreads();
      sum = 0.f;
      count = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        sum += rsum[w];
        count += rcount[w];
      }
    }
    if (in && t == 0) {
      const int e = ef - 1022;
      P.exps[r] = mag == 0 ? 0 : (ef == 0x7FF || e > 500 || e < -400) ? kSpecial : e;
      P.row[r] = {sum, (float)count};
    }
  }
}

int steps_of(int K) { return (K + KC - 1) / KC; }
size_t up256(size_t v) { return (v + 255) / 256 * 256; }
size_t planes_bytes(int rows, int K, int block) {
  return up256((size_t)((rows + block - 1) / block) * steps_of(K) * NS * block * ROW_BYTES);
}
size_t mags_bytes(int rows, int K, int block) {
  return up256((size_t)((rows + block - 1) / block) * ((steps_of(K) + 1) / 2) * block * 64);
}

}  // namespace

int slices_block(bool is_b) { return is_b ? BN : BM; }
size_t slices_bytes(int rows, int K, bool is_b) {
  const int block = slices_block(is_b);
  return planes_bytes(rows, K, block) + mags_bytes(rows, K, block) + up256((size_t)rows * sizeof(int)) +
         up256((size_t)rows * sizeof(SlRow));
}
size_t slices_scale_bytes(int K) { return up256((size_t)steps_of(K) * KC * sizeof(short)); }
size_t slices_list_bytes(long long M, long long N) {
  return up256(sizeof(SlList) + (size_t)((M + BM - 1) / BM) * (size_t)((N + BN - 1) / BN) * kTileRows *
                                    (sizeof(long long) + sizeof(uint32_t)));
}

bool slices_pay(const SlProblem* probs, const SlMat* mats, int n) {
  // Both sides modelled from measurement: the FP64 kernel at 1.05 TF/s; here
  // 2.1 us per K step of a CTA's tile, 5.4 us for its conversion, stores and S, 22
  // bytes of operand traffic per entry at 2.6 TB/s and 18 us of launches (model and
  // measured: 65536 x 32 x 16 52 and 53 us, 10368 x 666 x 666 317 and 290, 4096 x 64 x
  // 1024 127 and 114; the FP64 kernel's 64, 8760 and 511).
  double dfma = 0.0, tiles = 0.0, steps = 0.0, bytes = 0.0;
  const double sms = device_sms();
  for (int i = 0; i < n; ++i) {
    const SlMat &a = mats[probs[i].a], &b = mats[probs[i].b];
    const double K = (double)a.kseg * a.nseg;
    if (a.rows < 1 || b.rows < 1 || K < 4 || K > 65536) return false;
    const double t = (double)((a.rows + BM - 1) / BM) * ((b.rows + BN - 1) / BN);
    dfma += 2.0 * a.rows * (double)b.rows * K / 1.05e6;
    tiles += t;
    steps += t * ((K + KC - 1) / KC * 2.1 + 5.4);
    bytes += 22.0 * (a.rows + (double)b.rows) * K;
  }
  if (tiles < 1.0) return false;
  const double waves = tiles <= sms ? 1.0 : tiles / sms;
  const double here = 18.0 + bytes / 2.6e6 + steps / tiles * waves;
  return dfma > 1.25 * here;
}

cudaError_t launch_slice_scales(SlMat* mats, int nmat, const SlProblem* probs, int nprob, void* ws, cudaStream_t s) {
  if (nmat > kMaxSplit || nprob > kMaxProblems || nprob < 1) return cudaErrorInvalidValue;
  int set[kMaxSplit];  // of an operand: its first problem, over problems that share operands
  for (int i = 0; i < nmat; ++i) set[i] = kMaxProblems;
  for (int pass = 0; pass < nprob; ++pass)
    for (int i = 0; i < nprob; ++i) {
      int &a = set[probs[i].a], &b = set[probs[i].b];
      const int first = std::min(i, std::min(a, b));
      a = b = first;
    }
  ScaleSets sets{};
  short* scale[kMaxProblems] = {};
  int n = 0, kmax = 0;
  size_t off = 0;
  for (int i = 0; i < nprob; ++i) {
    const SlMat &a = mats[probs[i].a], &b = mats[probs[i].b];
    if (set[probs[i].a] != i) continue;
    scale[i] = reinterpret_cast<short*>(static_cast<char*>(ws) + off);
    sets.set[n++] = ScaleSet{{a, b}, scale[i]};
    off += slices_scale_bytes(a.kseg * a.nseg);
    kmax = std::max(kmax, a.kseg * a.nseg);
  }
  for (int i = 0; i < nmat; ++i) mats[i].scale = set[i] < kMaxProblems ? scale[set[i]] : nullptr;
  hs_launch(slice_scale_kernel, dim3((unsigned)steps_of(kmax), (unsigned)n), 1024, 0, s, sets);
  return cudaGetLastError();
}

cudaError_t launch_gemm_slices(const SlMat* mats, int nmat, const SlProblem* probs, int nprob, SliceBound bound,
                               bool accumulate,
                               void* ws, size_t ws_bytes, int* err, cudaStream_t s) {
  if (nmat > kMaxSplit || nprob > kMaxProblems || nprob < 1) return cudaErrorInvalidValue;
  SplitOp all[kMaxSplit] = {};
  SplitOps ops{};  // of the operands to be split
  size_t off = 0;
  int rmax = 0, kmax = 0, nsplit = 0;
  for (int i = 0; i < nmat; ++i) {
    SplitOp& o = all[i];
    if (!mats[i].scale) return cudaErrorInvalidValue;
    o.m = mats[i];
    o.scale = mats[i].scale;
    o.K = mats[i].kseg * mats[i].nseg;
    o.steps = steps_of(o.K);
    o.block = mats[i].is_b ? BN : BM;
    o.planes = static_cast<unsigned char*>(ws) + off;
    off += planes_bytes(o.m.rows, o.K, o.block);
    o.mags = static_cast<unsigned char*>(ws) + off;
    off += mags_bytes(o.m.rows, o.K, o.block);
    o.exps = reinterpret_cast<int*>(static_cast<char*>(ws) + off);
    off += up256((size_t)o.m.rows * sizeof(int));
    o.row = reinterpret_cast<SlRow*>(static_cast<char*>(ws) + off);
    off += up256((size_t)o.m.rows * sizeof(SlRow));
    if (mats[i].kept) continue;
    ops.op[nsplit++] = o;
    rmax = o.m.rows > rmax ? o.m.rows : rmax;
    kmax = o.K > kmax ? o.K : kmax;
  }
  if (nsplit < 1) return cudaErrorInvalidValue;
  SlList* const list = reinterpret_cast<SlList*>(static_cast<char*>(ws) + off);
  ops.list = list;
  SlGroup g{};
  int tiles = 0;
  for (int i = 0; i < nprob; ++i) {
    const SplitOp &a = all[probs[i].a], &b = all[probs[i].b];
    if (a.K != b.K || a.m.kseg != b.m.kseg || a.K < 1 || a.m.rows < 1 || b.m.rows < 1 || a.block != BM ||
        b.block != BN)
      return cudaErrorInvalidValue;
    SlUnit& u = g.u[g.n++];
    u.M = a.m.rows;
    u.N = b.m.rows;
    u.K = a.K;
    u.ldc = probs[i].ldc;
    u.c = probs[i].c;
    u.pa = a.planes;
    u.pb = b.planes;
    u.ga = a.mags;
    u.gb = b.mags;
    u.ea = a.exps;
    u.eb = b.exps;
    u.ra = a.row;
    u.rb = b.row;
    // bound <= b(K) 2^-53 S with b = 2 sqrt(K), and K - 1 (the last rounding takes one)
    // where that is less or a chain's bound will do. The 19
    // pairs of levels 7..9 take one FP32 add (truncated) each per 16 columns, up to 192
    // columns; random digits sum to `low`, 8 times that means that they are not
    const double sq = 2.0 * std::sqrt((double)u.K), bk = bound == kBoundEntry && sq < u.K - 1.0 ? sq : u.K > 1 ? u.K - 1.0 : 1e-9;
    const double adds = 19.0 * (u.K < CHUNK * KC ? (u.K + 15) / 16 : CHUNK * KC / 16);
    const double low = std::ldexp(std::sqrt(6.0 * u.K) / 3.0, 14 - 40);
    u.g_round = (float)(std::ldexp(1.0, 30 - 56 + 53) / bk);
    u.g_low = (float)(std::ldexp(adds * low, 30 - 14 - 23 + 53) / bk);
    u.low_max = (float)(8.0 * low);
    if (bound == kBoundRows) {  // marked rows only
      u.g_round = u.g_low = 0.f;
      u.low_max = INFINITY;
    }
    u.a = a.m;
    u.b = b.m;
    // |sum| < 1.01 2^46 K: the fraction takes the bits that are left of 62
    int lk = 0;
    while ((1ll << lk) < u.K) ++lk;
    u.frac = lk < 15 ? 15 - lk : 0;
    if (lk > 16) return cudaErrorInvalidValue;
    u.tile_start = tiles;
    u.tiles_n = (u.N + BN - 1) / BN;
    const long long t = (long long)((u.M + BM - 1) / BM) * u.tiles_n;
    if (tiles + t > INT_MAX) return cudaErrorInvalidValue;
    tiles += (int)t;
  }
  const size_t rows = (size_t)tiles * kTileRows;
  if (off + sizeof(SlList) + rows * (sizeof(long long) + sizeof(uint32_t)) > ws_bytes) return cudaErrorInvalidValue;
  const int sms = device_sms();
  // threads per row: one piece of 8 columns each up to a warp, then up to four,
  // then the block with up to three
  const int pieces = steps_of(kmax) * (KC / 8);
  int T = 4;
  while (T < 32 && T < pieces) T *= 2;
  if (pieces > 128) T = 256;
  const int nr = (pieces + T - 1) / T, per = 256 / T;
  int gx = (rmax + per - 1) / per;
  if (gx > sms * 32) gx = sms * 32;
  const dim3 grid((unsigned)gx, (unsigned)nsplit);
  if (nr == 1)
    hs_launch(slice_split_kernel<1>, grid, 256, 0, s, ops, T);
  else if (nr == 2)
    hs_launch(slice_split_kernel<2>, grid, 256, 0, s, ops, T);
  else if (nr == 3)
    hs_launch(slice_split_kernel<3>, grid, 256, 0, s, ops, T);
  else if (nr == 4 && T == 32)
    hs_launch(slice_split_kernel<4>, grid, 256, 0, s, ops, T);
  else
    hs_launch(slice_split_kernel<0>, grid, 256, 0, s, ops, T);
  const auto gemm = accumulate ? gemm_sl_kernel<true> : gemm_sl_kernel<false>;
  cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(gemm), SMEM);
  if (e == cudaSuccess) e = ensure_smem_attr(reinterpret_cast<const void*>(mag_kernel), MSMEM);
  if (e != cudaSuccess) return e;
  uint32_t* const masks = reinterpret_cast<uint32_t*>(list->at + rows);
  hs_launch(mag_kernel, (unsigned)(tiles < 2 * sms ? tiles : 2 * sms), MNT, MSMEM, s, g, tiles, masks, list, err);
  // a third of the work, where the product has tiles enough for fma_kernel's CTAs
  unsigned long long fmas = 0;
  long long tiles64 = 0;
  for (int i = 0; i < g.n; ++i) {
    fmas += (unsigned long long)g.u[i].M * g.u[i].N * g.u[i].K;
    tiles64 += (long long)((g.u[i].M + FT - 1) / FT) * ((g.u[i].N + FT - 1) / FT);
  }
  const unsigned long long limit = tiles64 >= 2 * sms && tiles64 < INT_MAX / 2 ? fmas / 3 : ~0ull;
  hs_launch(gemm, (unsigned)(tiles < sms ? tiles : sms), NT, SMEM, s, g, tiles, limit, masks, list, err);
  hs_launch(fma_kernel, (unsigned)(4 * sms), 256, 0, s, g, accumulate, limit, (const uint32_t*)masks,
            (const SlList*)list);
  return cudaGetLastError();
}

}  // namespace hs
