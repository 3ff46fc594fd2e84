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
// term was 1.7 times the error of an FP64 chain.) The one rounding left is that
// of the final 64-bit integer to FP64.
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
// A row or column that holds an infinity or NaN, or whose scale leaves
// [2^-400, 2^500], is marked; its entries are computed by plain FP64 dot
// products in the epilogue, so non-finite values propagate as in a chain of
// FP64 FMAs.
#include <climits>

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

struct SlUnit {
  int M, N, K, ldc;
  int tile_start, tiles_n;
  int frac;  // extra fraction bits of the 64-bit sums
  double* c;
  const unsigned char* pa;  // digit planes
  const unsigned char* pb;
  const int* ea;
  const int* eb;
  SlMat a, b;  // FP64 sources, for marked rows and columns
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

struct SlTile {
  int u, m0, n0;
};

__device__ __forceinline__ SlTile tile_at(const SlGroup& g, int t) {
  int u = 0;
  while (u + 1 < g.n && t >= g.u[u + 1].tile_start) ++u;
  t -= g.u[u].tile_start;
  return {u, (t / g.u[u].tiles_n) * BM, (t % g.u[u].tiles_n) * BN};
}

// Plain FP64 dot product of row m of A and row n of B.
__device__ __noinline__ double plain_dot(const SlMat& a, const SlMat& b, int m, int n) {
  double v = 0.0;
  for (int s = 0; s < a.nseg; ++s) {
    const double* pa = a.p[s] + (long long)m * a.ld;
    const double* pb = b.p[s] + (long long)n * b.ld;
    const bool neg = a.neg[s] != b.neg[s];
    for (int k = 0; k < a.kseg; ++k) v = fma(neg ? -pa[k] : pa[k], pb[k], v);
  }
  return v;
}

__global__ void __launch_bounds__(NT, 1) gemm_sl_kernel(const __grid_constant__ SlGroup g, int total_tiles,
                                                        bool accumulate, int* __restrict__ err) {
  hs_pdl_enter();
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
    long long it = 0, chunk = 0;
    bool any = false, ok = true, ready = false;
    for (int t = blockIdx.x; ok && t < total_tiles; t += gridDim.x) {
      const SlTile r = tile_at(g, t);
      const int steps = (g.u[r.u].K + KC - 1) / KC;
      for (int k0 = 0; ok && k0 < steps; k0 += CHUNK, ++chunk) {
        const int k1 = k0 + CHUNK < steps ? k0 + CHUNK : steps;
        for (int k = k0; k < k1; ++k) {
          const int s = (int)(it % STAGES);
          ok = ready || wait(&full[s], it / STAGES, 12);
          // the first half of the accumulators, then the second: a chunk's last
          // step hands the first half to the epilogue while the second still
          // multiplies, and its first step needs the second half later
          if (ok && k == k0 && chunk > 0)
            ok = wait(&tempty[0], chunk - 1, 14);
          if (!ok) break;
          fence_after();
          if (s == 0)
            step_mmas<0, 3>(leader, tmem, da0, db0, k == k0);
          else
            step_mmas<0, 3>(leader, tmem, da1, db1, k == k0);
          any = true;
          if (k == k1 - 1) mma_commit_by(leader, smem_u32(&tfull[0]));
          if (k == k0 && chunk > 0) {
            ok = wait(&tempty[1], chunk - 1, 15);
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
          if (k == k1 - 1) mma_commit_by(leader, smem_u32(&tfull[1]));
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
    long long chunk = 0;
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
      for (int k0 = 0; k0 < steps; k0 += CHUNK, ++chunk) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          // one lane polls: 512 polling threads slowed the products they wait for
          int got = 1;
          if (lane == 0) got = mbar_wait(smem_u32(&tfull[h]), (uint32_t)(chunk & 1), abort_flag, err, 13);
          ok = ok && __shfl_sync(0xffffffffu, got, 0);
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
        }
        if (!ok) break;
      }
      if (!ok) break;
      const int row0 = r.m0 + q * 32, row = row0 + lane;
      const int colp = r.n0 + part * PART;  // this warp's first column
      const int ea = row < U.M ? __ldg(U.ea + row) : 0;
      const int ebl = (lane < PART && colp + lane < U.N) ? __ldg(U.eb + colp + lane) : 0;
      if (__any_sync(0xffffffffu, ea == kSpecial || ebl == kSpecial)) {
        if (row < U.M)
          for (int n = colp; n < colp + PART && n < U.N; ++n) {
            double* dst = U.c + (long long)row * U.ldc + n;
            const double v = plain_dot(U.a, U.b, row, n);
            *dst = accumulate ? *dst + v : v;
          }
        continue;
      }
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
          if (row0 + i < U.M && col < U.N) {
            double2 x = *reinterpret_cast<const double2*>(&stg[i * STG_LD + 2 * (lane & 1)]);
            double* dst = U.c + (long long)(row0 + i) * U.ldc + col;
            if (vec && col + 1 < U.N) {
              if (accumulate) {
                const double2 y = *reinterpret_cast<const double2*>(dst);
                x.x += y.x;
                x.y += y.y;
              }
              *reinterpret_cast<double2*>(dst) = x;
            } else {
              dst[0] = accumulate ? dst[0] + x.x : x.x;
              if (col + 1 < U.N) dst[1] = accumulate ? dst[1] + x.y : x.y;
            }
          }
        }
        __syncwarp();
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

// ---- the digit planes -------------------------------------------------------------

// Row block rb (of `block` rows), K step ks: [NS][block][32] BF16 at
// ((rb * steps) + ks) * NS * block * 64 bytes, the 16-byte quarters of row r
// exchanged by the 64-byte swizzle (q ^ (r / 2) % 4). The columns past K are zero; rows past the
// end are left as they are (they only reach entries that are not stored).
struct SplitOp {
  SlMat m;
  int K, steps, block;
  unsigned char* planes;
  int* exps;  // [rows]
};
constexpr int kMaxSplit = 2 * kMaxProblems;
struct SplitOps {
  SplitOp op[kMaxSplit];
};

// Bits of entry k of a row, its sign flipped where the source is negated (as an
// integer: negating a double takes the FP64 pipe).
__device__ __forceinline__ unsigned long long sl_at(const SlMat& m, long long roff, int k) {
  const int s = k >= m.kseg;
  const double* p = s ? m.p[1] + roff - m.kseg : m.p[0] + roff;
  return f64_bits(p[k]) ^ ((unsigned long long)m.neg[s] << 63);
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
}

__device__ __forceinline__ unsigned long long sl_mag(const unsigned long long (&x)[8], unsigned long long mag) {
#pragma unroll
  for (int j = 0; j < 8; ++j) mag = max(mag, x[j] & 0x7FFFFFFFFFFFFFFFull);
  return mag;
}

__device__ __forceinline__ void sl_put(const SplitOp& P, unsigned char* row, int rr, int k, int emax,
                                       const unsigned long long (&x)[8]) {
  const size_t plane = (size_t)P.block * ROW_BYTES;
  unsigned char* o = row + (size_t)(k / KC) * NS * plane + (((k % KC) / 8) ^ ((rr >> 1) & 3)) * 16;
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
}

template <int NR>
__global__ void __launch_bounds__(256) slice_split_kernel(const __grid_constant__ SplitOps ops, int T) {
  hs_pdl_enter();
  const SplitOp& P = ops.op[blockIdx.y];
  const int Kp = P.steps * KC;
  // 16-byte loads: even strides and lengths, sources aligned and changing between pieces
  const bool vec = P.K % 2 == 0 && P.m.ld % 2 == 0 && (reinterpret_cast<uintptr_t>(P.m.p[0]) & 15) == 0 &&
                   (P.m.nseg == 1 || (P.m.kseg % 8 == 0 && (reinterpret_cast<uintptr_t>(P.m.p[1]) & 15) == 0));
  __shared__ unsigned long long red[8];
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
    if (!in) continue;
    // zero rows and rows of the smallest scales (marked) get zero digits
    const int ef = (int)(mag >> 52), emax = ef >= 100 ? ef : 0x7FF;
    if (t == 0) {
      const int e = ef - 1022;
      P.exps[r] = mag == 0 ? 0 : (ef == 0x7FF || e > 500 || e < -400) ? kSpecial : e;
    }
    const int rb = r / P.block, rr = r - rb * P.block;
    unsigned char* row = P.planes + (size_t)rb * P.steps * NS * P.block * ROW_BYTES + rr * ROW_BYTES;
    if (NR > 0) {
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        const int k = 8 * (t + i * T);
        if (k < Kp) sl_put(P, row, rr, k, emax, x[i]);
      }
    } else {
      for (int k = 8 * t; k < Kp; k += 8 * T) {
        if (k < P.K) {
          sl_load(P, vec, roff, k, x[0]);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) x[0][j] = 0ull;
        }
        sl_put(P, row, rr, k, emax, x[0]);
      }
    }
  }
}

int steps_of(int K) { return (K + KC - 1) / KC; }
size_t up256(size_t v) { return (v + 255) / 256 * 256; }
size_t planes_bytes(int rows, int K, int block) {
  return up256((size_t)((rows + block - 1) / block) * steps_of(K) * NS * block * ROW_BYTES);
}

}  // namespace

size_t slices_bytes(int rows, int K, bool is_b) {
  return planes_bytes(rows, K, is_b ? BN : BM) + up256((size_t)rows * sizeof(int));
}
int slices_block(bool is_b) { return is_b ? BN : BM; }

bool slices_pay(const SlProblem* probs, const SlMat* mats, int n) {
  // Both sides modelled from measurement: the FP64 kernel at 1.05 TF/s; here
  // 2.1 us per K step of a CTA's tile, 4.5 us for its conversion and stores, 22
  // bytes of operand traffic per entry at 3 TB/s and 15 us of launches.
  double dfma = 0.0, tiles = 0.0, steps = 0.0, bytes = 0.0;
  const double sms = device_sms();
  for (int i = 0; i < n; ++i) {
    const SlMat &a = mats[probs[i].a], &b = mats[probs[i].b];
    const double K = (double)a.kseg * a.nseg;
    if (a.rows < 1 || b.rows < 1 || K < 1 || K > 65536) return false;
    const double t = (double)((a.rows + BM - 1) / BM) * ((b.rows + BN - 1) / BN);
    dfma += 2.0 * a.rows * (double)b.rows * K / 1.05e6;
    tiles += t;
    steps += t * ((K + KC - 1) / KC * 2.1 + 4.5);
    bytes += 22.0 * (a.rows + (double)b.rows) * K;
  }
  if (tiles < 1.0) return false;
  const double waves = tiles <= sms ? 1.0 : tiles / sms;
  const double here = 15.0 + bytes / 3e6 + steps / tiles * waves;
  return dfma > 1.25 * here;
}

cudaError_t launch_gemm_slices(const SlMat* mats, int nmat, const SlProblem* probs, int nprob, bool accumulate,
                               void* ws, size_t ws_bytes, int* err, cudaStream_t s) {
  if (nmat > kMaxSplit || nprob > kMaxProblems || nprob < 1) return cudaErrorInvalidValue;
  SplitOps ops{};
  size_t off = 0;
  int rmax = 0, kmax = 0;
  for (int i = 0; i < nmat; ++i) {
    SplitOp& o = ops.op[i];
    o.m = mats[i];
    o.K = mats[i].kseg * mats[i].nseg;
    o.steps = steps_of(o.K);
    o.block = mats[i].is_b ? BN : BM;
    o.planes = static_cast<unsigned char*>(ws) + off;
    off += planes_bytes(o.m.rows, o.K, o.block);
    o.exps = reinterpret_cast<int*>(static_cast<char*>(ws) + off);
    off += up256((size_t)o.m.rows * sizeof(int));
    rmax = o.m.rows > rmax ? o.m.rows : rmax;
    kmax = o.K > kmax ? o.K : kmax;
  }
  if (off > ws_bytes) return cudaErrorInvalidValue;
  SlGroup g{};
  int tiles = 0;
  for (int i = 0; i < nprob; ++i) {
    const SplitOp &a = ops.op[probs[i].a], &b = ops.op[probs[i].b];
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
    u.ea = a.exps;
    u.eb = b.exps;
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
  const dim3 grid((unsigned)gx, (unsigned)nmat);
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
  const cudaError_t e = ensure_smem_attr(reinterpret_cast<const void*>(gemm_sl_kernel), SMEM);
  if (e != cudaSuccess) return e;
  hs_launch(gemm_sl_kernel, (unsigned)(tiles < sms ? tiles : sms), NT, SMEM, s, g, tiles, accumulate, err);
  return cudaGetLastError();
}

}  // namespace hs
