// FP64 complex GEMM on the tensor cores: operands cut into integer slices.
//
// GB300's FP64 pipe gives about 1.1 TF/s, its FP16 tensor cores 1900. Every
// operand element is written as a fixed-point number of 63 bits relative to
// the largest magnitude of its row (2^E above it), and that number as seven
// balanced base-512 digits d_1 .. d_7 in [-256, 256], which FP16 holds
// exactly (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59, 95 (2012), and Mukunoki et al., ISC 2020, for FP16 tensor
// cores). The product is
//   sum_g 2^(-9 (g - 1)) D_g,  D_g = sum_{i + j = g + 1} d_i(A) d_j(B)^T,
// for g = 1 .. 7: 28 digit products; what is left out is below 2^-63 of the
// two rows' largest magnitudes per term. Each digit product is at most 2^16
// in magnitude, so 256 of them (four K blocks of 64) add up without any
// rounding in the FP32 accumulators of tcgen05.mma; the epilogue warps then
// move the sums out of TMEM: groups 7 .. EX + 1 into FP32 (their rounding
// lies 2^-24 below 2^(-9 EX) of the result), groups EX .. 1 into 64-bit
// integers, exactly. EX is 5 where the rows' and columns' 2-norms bound the
// integers below 2^63 (Cauchy-Schwarz; the norms, relative to 2^E, come from
// the packing), else 4; the sum may wrap on the way, only its value counts.
//
// Accuracy, RMS error over |a_m| |b_n| against quadruple precision, here and
// from the FP64 kernel, normal operands: K = 160 7.9e-18 / 1.3e-17, K = 1200
// 2.7e-18 / 6.0e-18, K = 20000 1.1e-18 / 4.3e-18.
//
// Measured against the FP64 kernels: product of 1536 x 1000 x 1200 14.7 ->
// 1.3 ms, ladder at o = 15, v = 131, X = 517 983 -> 38 ms, FP64 residual at
// o = 12, v = 72, X = 288 80.7 -> 9.0 ms.
//
// Rows that hold an Inf or NaN cannot be cut: the packing raises a flag on
// the device, the slice kernel then stores nothing, and a guarded launch of
// the FP64 kernel, which otherwise returns at once, computes the product.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace cdfns {

namespace {

constexpr int NS = SLICE_COUNT;  // digits per element
constexpr int SBN = 128;         // output columns per tile
constexpr int CHUNK = 4;         // K blocks per TMEM accumulation (256 terms)
constexpr int NBUF = 3;          // TMEM accumulators in flight (128 columns each)
constexpr uint32_t STASH = NBUF * SBN;  // TMEM columns that hold the FP32 part

// 12 warps: 0-7 epilogue, 8 TMA producer, 9 MMA issuer, 10-11 idle (they
// complete the warpgroup that gives registers away). Launched with 168
// registers a thread (64512 in all); warps 8-11 drop to 56, the epilogue's
// 256 threads rise to 224: 256 x 224 + 128 x 56 = 64512.
constexpr int SLICE_THREADS = 384;

enum { SW_STORE = 0, SW_ADD = 1, SW_BETA = 2 };

struct alignas(64) SliceArgs {
  CUtensorMap mA, mB;  // [slice][row][Kp] planes as one matrix of slice * rows rows
  long M, N;           // complex rows, columns of this product
  long rows_a, rows_b; // plane rows per slice
  long a_row0, b_row0; // first plane row of this product
  const int *ea, *eb;  // per complex row: biased exponent of the largest magnitude
  const int *fa, *fb;  // != 0: the operand holds Inf or NaN
  const float *na, *nb;  // per complex row: squared 2-norm over 4^E
  double2 *C;
  const long *cm, *cn;
  long ldc;
  double2 alpha, beta;
  int alpha_p2;        // alpha is +-2^alpha_e
  int alpha_e, alpha_neg;
  int wmode;
  int num_kb, kb_per_split, m_tiles, n_tiles, k_splits, group_m;
  int *err;
  unsigned long long wait_ns;
};

__device__ __forceinline__ void slice_coords(const SliceArgs &a, int t, int &m, int &n, int &z) {
  const int mn = a.m_tiles * a.n_tiles;
  z = t / mn;
  const int r0 = t - z * mn;
  const int per_group = a.group_m * a.n_tiles;
  const int g = r0 / per_group;
  const int first_m = g * a.group_m;
  const int gsize = min(a.group_m, a.m_tiles - first_m);
  const int r = r0 - g * per_group;
  m = first_m + r % gsize;
  n = r / gsize;
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float *v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
      "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
      "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
      "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
      "r"(__float_as_uint(v[15]))
      : "memory");
}

// d 2^e; the exponent field is adjusted in place unless the value or the
// result is not a normal number
__device__ __forceinline__ double scale_exp(double d, int e) {
  const int hi = __double2hiint(d);
  const int ex = (hi >> 20) & 0x7ff;
  const int ne = ex + e;
  if (ex != 0 && ne > 0 && ne < 2047)
    return __hiloint2double(hi + (e << 20), __double2loint(d));
  return scalbn(d, e);
}

// t as a double, rounded to nearest even, on the integer pipes (the hardware
// conversion runs at the FP64 pipe's rate)
__device__ __forceinline__ double i64_to_f64(long long t) {
  if (t == 0) return 0.0;
  const unsigned long long s = static_cast<unsigned long long>(t) & 0x8000000000000000ull;
  unsigned long long u = t < 0 ? 0ull - static_cast<unsigned long long>(t) : static_cast<unsigned long long>(t);
  const int lz = __clzll(static_cast<long long>(u));
  u <<= lz;
  unsigned long long m = u >> 11;
  const unsigned rem = static_cast<unsigned>(u) & 0x7ffu;
  m += (rem > 0x400u || (rem == 0x400u && (m & 1ull))) ? 1ull : 0ull;
  // the implicit bit of m adds one to the exponent field
  const unsigned long long b = (static_cast<unsigned long long>(1023 + 63 - lz - 1) << 52) + m;
  return __longlong_as_double(static_cast<long long>(b | s));
}

// Persistent CTA or CTA pair, warps as in tc_gemm_kernel (gemm_tc.cu): 0-7
// epilogue, 8 TMA producer, 9 TMEM allocator and MMA issuer; every wait
// bounded. Tiles of UNIT_ROWS real rows x 128 columns: 64-bit sums for 256
// columns would not fit the epilogue's registers. A pair's MMA (256 x 128)
// then reads 96 B of shared memory per SM clock and the copies write as
// much, the same as tc_gemm_kernel's 128 x 256 single-CTA tile. Per tile the
// groups run from 7 to 1, and in each the digit pairs (i, g + 1 - i) over
// the K range, cut into TMEM chunks of four K blocks regardless of the pair.
template <int STAGES, bool PAIR>
__global__ void __launch_bounds__(SLICE_THREADS, 1) slice_gemm_kernel(const __grid_constant__ SliceArgs P) {
  constexpr int A_BYTES = BM * ROW_BYTES;
  constexpr int B_BYTES = (PAIR ? SBN / 2 : SBN) * ROW_BYTES;
  constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  constexpr int UNIT_ROWS = PAIR ? 2 * BM : BM;
  constexpr uint32_t IDESC = make_idesc(UNIT_ROWS, SBN, 0u);
  constexpr int HALF = SBN / 2;  // columns per epilogue warp
  constexpr uint32_t TMEM_COLS = 512;

  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + STAGES * STAGE_BYTES);
  uint64_t *empty = full + STAGES;
  uint64_t *tfull = empty + STAGES;    // [NBUF]
  uint64_t *tempty = tfull + NBUF;     // [NBUF]
  uint64_t *mdone = tempty + NBUF;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mdone + 1);
  double *stage = reinterpret_cast<double *>(smem + STAGES * STAGE_BYTES + 256);  // 8 x 4 KB

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int n_units = P.m_tiles * P.n_tiles * P.k_splits;
#define TC_RANK (PAIR ? static_cast<int>(cluster_rank()) : 0)
#define TC_UNIT0 (PAIR ? static_cast<int>(cluster_id_x()) : static_cast<int>(blockIdx.x))
#define TC_USTEP (PAIR ? static_cast<int>(cluster_count_x()) : static_cast<int>(gridDim.x))

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], PAIR ? 16 : 8);
    }
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 9) tmem_alloc<PAIR>(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
    if (warp == 8) {
      if (lane == 0) {
        // ---------------- TMA producer ----------------
        long it = 0;
        int s = 0;
        uint32_t ph = 1;  // parity of the wait for a free stage
        bool ok = true;
        for (int t = TC_UNIT0; t < n_units && ok; t += TC_USTEP) {
          int m_tile, n_tile, z;
          slice_coords(P, t, m_tile, n_tile, z);
          const int kb0 = z * P.kb_per_split;
          const int kb1 = min(P.num_kb, kb0 + P.kb_per_split);
          const int ya = static_cast<int>(P.a_row0) + m_tile * UNIT_ROWS + TC_RANK * BM;
          const int yb = static_cast<int>(P.b_row0) + n_tile * SBN + (PAIR ? TC_RANK * (SBN / 2) : 0);
          for (int g = NS; g >= 1 && ok; --g)
            for (int p = 0; p < g && ok; ++p) {
              const int yap = ya + p * static_cast<int>(P.rows_a);
              const int ybp = yb + (g - 1 - p) * static_cast<int>(P.rows_b);
              for (int kb = kb0; kb < kb1; ++kb, ++it) {
                if (!mbar_wait(&empty[s], ph, P.wait_ns)) {
                  atomicExch(P.err, 1);
                  ok = false;
                  break;
                }
                uint8_t *st = smem + s * STAGE_BYTES;
                if constexpr (PAIR) {
                  if (TC_RANK == 0) mbar_expect_tx(&full[s], 2 * STAGE_BYTES);
                  const uint32_t fb = leader_addr(smem_u32(&full[s]));
                  tma_load_2d_pair(st, &P.mA, fb, kb * 64, yap);
                  tma_load_2d_pair(st + A_BYTES, &P.mB, fb, kb * 64, ybp);
                } else {
                  mbar_expect_tx(&full[s], STAGE_BYTES);
                  tma_load_2d(st, &P.mA, &full[s], kb * 64, yap);
                  tma_load_2d(st + A_BYTES, &P.mB, &full[s], kb * 64, ybp);
                }
                if (++s == STAGES) {
                  s = 0;
                  ph ^= 1u;
                }
              }
            }
        }
        // no copy may outlive the CTA's shared memory (see tc_gemm_kernel)
        if (TC_RANK == 0) {
          for (long i = (it > STAGES ? it - STAGES : 0); i < it; ++i) {
            if (!mbar_wait(&full[i % STAGES], static_cast<uint32_t>(i / STAGES) & 1u, DRAIN_NS))
              atomicExch(P.err, 1);
          }
        }
      }
    } else if (warp == 9) {
      if (TC_RANK == 0 && elect_one()) {
        // ---------------- MMA issuer (the leader of a pair) ----------------
        long c = 0;
        int buf = 0, s = 0;
        uint32_t bph = 0, ph = 0;  // parities of the TMEM buffers and the stages
        bool ok = true;
        const uint64_t desc0 = sw128_desc(smem_u32(smem));
        for (int t = TC_UNIT0; t < n_units && ok; t += TC_USTEP) {
          int m_tile, n_tile, z;
          slice_coords(P, t, m_tile, n_tile, z);
          const int kb0 = z * P.kb_per_split;
          const int nkb = min(P.num_kb, kb0 + P.kb_per_split) - kb0;
          for (int g = NS; g >= 1 && ok; --g) {
            for (int left = g * nkb; left > 0 && ok; left -= CHUNK, ++c) {
              if (c >= NBUF && !mbar_wait(&tempty[buf], bph ^ 1u, P.wait_ns)) {
                atomicExch(P.err, 1);
                ok = false;
                break;
              }
              tc_fence_after();
              const uint32_t dt = tmem + buf * SBN;
              const int nb = min(left, CHUNK);
              for (int i = 0; i < nb; ++i) {
                if (!mbar_wait(&full[s], ph, P.wait_ns)) {
                  atomicExch(P.err, 1);
                  ok = false;
                  break;
                }
                tc_fence_after();
                // descriptor addresses count 16 bytes
                const uint64_t da = desc0 + static_cast<uint32_t>(s * (STAGE_BYTES >> 4));
#pragma unroll
                for (int kk = 0; kk < ROW_BYTES / 32; ++kk)
                  mma<true, PAIR>(dt, da + 2 * kk, da + (A_BYTES >> 4) + 2 * kk, IDESC,
                                  (i > 0 || kk > 0) ? 1u : 0u);
                mma_commit_both<PAIR>(&empty[s]);
                if (++s == STAGES) {
                  s = 0;
                  ph ^= 1u;
                }
              }
              mma_commit_both<PAIR>(&tfull[buf]);
              if (++buf == NBUF) {
                buf = 0;
                bph ^= 1u;
              }
            }
          }
        }
        mma_commit_self<PAIR>(mdone);
        if (!mbar_wait(mdone, 0u, DRAIN_NS)) atomicExch(P.err, 1);
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    // ---------------- epilogue: 8 warps ----------------
    const int q = warp & 3;
    const int h = warp >> 2;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    int buf = 0;
    uint32_t bph = 0;
    bool ok = true;
    // one chunk: wait for it, hand its 64 columns to f(column, value), free it
    auto drain = [&](auto &&f) {
      if (!mbar_wait(&tfull[buf], bph, P.wait_ns)) {
        ok = false;
        return;
      }
      tc_fence_after();
      const uint32_t base = tmem + lanes + buf * SBN + h * HALF;
#pragma unroll
      for (int j = 0; j < HALF; j += 16) {
        float v[16];
        tmem_ld16(base + j, v);
#pragma unroll
        for (int u = 0; u < 16; ++u) f(j + u, v[u]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR)
          mbar_arrive_cluster(leader_addr(smem_u32(&tempty[buf])));
        else
          mbar_arrive(&tempty[buf]);
      }
      if (++buf == NBUF) {
        buf = 0;
        bph ^= 1u;
      }
    };
    for (int t = TC_UNIT0; t < n_units && ok; t += TC_USTEP) {
      int m_tile, n_tile, z;
      slice_coords(P, t, m_tile, n_tile, z);
      const int kb0 = z * P.kb_per_split;
      const int nkb = min(P.num_kb, kb0 + P.kb_per_split) - kb0;
      // exponents (stored biased by 1022: row below 2^(e - 1022)) and norms
      // of this warp's rows and columns; those beyond the product are
      // computed on whatever the planes hold there and not stored
      const long nbase = static_cast<long>(n_tile) * SBN + h * HALF;
      const long mbase = (static_cast<long>(m_tile) * UNIT_ROWS + TC_RANK * BM) / 2 + q * 16;
      const long mrow = mbase + (lane >> 1);
      bool ex5;
      {
        const float na = mrow < P.M ? P.na[P.a_row0 / 2 + mrow] : 0.f;
        const float nb0 = nbase + lane < P.N ? P.nb[P.b_row0 + nbase + lane] : 0.f;
        const float nb1 = nbase + 32 + lane < P.N ? P.nb[P.b_row0 + nbase + 32 + lane] : 0.f;
        const float a = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(na)));
        const float b = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(nb0, nb1))));
        ex5 = a * b < 0x1p19f;  // |a| |b| < 725: sums below 2^52 725 < 2^62
      }
      {
        float lf[HALF];
#pragma unroll
        for (int j = 0; j < HALF; ++j) lf[j] = 0.f;
        for (int g = NS; g > (ex5 ? 5 : 4) && ok; --g) {
#pragma unroll
          for (int j = 0; j < HALF; ++j) lf[j] *= 0x1p-9f;
          for (int left = g * nkb; left > 0 && ok; left -= CHUNK)
            drain([&](int j, float x) { lf[j] += x; });
        }
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < HALF; j += 16) tmem_st16(tmem + lanes + STASH + h * HALF + j, lf + j);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      }
      long long acc[HALF];
#pragma unroll
      for (int j = 0; j < HALF; ++j) acc[j] = 0;
      // group g counts 2^(9 (EX - g)) in units of group EX's last place:
      // group 1 in the upper word (36 places) or by a 32 x 32 -> 64 product
      for (int g = ex5 ? 5 : 4; g >= 1 && ok; --g) {
        const int sh = 9 * ((ex5 ? 5 : 4) - g);
        if (sh < 32) {
          const int mul = 1 << sh;
          for (int left = g * nkb; left > 0 && ok; left -= CHUNK)
            drain([&](int j, float x) {
              asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc[j]) : "r"(__float2int_rn(x)), "r"(mul));
            });
        } else {
          for (int left = g * nkb; left > 0 && ok; left -= CHUNK)
            drain([&](int j, float x) {
              const unsigned xi = static_cast<unsigned>(__float2int_rn(x)) << 4;
              acc[j] += static_cast<long long>(static_cast<unsigned long long>(xi) << 32);
            });
        }
      }
      if (!ok) break;
      // value = (acc + 2^-9 lf) 2^(Ea + Eb - 16 - 9 (EX - 1))
      const bool skip = (*P.fa | *P.fb) != 0;
      const int ea = (mrow < P.M ? P.ea[P.a_row0 / 2 + mrow] : 1) - 2 * 1022 - 25 - (ex5 ? 36 : 27) +
                     (P.alpha_p2 ? P.alpha_e : 0);
      const int ebl = nbase + lane < P.N ? P.eb[P.b_row0 + nbase + lane] : 1;
      const int ebh = nbase + 32 + lane < P.N ? P.eb[P.b_row0 + nbase + 32 + lane] : 1;
      long roff = 0;
      if (lane < 16 && mbase + lane < P.M)
        roff = P.cm ? P.cm[mbase + lane] : (mbase + lane) * P.ldc;
      double *stg = stage + warp * 512;  // 32 rows x 16 columns
      const int col = lane & 15, hf = lane >> 4;
#pragma unroll
      for (int j = 0; j < HALF; j += 16) {
        float lf[16];
        tmem_ld16(tmem + lanes + STASH + h * HALF + j, lf);
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const int eb = __shfl_sync(0xffffffffu, j < 32 ? ebl : ebh, (j + u) & 31);
          const long long a = acc[j + u];
          double d = scale_exp(i64_to_f64(a), a == 0 ? 0 : 9) + f32_to_f64(lf[u]);
          d = d == 0.0 ? 0.0 : scale_exp(d, ea + eb);
          if (P.alpha_neg) d = -d;
          stg[lane * 16 + (u ^ (lane & 15))] = d;
        }
        __syncwarp();
        const long n = nbase + j + col;
        const bool col_ok = n < P.N && !skip;
        const long cno = col_ok ? (P.cn ? P.cn[n] : n) : 0;
#pragma unroll
        for (int rr = 0; rr < 8; ++rr) {
          const int r = 2 * rr + hf;
          double re = stg[(2 * r) * 16 + (col ^ ((2 * r) & 15))];
          double im = stg[(2 * r + 1) * 16 + (col ^ ((2 * r + 1) & 15))];
          const long ro = __shfl_sync(0xffffffffu, roff, r);
          if (!col_ok || mbase + r >= P.M) continue;
          double2 *o = P.C + ro + cno;
          if (!P.alpha_p2) {
            const double2 x = cmul(P.alpha, make_double2(re, im));
            re = x.x;
            im = x.y;
          }
          if (P.wmode == SW_ADD) {
            atomicAdd(&o->x, re);
            atomicAdd(&o->y, im);
          } else if (P.wmode == SW_STORE) {
            *o = make_double2(re, im);
          } else {
            *o = cadd(make_double2(re, im), cmul(P.beta, *o));
          }
        }
        __syncwarp();
      }
    }
    if (!ok && lane == 0) atomicExch(P.err, 1);
  }
  tc_fence_before();
  if constexpr (PAIR) {
    // as in tc_gemm_kernel: after an expired wait let copies still in flight land
    if (threadIdx.x == 0 && *reinterpret_cast<volatile int *>(P.err)) {
      const unsigned long long t0 = global_ns();
      while (global_ns() - t0 < 50000000ull) {
      }
    }
  }
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();
  if (warp == 9) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc<PAIR>(tmem, TMEM_COLS);
  }
#undef TC_RANK
#undef TC_UNIT0
#undef TC_USTEP
}

// ---------------------------------------------------------------------------
// operands: row exponents, then digits
// ---------------------------------------------------------------------------
struct SideArgs {
  const double2 *src;
  const long *rt, *kt;
  long ld, rows;
  bool conj, rows_unit, expand;
  __half *planes;
  int *e;     // [rows] exponent fields, then the Inf/NaN flag
  float *n2;  // [rows] squared 2-norms over 4^E
};

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// e[row] = the largest exponent field of the row's components (at least 1),
// e[rows] != 0 if any is 2047. One warp per item: 32 rows x 16 k with lanes
// along the rows where those are neighbours in memory, else one row x 256 k
// with lanes along k, 8 loads in flight: on small operands the time is one
// item's latency (items four times as long took 36 us at any size), on
// large ones the read of the operand.
__global__ void __launch_bounds__(256) slice_exp_kernel(SideArgs a, SideArgs b, long K, long items_a,
                                                        long items) {
  const int lane = threadIdx.x & 31;
  const long nw = static_cast<long>(gridDim.x) * 8;
  for (long w = blockIdx.x * 8L + (threadIdx.x >> 5); w < items; w += nw) {
    const SideArgs &s = w < items_a ? a : b;
    const long it = w < items_a ? w : w - items_a;
    int m = 1;
    if (s.rows_unit) {
      const long nk = (K + 15) / 16;
      const long r = (it / nk) * 32 + lane, k0 = (it % nk) * 16, k1 = min(K, k0 + 16);
      if (r < s.rows) {
        const long ro = s.rt ? s.rt[r] : r * s.ld;
#pragma unroll 8
        for (long k = k0; k < k1; ++k) {
          const double2 x = s.src[ro + (s.kt ? s.kt[k] : k)];
          m = max(m, max(exp_field(x.x), exp_field(x.y)));
        }
        atomicMax(&s.e[r], m);
        if (m == 2047) s.e[s.rows] = 1;
      }
    } else {
      const long nk = (K + 255) / 256;
      const long r = it / nk, k0 = (it % nk) * 256, k1 = min(K, k0 + 256);
      const long ro = s.rt ? s.rt[r] : r * s.ld;
#pragma unroll 8
      for (long k = k0 + lane; k < k1; k += 32) {
        const double2 x = s.src[ro + (s.kt ? s.kt[k] : k)];
        m = max(m, max(exp_field(x.x), exp_field(x.y)));
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) {
        atomicMax(&s.e[r], m);
        if (m == 2047) s.e[s.rows] = 1;
      }
    }
  }
}

// x 2^(62 - E) rounded to an integer, E = field - 1022
__device__ __forceinline__ long long to_fixed(double x, int field) {
  const long long b = __double_as_longlong(x);
  const int f = static_cast<int>(b >> 52) & 0x7ff;
  long long m = b & 0xfffffffffffffll;
  if (f) m |= 1ll << 52;
  const int sh = 9 - (field - max(f, 1));
  if (sh >= 0) m <<= sh;
  else if (sh >= -54) m = (m + (1ll << (-sh - 1))) >> -sh;
  else m = 0;
  return b < 0 ? -m : m;
}

// two digits in [-256, 256] as FP16, exactly: 1024 + (d + 256) is a half with
// unit last place
__device__ __forceinline__ __half2 digits2(int x, int y) {
  const unsigned u = (0x6500u + static_cast<unsigned>(x)) | ((0x6500u + static_cast<unsigned>(y)) << 16);
  return __hsub2(*reinterpret_cast<const __half2 *>(&u), __float2half2_rn(1280.0f));
}

// one complex element's digits into its place of every slice; the lanes of a
// warp hold 32 neighbouring k of one row
__device__ __forceinline__ void store_digits(const SideArgs &s, long r, long kc, long Kp, double2 x,
                                             int field) {
  long long re = to_fixed(x.x, field), im = to_fixed(x.y, field);
  if (s.conj) im = -im;
  // |x|^2 4^-E of this element, summed over the warp's 32 k
  const float fr = static_cast<float>(static_cast<int>(re >> 32)) * 0x1p-30f;
  const float fi = static_cast<float>(static_cast<int>(im >> 32)) * 0x1p-30f;
  float n2 = fr * fr + fi * fi;
  for (int o = 16; o > 0; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s.n2[r], n2);
  __half2 *pl = reinterpret_cast<__half2 *>(s.planes);
  const long hk = Kp / 2;
  const long prow = s.expand ? 2 * r : r, prows = s.expand ? 2 * s.rows : s.rows;
#pragma unroll
  for (int d = NS - 1; d >= 0; --d) {
    int dr, di;
    if (d > 0) {
      dr = static_cast<int>((re + 256) & 511) - 256;
      di = static_cast<int>((im + 256) & 511) - 256;
      re = (re - dr) >> 9;
      im = (im - di) >> 9;
    } else {
      dr = static_cast<int>(re);
      di = static_cast<int>(im);
    }
    const long o = (d * prows + prow) * hk + kc;
    if (s.expand) {
      pl[o] = digits2(dr, -di);
      pl[o + hk] = digits2(di, dr);
    } else {
      pl[o] = digits2(dr, di);
    }
  }
}

// Digit planes of both operands: 32 x 32 tiles, read along the direction that
// is contiguous in the source (transposed through shared memory when that is
// the rows) and written along k. HBM bound: 16 B read, 28 B (56 B for the
// expanded A side) written per element.
__global__ void __launch_bounds__(256) slice_pack_kernel(SideArgs a, SideArgs b, long K, long Kp,
                                                         long items_a, long items) {
  __shared__ double2 tile[32][33];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const long nk = Kp / 64;
  for (long w = blockIdx.x; w < items; w += gridDim.x) {
    const SideArgs &s = w < items_a ? a : b;
    const long it = w < items_a ? w : w - items_a;
    const long r0 = (it / nk) * 32, k0 = (it % nk) * 32;
    if (s.rows_unit) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long k = k0 + ty + 8 * j, r = r0 + tx;
        double2 x = make_double2(0.0, 0.0);
        if (k < K && r < s.rows) x = s.src[(s.rt ? s.rt[r] : r * s.ld) + (s.kt ? s.kt[k] : k)];
        tile[ty + 8 * j][tx] = x;
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long r = r0 + ty + 8 * j;
        if (r < s.rows) store_digits(s, r, k0 + tx, Kp, tile[tx][ty + 8 * j], max(s.e[r], 1));
      }
      __syncthreads();
    } else {
      double2 x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long k = k0 + tx, r = r0 + ty + 8 * j;
        x[j] = make_double2(0.0, 0.0);
        if (k < K && r < s.rows) x[j] = s.src[(s.rt ? s.rt[r] : r * s.ld) + (s.kt ? s.kt[k] : k)];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long r = r0 + ty + 8 * j;
        if (r < s.rows) store_digits(s, r, k0 + tx, Kp, x[j], max(s.e[r], 1));
      }
    }
  }
}

template <int STAGES, bool PAIR>
void launch_slices(SliceArgs &a, const SlicePlanes &A, const SlicePlanes &B, int units, int sms,
                   cudaStream_t st) {
  constexpr int STAGE_BYTES = (BM + (PAIR ? SBN / 2 : SBN)) * ROW_BYTES;
  constexpr int SMEM = STAGES * STAGE_BYTES + 256 + 8 * 4096 + 1024;
  static_assert((2 * STAGES + 2 * NBUF + 1) * 8 + 8 <= 256, "barrier block");
  static_assert(SMEM <= 232448, "shared memory budget");
  auto kern = slice_gemm_kernel<STAGES, PAIR>;
  static const bool attr = [&] {
    CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
    return true;
  }();
  (void)attr;
  a.mA = make_map(A.planes, NS * A.plane_rows, A.Kp, BM, 2);
  a.mB = make_map(B.planes, NS * B.plane_rows, B.Kp, PAIR ? SBN / 2 : SBN, 2);
  if constexpr (!PAIR) {
    kern<<<static_cast<unsigned>(std::min(units, sms)), SLICE_THREADS, SMEM, st>>>(a);
  } else {
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(SLICE_THREADS);
    cfg.dynamicSmemBytes = SMEM;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    static const int max_clusters = [&] {
      int mc = 0;
      cfg.gridDim = dim3(static_cast<unsigned>(2 * (sms / 2)));
      CUDA_CHECK(cudaOccupancyMaxActiveClusters(&mc, kern, &cfg));
      if (mc < 1) fail(CC_ERR_UNSUPPORTED, "gemm_slices: no resident CTA pair");
      return mc;
    }();
    cfg.gridDim = dim3(static_cast<unsigned>(2 * std::min(units, max_clusters)));
    CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, a));
  }
  LAUNCH_CHECK();
  count_launch();
}

// Work of one launch in tile-K-blocks per resident unit (28 digit products of
// a K block), the epilogue counted as 3 K blocks: what a split is chosen by.
double makespan(long tiles, long nkb, long split, long P) {
  const long per = (nkb + split - 1) / split;
  return static_cast<double>((tiles * ((nkb + per - 1) / per) + P - 1) / P) * (static_cast<double>(per) + 3.0);
}

SideArgs side(const SliceOperand &x, const SlicePlanes &p, bool expand) {
  SideArgs s;
  s.src = x.src;
  s.rt = x.rt;
  s.kt = x.kt;
  s.ld = x.ld;
  s.rows = x.rows;
  s.conj = x.conj;
  s.rows_unit = x.rows_unit;
  s.expand = expand;
  s.planes = static_cast<__half *>(p.planes);
  s.e = p.e;
  s.n2 = p.n2;
  return s;
}

}  // namespace

long slice_kp(long K) { return (2 * K + 63) / 64 * 64; }

namespace {
// [exponents, flag, norms, padded to 256 B][NS planes]
size_t slice_head(long rows) { return (sizeof(int) * (2 * rows + 1) + 255) / 256 * 256; }
}  // namespace

size_t slice_bytes(bool a_side, long rows, long K) {
  return slice_head(rows) + sizeof(__half) * NS * (a_side ? 2 : 1) * rows * slice_kp(K);
}

SlicePlanes slice_planes(void *mem, bool a_side, long rows, long K) {
  SlicePlanes p;
  p.e = static_cast<int *>(mem);
  p.n2 = reinterpret_cast<float *>(p.e + rows + 1);
  p.planes = static_cast<char *>(mem) + slice_head(rows);
  p.rows = rows;
  p.plane_rows = (a_side ? 2 : 1) * rows;
  p.Kp = slice_kp(K);
  return p;
}

void slice_pack(const SliceOperand *A, const SlicePlanes *pa, const SliceOperand *B,
                const SlicePlanes *pb, long K, cudaStream_t st, int num_sms) {
  SideArgs a = {}, b = {};
  long exp_a = 0, exp_b = 0, tiles_a = 0, tiles_b = 0, Kp = 0;
  auto setup = [&](const SliceOperand &x, const SlicePlanes &p, bool expand, SideArgs &s, long &ne,
                   long &nt) {
    s = side(x, p, expand);
    ne = x.rows_unit ? (x.rows + 31) / 32 * ((K + 15) / 16) : x.rows * ((K + 255) / 256);
    nt = (x.rows + 31) / 32 * (p.Kp / 64);
    Kp = p.Kp;
    CUDA_CHECK(cudaMemsetAsync(p.e, 0, sizeof(int) * (2 * x.rows + 1), st));
  };
  if (A) setup(*A, *pa, true, a, exp_a, tiles_a);
  if (B) setup(*B, *pb, false, b, exp_b, tiles_b);
  const long ne = exp_a + exp_b, nt = tiles_a + tiles_b;
  if (nt == 0) return;
  slice_exp_kernel<<<static_cast<unsigned>(std::min<long>((ne + 7) / 8, 8L * num_sms)), 256, 0, st>>>(
      a, b, K, exp_a, ne);
  LAUNCH_CHECK();
  slice_pack_kernel<<<static_cast<unsigned>(std::min<long>(nt, 32L * num_sms)), 256, 0, st>>>(
      a, b, K, Kp, tiles_a, nt);
  LAUNCH_CHECK();
  count_launch(2);
}

void gemm_slices(const SliceGemm &g, cudaStream_t st, int *err, int num_sms) {
  if (g.M <= 0 || g.N <= 0) return;
  const SlicePlanes &A = g.A, &B = g.B;
  if (A.Kp != B.Kp || NS * A.plane_rows > 0x7fffffffL || NS * B.plane_rows > 0x7fffffffL)
    fail(CC_ERR_ARG, "gemm_slices: operand planes");
  SliceArgs a = {};
  a.M = g.M;
  a.N = g.N;
  a.rows_a = A.plane_rows;
  a.rows_b = B.plane_rows;
  a.a_row0 = 2 * g.a_row0;
  a.b_row0 = g.b_row0;
  a.ea = A.e;
  a.eb = B.e;
  a.fa = A.e + A.rows;
  a.fb = B.e + B.rows;
  a.na = A.n2;
  a.nb = B.n2;
  a.C = g.C;
  a.cm = g.cm;
  a.cn = g.cn;
  a.ldc = g.ldc;
  a.alpha = g.alpha;
  a.beta = g.beta;
  int ex = 0;
  if (g.alpha.y == 0.0 && std::fabs(std::frexp(g.alpha.x, &ex)) == 0.5) {
    a.alpha_p2 = 1;
    a.alpha_e = ex - 1;
    a.alpha_neg = g.alpha.x < 0;
  }
  a.num_kb = static_cast<int>(A.Kp / 64);
  a.err = err;
  a.wait_ns = tc_wait_limit();
  // CTA pairs when they leave no more work to the slowest SM than single CTAs
  // (whose 128-row tiles pad less but stream a third more per product)
  const long nt = (g.N + SBN - 1) / SBN;
  const long t1 = (2 * g.M + BM - 1) / BM * nt, t2 = (2 * g.M + 2 * BM - 1) / (2 * BM) * nt;
  auto best_split = [&](long tiles, long P, double &cost) {
    long sp = 1;
    cost = makespan(tiles, a.num_kb, 1, P);
    if (tiles < 2 * P)
      for (long s = 2; s <= std::min<long>(a.num_kb, 64); ++s) {
        // a split adds its partial sums to the output in FP64: one more K
        // block's worth of epilogue
        const double c = makespan(tiles, a.num_kb, s, P) + 1.0;
        if (c < 0.95 * cost) {
          cost = c;
          sp = s;
        }
      }
    return sp;
  };
  double c1, c2;
  const long s1 = best_split(t1, num_sms, c1), s2 = best_split(t2, num_sms / 2, c2);
  const bool pair = c2 <= 1.05 * c1;
  const long split = pair ? s2 : s1;
  a.kb_per_split = static_cast<int>((a.num_kb + split - 1) / split);
  a.k_splits = (a.num_kb + a.kb_per_split - 1) / a.kb_per_split;
  a.n_tiles = static_cast<int>(nt);
  a.m_tiles = static_cast<int>((2 * g.M + (pair ? 2 * BM : BM) - 1) / (pair ? 2 * BM : BM));
  const double square = std::sqrt(static_cast<double>(pair ? num_sms / 2 : num_sms) * SBN / (pair ? 2 * BM : BM));
  a.group_m = std::max(1, std::min(a.m_tiles, static_cast<int>(square)));
  const long units = static_cast<long>(a.m_tiles) * a.n_tiles * a.k_splits;
  if (units > 0x7fffffffL) fail(CC_ERR_ARG, "gemm_slices: too many tiles");
  a.wmode = (g.beta.x == 0.0 && g.beta.y == 0.0) ? SW_STORE
            : (g.beta.x == 1.0 && g.beta.y == 0.0) ? SW_ADD
                                                   : SW_BETA;
  cplx guard_beta = g.beta;
  if (a.k_splits > 1) {
    scale_2d(g.C, g.cm, g.cn, g.ldc, g.M, g.N, g.beta, st);
    a.wmode = SW_ADD;
    guard_beta = make_double2(1.0, 0.0);
  }
  const int u = static_cast<int>(units);
  if (pair) launch_slices<8, true>(a, A, B, u, num_sms, st);
  else launch_slices<6, false>(a, A, B, u, num_sms, st);
  // Inf or NaN in an operand: the FP64 kernel computes this product instead
  GemmDesc f = g.src;
  f.M = g.M;
  f.N = g.N;
  f.C = g.C;
  f.cm = g.cm;
  f.cn = g.cn;
  f.ldc = g.ldc;
  f.alpha = g.alpha;
  f.beta = guard_beta;
  gemm_f64_if(f, a.fa, a.fb, st);
}

// Estimated times (s) of an M x N x K product here and on the FP64 pipe. The
// tensor side: 28 digit products of every 128 x 128 x 64 block at about 1
// PF/s, an epilogue of three K blocks per tile, the planes written and read,
// five launches. The FP64 side: 1 TF/s or its operands at 5 TB/s, on whole
// 64 x 64 tiles where the tiled kernel takes the product (a tile's rows cost
// the same empty: 5 x 64000 x 160 took 4.5 ms there).
bool slices_pay(long M, long N, long K) {
  const double m = (2 * M + 127) / 128 * 128.0, n = (N + 127) / 128 * 128.0;
  const double kb = static_cast<double>((2 * K + 63) / 64);
  const double mma = 2.0 * m * n * 64.0 * 28.0 * (kb + 3.0) / 1e15;
  const double pack = (static_cast<double>(M) * K * (32 + 112) + static_cast<double>(N) * K * (32 + 56)) / 5e12;
  const double out = 32.0 * M * N / 5e12;
  const double t_slices = 20e-6 + std::max(mma, 20e-6) + pack + out;
  const long tm = (M + 63) / 64, tn = (N + 63) / 64;
  const bool skinny = K <= SKINNY64_MAX_K && std::min(M, N) <= 256 && std::max(M, N) >= 1024;
  const bool tiled = M > 1 && N > 1 && !skinny && tm * tn >= 152;
  const double mn = tiled ? 4096.0 * tm * tn : static_cast<double>(M) * N;
  const double t_f64 = 4e-6 + std::max(8.0 * mn * K / 1e12, 16.0 * (static_cast<double>(M) * K + static_cast<double>(N) * K) / 5e12);
  return t_slices < 0.8 * t_f64;
}

}  // namespace cdfns
