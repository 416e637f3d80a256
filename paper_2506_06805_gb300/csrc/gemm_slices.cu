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
// for g = 1 .. 7: 28 digit products. What is left out (groups 8 .. 13, the
// rounding to 63 bits) is at most 2^-60 2^(Ea + Eb) per real term, 2^-62.9
// sqrt(K) 2^(Ea + Eb) RMS over K complex ones. Each digit product is at most 2^16
// in magnitude, so 256 of them (four K blocks of 64) add up without any
// rounding in the FP32 accumulators of tcgen05.mma; the epilogue warps then
// move the sums out of TMEM: groups 7 and 6 into FP32 (whose rounding lies
// 2^-24 below 2^-45 of the result), groups 5 .. 1 into 64-bit integers. Those
// are exact while the rows' and columns' 2-norms (relative to 2^E, from the
// packing) bound the sum below 2^62; for the larger ones of long, even rows,
// group 5 joins the FP32 part. The sum may wrap on the way, only its value
// counts.
//
// Accuracy, RMS error over |a_m| |b_n| against twice the precision, here and
// from the FP64 kernel, normal operands: K = 160 5.7e-18 / 1.2e-17, K = 1200
// 2.4e-18 / 5.8e-18, K = 20000 0.9e-18 / 4.2e-18.
//
// The digits' error is relative to the rows' largest magnitudes, FP64's (2^-55
// to 2^-54 RMS) to S = sum_k |a_mk| |b_nk|, which is far smaller where large
// elements of A meet small ones of B (columns scaled one way in A and the
// other in B, sparse rows, small imaginary parts). So an eighth plane holds
// the rounded magnitudes, whose product, one more beside the 28, gives S of
// every real and imaginary part. Elements with 0 < S < t sqrt(K) 2^(Ea + Eb)
// are not stored but listed for slice_fix_kernel, which computes them on the
// FP64 pipe; so are the elements of rows with an Inf or NaN, which cannot be
// cut. (Where group 5 is in FP32, whose error grows by another 2^-63.8 K
// 2^(Ea + Eb), the line is the larger of 8 t sqrt(K) and t K / 2.) t is 2^-8.5,
// where the digits' error reaches 0.38 RMS and 1.4 at most in units of 2^-53 S,
// that of the FP64 tiles being 0.45 and 2.2, and 2^-7 (0.13) for the few
// outputs that the FP64 pipe would sum by warps. 2^-7 for all: an FP64 CCSD
// iteration at o = 40, v = 300, X = 1200 takes 3.3 s instead of 2.4.
//
// RMS error over S in units of 2^-53 at 1536 x 1000 x 1200, here / FP64 kernel:
// normal operands 0.024 / 0.47, columns scaled by 10^(+-2 k / K) 0.045 / 0.47,
// by 10^(+-4 k / K) and more, where every element is listed, 0.071 / 0.47.
// That product takes 0.59 ms with none listed, 15.3 with all; 14.7 on the FP64
// pipe alone. Ladder at o = 15, v = 131, X = 517 983 -> 21.7 ms, FP64 residual
// at o = 12, v = 72, X = 288 80.7 -> 5.4 ms.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace cdfns {

namespace {

constexpr int NS = SLICE_COUNT;  // digits per element; plane NS holds the magnitudes
constexpr int PATCH_M = 16, PATCH_N = 32;  // complex elements of one epilogue warp
constexpr int SBN = 128;         // output columns per tile
constexpr int SKB = 2;           // K blocks of 64 per shared-memory slot and step
constexpr int CHUNK = 2;         // steps per TMEM accumulation (at most 256 terms)
constexpr int NBUF = 3;          // TMEM accumulators in flight (128 columns each)
constexpr int BAR_BYTES = 512;  // barriers
constexpr uint32_t STASH = NBUF * SBN;  // TMEM columns that hold the FP32 part

// 20 warps: 0-15 epilogue, 16 TMA producer of A, 17 MMA issuer, 18 TMA
// producer of B, 19 idle (it completes the warpgroup that gives registers
// away). Launched with 96 registers a thread (61440 in all); warps 16-19 drop
// to 48, the epilogue's 512 threads rise to 104: 512 x 104 + 128 x 48 = 59392.
constexpr int EPI_WARPS = 16;
constexpr int SLICE_THREADS = (EPI_WARPS + 4) * 32;

enum { SW_STORE = 0, SW_ADD = 1, SW_BETA = 2 };

// Elements that the digits are not accurate enough for, per K split: those of
// patches with few of them by themselves, from the front of the list, entry
// patch << 16 | element; other patches in units of FIX_UNIT elements, from its
// back, entry patch << 16 | unit, and as a mask with one bit per column.
constexpr int FIX_THREADS = 256, FIX_K = 32, FIX_CHUNK = 512;
constexpr int FIX_BLOCKS = 3;          // per SM
// (units of 64 read their operands more often, 16.9 ms against 15.3 where a
// product of 1536 x 1000 x 1200 is all units; 256 take 8 us longer where few
// SMs have one)
constexpr int FIX_UNIT = 128;
constexpr int FIX_FEW = 8;
struct FixList {
  int *queue;                // elements, units, next unit
  unsigned *mask;            // [patch][PATCH_M]
  unsigned long long *list;  // [patches * FIX_FEW]
  long patches;              // along m, n and the K splits
};

// a warp's entries: left = the bits of complex row lane / 2 of patch pt
__device__ __noinline__ void fix_push(const FixList &x, long pt, unsigned left) {
  const int lane = threadIdx.x & 31;
  const unsigned w = lane & 1 ? 0u : left;
  const int n = __reduce_add_sync(0xffffffffu, __popc(w));
  const unsigned long long id = static_cast<unsigned long long>(pt) << 16;
  if (n > FIX_FEW) {
    if ((lane & 1) == 0) x.mask[pt * PATCH_M + (lane >> 1)] = left;
    const int units = (n + FIX_UNIT - 1) / FIX_UNIT;
    if (lane == 0) {
      const int at = atomicAdd(&x.queue[1], units);
      for (int u = 0; u < units; ++u) x.list[x.patches * FIX_FEW - 1 - at - u] = id | u;
    }
    return;
  }
  int at = 0;
  if (lane == 0) at = atomicAdd(&x.queue[0], n);
  at = __shfl_sync(0xffffffffu, at, 0);
  for (int l = 0; l < 32; l += 2) {
    const int c = __popc(__shfl_sync(0xffffffffu, w, l));
    if (l < lane) at += c;
  }
  for (unsigned b = w; b; b &= b - 1) x.list[at++] = id | ((lane >> 1) * PATCH_N + __ffs(b) - 1);
}

struct alignas(64) SliceArgs {
  CUtensorMap mA, mB;  // [slice][row][Kp] planes as one matrix of slice * rows rows
  long M, N, K;        // complex rows, columns, terms of this product
  long rows_a, rows_b; // plane rows per slice
  long a_row0, b_row0; // first plane row of this product
  const int *ea, *eb;  // per complex row: biased exponent of the largest magnitude
  const float *na, *nb;  // per complex row: squared 2-norm over 4^E
  FixList fix;           // elements left to slice_fix_kernel
  float least;           // S / sqrt(K) they lie below (over 2^(Ea + Eb))
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

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4]) {
  uint32_t r[4];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
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

__device__ __noinline__ double scale_slow(double d, int e) { return scalbn(d, e); }

// d 2^e; the exponent field is adjusted in place unless the value or the
// result is not a normal number
__device__ __forceinline__ double scale_exp(double d, int e) {
  const int hi = __double2hiint(d);
  const int ex = (hi >> 20) & 0x7ff;
  const int ne = ex + e;
  if (ex != 0 && ne > 0 && ne < 2047)
    return __hiloint2double(hi + (e << 20), __double2loint(d));
  return scale_slow(d, e);
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

// The order of the digit products, shared by the three roles, after that of
// the magnitudes (one accumulation over all K blocks). Groups go in
// pairs (G, G - 1) for G = 7, 5, 3, 1, and within a K block the 2 G - 1
// products of such a pair zigzag through the digits,
//   (A_1, B_G), (A_1, B_G-1), (A_2, B_G-1), (A_2, B_G-2), ..., (A_G, B_1):
// even steps belong to group G, odd ones to G - 1, and each step brings in
// one new digit plane block, A on even steps, B on odd ones. A group's
// products collect in a TMEM buffer of its own, CHUNK of them at a time. A
// "K block" of this order is SKB blocks of 64 (one at the end of an odd
// range).
struct BufQueue {  // free TMEM buffers in the order they were handed over
  uint32_t q = 0u | (1u << 2) | (2u << 4);
  int n = NBUF;
  __device__ __forceinline__ int pop() {
    const int b = q & 3u;
    q >>= 2;
    --n;
    return b;
  }
  __device__ __forceinline__ void push(int b) { q |= static_cast<uint32_t>(b) << (2 * n++); }
};

// Persistent CTA or CTA pair, roles as in tc_gemm_kernel (gemm_tc.cu); every
// wait bounded. Tiles of UNIT_ROWS real rows x 128 columns: 64-bit sums for
// 256 columns would not fit the epilogue's registers. Such a tile needs 24 KB
// of operands per 256 clocks of MMA, about twice what L2 delivers; the
// zigzag uses every block of a plane twice and halves that. A step costs its
// single issuing threads a few hundred clocks of instructions and barrier
// round trips, so it spans two K blocks, 512 clocks of MMA. The epilogue
// (an integer conversion and a 64-bit add for every value of every chunk)
// needs four warps a scheduler to keep up. Kernel alone, 4096 x 4096 x K
// (group by group with eight epilogue warps -> this): K = 512 2.41 -> 1.58
// ms, K = 2048 6.46 -> 5.46 ms (5.54 with the magnitudes' product), 400 clocks
// a K block where the MMAs take 256.
template <int STAGES, bool PAIR>
__global__ void __launch_bounds__(SLICE_THREADS, 1) slice_gemm_kernel(const __grid_constant__ SliceArgs P) {
  constexpr int A_BLK = BM * ROW_BYTES;  // one K block
  constexpr int B_BLK = (PAIR ? SBN / 2 : SBN) * ROW_BYTES;
  constexpr int A_BYTES = SKB * A_BLK, B_BYTES = SKB * B_BLK;  // one slot
  constexpr int UNIT_ROWS = PAIR ? 2 * BM : BM;
  constexpr uint32_t IDESC = make_idesc(UNIT_ROWS, SBN, 0u);
  constexpr int COLS = SBN * 4 / EPI_WARPS;  // columns per epilogue warp
  static_assert(COLS == PATCH_N, "one mask bit per column");
  constexpr uint32_t TMEM_COLS = 512;

  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t *smem_b = smem + STAGES * A_BYTES;  // rings of A and of B blocks
  uint64_t *fullA = reinterpret_cast<uint64_t *>(smem + STAGES * (A_BYTES + B_BYTES));
  uint64_t *fullB = fullA + STAGES, *emptyA = fullB + STAGES, *emptyB = emptyA + STAGES;
  uint64_t *tfull = emptyB + STAGES;   // [NBUF]
  uint64_t *tempty = tfull + NBUF;     // [NBUF]
  uint64_t *mdone = tempty + NBUF;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mdone + 1);
  long long *stage = reinterpret_cast<long long *>(smem + STAGES * (A_BYTES + B_BYTES) + BAR_BYTES);  // 1.5 KB a warp

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int n_units = P.m_tiles * P.n_tiles * P.k_splits;
#define TC_RANK (PAIR ? static_cast<int>(cluster_rank()) : 0)
#define TC_UNIT0 (PAIR ? static_cast<int>(cluster_id_x()) : static_cast<int>(blockIdx.x))
#define TC_USTEP (PAIR ? static_cast<int>(cluster_count_x()) : static_cast<int>(gridDim.x))

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&fullA[s], 1);
      mbar_init(&fullB[s], 1);
      mbar_init(&emptyA[s], 1);
      mbar_init(&emptyB[s], 1);
    }
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], PAIR ? 2 * EPI_WARPS : EPI_WARPS);
    }
    mbar_init(mdone, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == EPI_WARPS + 1) tmem_alloc<PAIR>(tmem_slot, TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp >= EPI_WARPS) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 48;");
    if (warp == EPI_WARPS || warp == EPI_WARPS + 2) {
      if (lane == 0) {
        // ---------------- TMA producers of A and of B ----------------
        const bool is_a = warp == EPI_WARPS;
        uint64_t *const full = is_a ? fullA : fullB, *const empty = is_a ? emptyA : emptyB;
        uint8_t *const ring = is_a ? smem : smem_b;
        const CUtensorMap *const map = is_a ? &P.mA : &P.mB;
        const int blk = is_a ? A_BLK : B_BLK;
        const int rows = static_cast<int>(is_a ? P.rows_a : P.rows_b);
        long n = 0;  // slots filled
        int s = 0;
        uint32_t par = 1;  // parity of the wait for a free slot
        bool ok = true;
        for (int t = TC_UNIT0; t < n_units && ok; t += TC_USTEP) {
          int m_tile, n_tile, z;
          slice_coords(P, t, m_tile, n_tile, z);
          const int kb0 = z * P.kb_per_split;
          const int kb1 = min(P.num_kb, kb0 + P.kb_per_split);
          const int y = is_a ? static_cast<int>(P.a_row0) + m_tile * UNIT_ROWS + TC_RANK * BM
                             : static_cast<int>(P.b_row0) + n_tile * SBN + (PAIR ? TC_RANK * (SBN / 2) : 0);
          // (the magnitudes first, plane NS of both; then the digits)
          for (int G = NS + 2; G >= 1 && ok; G -= 2)
            for (int kb = kb0; kb < kb1 && ok; kb += SKB) {
              const int nb = min(SKB, kb1 - kb);
              const bool mag = G > NS;
              int yi = mag ? y + NS * rows : is_a ? y : y + (G - 1) * rows;  // A's digits ascend, B's descend
              for (int i = 0; i < (mag ? 1 : G); ++i, yi += is_a ? rows : -rows) {
                if (!mbar_wait(&empty[s], par, P.wait_ns)) {
                  atomicExch(P.err, 1);
                  ok = false;
                  break;
                }
                uint8_t *dst = ring + s * SKB * blk;
                if constexpr (PAIR) {
                  if (TC_RANK == 0) mbar_expect_tx(&full[s], 2 * nb * blk);
                  const uint32_t fb = leader_addr(smem_u32(&full[s]));
                  tma_load_2d_pair(dst, map, fb, kb * 64, yi);
                  if (nb == 2) tma_load_2d_pair(dst + blk, map, fb, kb * 64 + 64, yi);
                } else {
                  mbar_expect_tx(&full[s], nb * blk);
                  tma_load_2d(dst, map, &full[s], kb * 64, yi);
                  if (nb == 2) tma_load_2d(dst + blk, map, &full[s], kb * 64 + 64, yi);
                }
                ++n;
                if (++s == STAGES) {
                  s = 0;
                  par ^= 1u;
                }
              }
            }
        }
        // no copy may outlive the CTA's shared memory (see tc_gemm_kernel)
        if (TC_RANK == 0)
          for (long i = (n > STAGES ? n - STAGES : 0); i < n; ++i)
            if (!mbar_wait(&full[i % STAGES], static_cast<uint32_t>(i / STAGES) & 1u, DRAIN_NS))
              atomicExch(P.err, 1);
      }
    } else if (warp == EPI_WARPS + 1) {
      if (TC_RANK == 0 && elect_one()) {
        // ---------------- MMA issuer (the leader of a pair) ----------------
        BufQueue bq;
        uint32_t waits = 0, par = 0;  // per TMEM buffer: used before; parity of its next release
        int sa = STAGES - 1, sb = STAGES - 1;  // slots in use
        uint32_t pa = 1, pb = 1;               // parities of their fills
        bool ok = true;
        const uint64_t desc_a = sw128_desc(smem_u32(smem)), desc_b = sw128_desc(smem_u32(smem_b));
        auto next_a = [&] {
          if (++sa == STAGES) {
            sa = 0;
            pa ^= 1u;
          }
          return mbar_wait(&fullA[sa], pa, P.wait_ns);
        };
        auto next_b = [&] {
          if (++sb == STAGES) {
            sb = 0;
            pb ^= 1u;
          }
          return mbar_wait(&fullB[sb], pb, P.wait_ns);
        };
        // the product of the two current slots, collected in its group's buffer
        auto product = [&](int nb, int &cnt, int &buf) {
          if (cnt == 0) {
            buf = bq.pop();
            if ((waits >> buf) & 1u) {
              if (!mbar_wait(&tempty[buf], (par >> buf) & 1u, P.wait_ns)) return false;
              par ^= 1u << buf;
            }
            waits |= 1u << buf;
          }
          tc_fence_after();
          const uint64_t da = desc_a + static_cast<uint32_t>(sa * (A_BYTES >> 4));  // in 16 bytes
          const uint64_t db = desc_b + static_cast<uint32_t>(sb * (B_BYTES >> 4));
          const uint32_t dt = tmem + buf * SBN;
#pragma unroll
          for (int kk = 0; kk < ROW_BYTES / 32; ++kk)
            mma<true, PAIR>(dt, da + 2 * kk, db + 2 * kk, IDESC, (cnt > 0 || kk > 0) ? 1u : 0u);
          if (nb == 2) {
#pragma unroll
            for (int kk = 0; kk < ROW_BYTES / 32; ++kk)
              mma<true, PAIR>(dt, da + (A_BLK >> 4) + 2 * kk, db + (B_BLK >> 4) + 2 * kk, IDESC, 1u);
          }
          ++cnt;
          return true;
        };
        auto hand_over = [&](int &cnt, int buf) {
          mma_commit_both<PAIR>(&tfull[buf]);
          bq.push(buf);
          cnt = 0;
        };
        for (int t = TC_UNIT0; t < n_units && ok; t += TC_USTEP) {
          int m_tile, n_tile, z;
          slice_coords(P, t, m_tile, n_tile, z);
          const int kb0 = z * P.kb_per_split;
          const int nkb = min(P.num_kb, kb0 + P.kb_per_split) - kb0;
          int cntm = 0, bufm = 0;  // the magnitudes' product: one accumulation
          for (int kb = 0; kb < nkb && ok; kb += SKB) {
            if (!(ok = next_a() && next_b() && product(min(SKB, nkb - kb), cntm, bufm))) break;
            mma_commit_both<PAIR>(&emptyB[sb]);
            mma_commit_both<PAIR>(&emptyA[sa]);
          }
          if (ok) hand_over(cntm, bufm);
          for (int G = NS; G >= 1 && ok; G -= 2) {
            int cnt0 = 0, cnt1 = 0, buf0 = 0, buf1 = 0;  // groups G and G - 1
            for (int kb = 0; kb < nkb && ok; kb += SKB) {
              const int nb = min(SKB, nkb - kb);
              ok = next_a() && next_b();
              for (int i = 0; ok; ++i) {
                if (!(ok = product(nb, cnt0, buf0))) break;
                mma_commit_both<PAIR>(&emptyB[sb]);
                if (cnt0 == CHUNK) hand_over(cnt0, buf0);
                if (i == G - 1) {
                  mma_commit_both<PAIR>(&emptyA[sa]);
                  break;
                }
                if (!(ok = next_b() && product(nb, cnt1, buf1))) break;
                mma_commit_both<PAIR>(&emptyA[sa]);
                if (cnt1 == CHUNK) hand_over(cnt1, buf1);
                ok = next_a();
              }
            }
            if (ok && cnt0) hand_over(cnt0, buf0);
            if (ok && cnt1) hand_over(cnt1, buf1);
          }
        }
        if (!ok) atomicExch(P.err, 1);
        mma_commit_self<PAIR>(mdone);
        if (!mbar_wait(mdone, 0u, DRAIN_NS)) atomicExch(P.err, 1);
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 104;");
    // ---------------- epilogue ----------------
    const int q = warp & 3;
    const int h = warp >> 2;
    const uint32_t lanes = static_cast<uint32_t>(q * 32) << 16;
    BufQueue bq;
    uint32_t par = 0;  // per TMEM buffer: parity of its next filling
    bool ok = true;
    // one chunk: wait for it, hand 16 columns at a time to f(column, values), free it
    auto drain = [&](int buf, auto &&f) {
      if (!mbar_wait(&tfull[buf], (par >> buf) & 1u, P.wait_ns)) {
        ok = false;
        return;
      }
      par ^= 1u << buf;
      tc_fence_after();
      const uint32_t base = tmem + lanes + buf * SBN + h * COLS;
#pragma unroll
      for (int j = 0; j < COLS; j += 16) {
        float v[16];
        tmem_ld16(base + j, v);
        f(j, v);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR)
          mbar_arrive_cluster(leader_addr(smem_u32(&tempty[buf])));
        else
          mbar_arrive(&tempty[buf]);
      }
    };
    // the chunks of groups (G, G - 1) in the issuer's order, each given to f
    // (one place: the epilogue's unrolled code has to stay in the
    // instruction cache)
    auto chunks = [&](int G, int nkb, auto &&f) {
      int cnt0 = 0, cnt1 = 0, buf0 = 0, buf1 = 0, p = 0, left = (nkb + SKB - 1) / SKB * (2 * G - 1);
      while (ok) {
        int buf = -1, g = G;
        for (; left > 0 && buf < 0; --left) {
          if ((p & 1) == 0) {
            if (cnt0 == 0) buf0 = bq.pop();
            if (++cnt0 == CHUNK) {
              buf = buf0;
              cnt0 = 0;
            }
          } else {
            if (cnt1 == 0) buf1 = bq.pop();
            if (++cnt1 == CHUNK) {
              buf = buf1;
              g = G - 1;
              cnt1 = 0;
            }
          }
          if (++p == 2 * G - 1) p = 0;
        }
        if (buf < 0) {  // the incomplete chunks at the end
          if (cnt0) {
            buf = buf0;
            cnt0 = 0;
          } else if (cnt1) {
            buf = buf1;
            g = G - 1;
            cnt1 = 0;
          } else {
            break;
          }
        }
        f(buf, g);
        bq.push(buf);
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
      const long nbase = static_cast<long>(n_tile) * SBN + h * COLS;
      const long mbase = (static_cast<long>(m_tile) * UNIT_ROWS + TC_RANK * BM) / 2 + q * 16;
      const long mrow = mbase + (lane >> 1);
      // the integers count 2^u last places of group 5, with |a| |b| 2^(52 - u)
      // below 2^62 (u = 5 would make group 1's factor 2^31)
      int u;
      {
        const float na = mrow < P.M ? P.na[P.a_row0 / 2 + mrow] : 0.f;
        const float nb = nbase + lane < P.N ? P.nb[P.b_row0 + nbase + lane] : 0.f;
        const float a = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(na)));
        const float b = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(nb)));
        const int e = static_cast<int>(__float_as_uint(a * b) >> 23) - 126;  // a b < 2^e
        u = max(0, (e - 18) / 2);
        if (u == 5) u = 6;
      }
      // Elements whose S = sum_k |a||b| (the magnitudes' product, over 2^(Ea +
      // Eb - 30)) is too small against the rows' largest magnitudes for the
      // digits to be as accurate as FP64, and those of rows or columns with an
      // Inf or NaN (exponent field 2047): one bit per column in this lane's
      // mask, left to slice_fix_kernel. S = 0 has no nonzero term: 0 exactly.
      unsigned left;
      {
        // (sqrt(K); a shorter last split may have that much less: the others
        // make up for it)
        const float full = static_cast<float>(min(P.K, 32L * P.kb_per_split));
        const float rk = static_cast<float>(min(P.K - 32L * kb0, 32L * nkb)) * rsqrtf(full);
        const float thr = 0x1p30f * rk * P.least * (u ? fmaxf(8.0f, 0.5f * rk) : 1.0f);
        left = 0;
        const int buf = bq.pop();
        drain(buf, [&](int j, const float (&x)[16]) {
#pragma unroll
          for (int k = 0; k < 16; ++k) left |= (x[k] > 0.f && x[k] < thr) ? 1u << (j + k) : 0u;
        });
        bq.push(buf);
        if (!ok) break;
        const bool col = nbase + lane < P.N;
        const unsigned cols = __ballot_sync(0xffffffffu, col);
        left |= __ballot_sync(0xffffffffu, col && P.eb[P.b_row0 + nbase + lane] == 2047);
        if (mrow >= P.M) left = 0;
        else if (P.ea[P.a_row0 / 2 + mrow] == 2047) left = ~0u;
        left &= cols;
        left |= __shfl_xor_sync(0xffffffffu, left, 1);
        const long pt = (static_cast<long>(z) * P.m_tiles * (UNIT_ROWS / 2 / PATCH_M) + mbase / PATCH_M) *
                            P.n_tiles * (SBN / PATCH_N) + nbase / PATCH_N;
        if (__any_sync(0xffffffffu, left != 0)) fix_push(P.fix, pt, left);
      }
      {
        float lf[COLS];
#pragma unroll
        for (int j = 0; j < COLS; ++j) lf[j] = 0.f;
        chunks(NS, nkb, [&](int buf, int g) {
          const float w = g == NS ? 0x1p-9f : 1.0f;
          drain(buf, [&](int j, const float (&x)[16]) {
#pragma unroll
            for (int k = 0; k < 16; ++k) lf[j + k] = fmaf(w, x[k], lf[j + k]);
          });
        });
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < COLS; j += 16) tmem_st16(tmem + lanes + STASH + h * COLS + j, lf + j);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      }
      long long acc[COLS], bias = 0;
#pragma unroll
      for (int j = 0; j < COLS; ++j) acc[j] = 0;
      // A sum x below 2^22 becomes the integer MAGIC + x in the bits of
      // x + 1.5 2^23 (the hardware conversion gives 16 values per clock and
      // SM, a quarter of what the chunks need); larger ones, which a few
      // hundred random digits do not reach, are converted. MAGIC times the
      // factor is taken off once per tile.
      constexpr int MAGIC = 0x4b400000;
      for (int G = NS - 2; G >= 1; G -= 2)
        chunks(G, nkb, [&](int buf, int g) {
          const int sh = 9 * (5 - g) - u;
          const int mul = 1 << min(max(sh, 0), 30);
          const int up = sh - 32;
          const bool fp = sh < 0;  // group 5 of a long, even row: to the FP32 part
          if (!fp) bias += static_cast<long long>(static_cast<unsigned long long>(MAGIC) << max(sh, 0));
          drain(buf, [&](int j, const float (&x)[16]) {
            if (fp) {
              float lf[16];
              const uint32_t at = tmem + lanes + STASH + h * COLS + j;
              tmem_ld16(at, lf);
#pragma unroll
              for (int k = 0; k < 16; ++k) lf[k] = fmaf(512.0f, x[k], lf[k]);
              tmem_st16(at, lf);
              asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
              return;
            }
            float m = 0.f;
#pragma unroll
            for (int k = 0; k < 16; ++k) m = fmaxf(m, fabsf(x[k]));
            int xi[16];
            if (!__any_sync(0xffffffffu, m >= 0x1p22f)) {
#pragma unroll
              for (int k = 0; k < 16; ++k) xi[k] = __float_as_int(x[k] + 12582912.0f);
            } else {
#pragma unroll
              for (int k = 0; k < 16; ++k) xi[k] = MAGIC + __float2int_rn(x[k]);
            }
            if (up < 0) {
#pragma unroll
              for (int k = 0; k < 16; ++k)
                asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(acc[j + k]) : "r"(xi[k]), "r"(mul));
            } else {
#pragma unroll
              for (int k = 0; k < 16; ++k)
                acc[j + k] += static_cast<long long>(static_cast<unsigned long long>(static_cast<unsigned>(xi[k]) << up) << 32);
            }
          });
        });
      if (!ok) break;
      // value = (2^(9 + u) acc + lf) 2^(Ea + Eb - 16 - 45), four columns at a
      // time through shared memory: lane = real row on the way in, (row of
      // eight, column) of complex results on the way out. The conversion
      // sits on the way out, in a loop: unrolled over the accumulators it was
      // far larger than the instruction cache (110 000 clocks a tile).
      const int ea = (mrow < P.M ? P.ea[P.a_row0 / 2 + mrow] : 1) - 2 * 1022 - 61 + (P.alpha_p2 ? P.alpha_e : 0);
      const int ebl = nbase + lane < P.N ? P.eb[P.b_row0 + nbase + lane] : 1;
      long roff = 0;
      if (lane < 16 && mbase + lane < P.M)
        roff = P.cm ? P.cm[mbase + lane] : (mbase + lane) * P.ldc;
      long long *sacc = stage + warp * 192;  // [32][4] integers, then [32][4] floats
      float *slf = reinterpret_cast<float *>(sacc + 128);
      const int col = lane & 3, hf = lane >> 2;
#pragma unroll 1
      for (int seg = 0; seg < COLS / 4; ++seg) {
        float lf[4];
        tmem_ld4(tmem + lanes + STASH + h * COLS + 4 * seg, lf);
#pragma unroll
        for (int k = 0; k < 4; ++k) slf[lane * 4 + (k ^ ((lane >> 1) & 3))] = lf[k];
#pragma unroll
        for (int j = 0; j < COLS; j += 4)
          if (j == 4 * seg) {
#pragma unroll
            for (int k = 0; k < 4; ++k) sacc[lane * 4 + (k ^ ((lane >> 1) & 3))] = acc[j + k];
          }
        __syncwarp();
        const int c = 4 * seg + col;
        const int eb = __shfl_sync(0xffffffffu, ebl, c);
        const long n = nbase + c;
        const bool col_ok = n < P.N;
        const long cno = col_ok ? (P.cn ? P.cn[n] : n) : 0;
#pragma unroll 1
        for (int rr = 0; rr < 2; ++rr) {
          const int r = 8 * rr + hf;
          const long ro = __shfl_sync(0xffffffffu, roff, r);
          const int e = __shfl_sync(0xffffffffu, ea, 2 * r) + eb;
          const unsigned skip = __shfl_sync(0xffffffffu, left, 2 * r);
          double v[2];
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const int at = (2 * r + w) * 4 + (col ^ (r & 3));
            const long long x = sacc[at] - bias;
            double d = f32_to_f64(slf[at]);
            if (x != 0) d += scale_exp(i64_to_f64(x), 9 + u);
            v[w] = scale_exp(d, e);
            if (P.alpha_neg) v[w] = __hiloint2double(__double2hiint(v[w]) ^ 0x80000000, __double2loint(v[w]));
          }
          if (!col_ok || mbase + r >= P.M || ((skip >> c) & 1u)) continue;
          double2 *o = P.C + ro + cno;
          double2 y = make_double2(v[0], v[1]);
          if (!P.alpha_p2) y = cmul(P.alpha, y);
          if (P.wmode == SW_ADD) {
            atomicAdd(&o->x, y.x);
            atomicAdd(&o->y, y.y);
          } else if (P.wmode == SW_STORE) {
            *o = y;
          } else {
            *o = cadd(y, cmul(P.beta, *o));
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
  if (warp == EPI_WARPS + 1) {
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
  int *e;     // [rows] exponent fields
  float *n2;  // [rows] squared 2-norms over 4^E
};

__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// e[row] = the largest exponent field of the row's components (at least 1;
// 2047: an Inf or NaN). One warp per item: 32 rows x 16 k with lanes
// along the rows where those are neighbours in memory, else one row x 256 k
// with lanes along k, 8 loads in flight: on small operands the time is one
// item's latency (items four times as long took 36 us at any size), on
// large ones the read of the operand.
__global__ void __launch_bounds__(256) slice_exp_kernel(SideArgs a, SideArgs b, long K, long items_a,
                                                        long items, int *reset) {
  if (reset && blockIdx.x == 0 && threadIdx.x < SLICE_RESET_BYTES / sizeof(int)) reset[threadIdx.x] = 0;
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
      if (lane == 0) atomicMax(&s.e[r], m);
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

// one complex element's digits and magnitudes into its place of every plane;
// the lanes of a warp hold 32 neighbouring k of one row
__device__ __forceinline__ void store_digits(const SideArgs &s, long r, long kc, long Kp, double2 x,
                                             int field) {
  const bool nr = (__double_as_longlong(x.x) << 1) != 0, ni = (__double_as_longlong(x.y) << 1) != 0;
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
  {
    // magnitudes over 2^(E - 15); nonzero ones stay normal halves (2^-14)
    const __half2 mg = __floats2half2_rn(fmaxf(fabsf(fr) * 32768.f, nr ? 0x1p-14f : 0.f),
                                         fmaxf(fabsf(fi) * 32768.f, ni ? 0x1p-14f : 0.f));
    const long o = (NS * prows + prow) * hk + kc;
    pl[o] = mg;
    if (s.expand) pl[o + hk] = __lowhigh2highlow(mg);
  }
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
// the rows) and written along k. HBM bound: 16 B read, 32 B (64 B for the
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

// ---------------------------------------------------------------------------
// elements the digits are not accurate enough for, on the FP64 pipe
// ---------------------------------------------------------------------------
struct FixSide {
  const double2 *p;
  const long *rt, *kt;
  long ld;
  bool conj, rows_unit;
};
struct FixArgs {
  long M, N, K, k_per_split;
  long pm, pn;  // patches along m and along n
  FixList fix;
  const int *err;
  FixSide A, B;
  double2 *C;
  const long *cm, *cn;
  long ldc;
  double2 alpha, beta;
  int wmode;
};
// ROWS rows x FIX_K of an operand on their way into shared memory [k][row],
// read along whichever of the two is contiguous. Rows and k beyond the end
// read the last valid ones, so that a thread's loads are in flight together
// (tested one by one they ran one after another, 9 us a tile); k beyond the
// end count as zero, rows beyond it are not used.
template <int ROWS>
struct FixTile {
  static constexpr int N = ROWS * FIX_K / FIX_THREADS;
  long ro[N];
  double2 x[N];
  __device__ __forceinline__ int row(const FixSide &s, int i) const {
    const int t = threadIdx.x + FIX_THREADS * i;
    return s.rows_unit ? t % ROWS : t / FIX_K;
  }
  __device__ __forceinline__ int col(const FixSide &s, int i) const {
    const int t = threadIdx.x + FIX_THREADS * i;
    return s.rows_unit ? t / ROWS : t % FIX_K;
  }
  __device__ __forceinline__ void rows(const FixSide &s, long r0, long rows) {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const long r = min(r0 + row(s, i), rows - 1);
      ro[i] = s.rt ? s.rt[r] : r * s.ld;
    }
  }
  __device__ __forceinline__ void load(const FixSide &s, long k0, long k1) {
    long ko[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const long k = min(k0 + col(s, i), k1 - 1);
      ko[i] = s.kt ? s.kt[k] : k;
    }
#pragma unroll
    for (int i = 0; i < N; ++i) x[i] = s.p[ro[i] + ko[i]];
  }
  __device__ __forceinline__ void store(const FixSide &s, long k0, long k1, double2 (&to)[FIX_K][ROWS + 1]) const {
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int c = col(s, i);
      double2 y = x[i];
      if (s.conj) y.y = -y.y;
      to[c][row(s, i)] = k0 + c < k1 ? y : make_double2(0.0, 0.0);
    }
  }
};

struct FixPatch {
  long z, m0, n0, k0, k1;  // split, first row and column, K range
  unsigned cols;           // columns within the product
};
__device__ __forceinline__ FixPatch fix_patch(const FixArgs &P, long pt) {
  FixPatch q;
  q.z = pt / (P.pm * P.pn);
  const long mn = pt - q.z * (P.pm * P.pn);
  q.m0 = mn / P.pn * PATCH_M;
  q.n0 = mn % P.pn * PATCH_N;
  q.k0 = q.z * P.k_per_split;
  q.k1 = min(P.K, q.k0 + P.k_per_split);
  q.cols = q.n0 + PATCH_N <= P.N ? ~0u : q.n0 < P.N ? (1u << (P.N - q.n0)) - 1u : 0u;
  return q;
}
__device__ __forceinline__ unsigned fix_mask(const FixArgs &P, const FixPatch &q, long pt, int r) {
  return q.m0 + r < P.M ? P.fix.mask[pt * PATCH_M + r] & q.cols : 0u;
}

__device__ __forceinline__ void fix_store(const FixArgs &P, long m, long n, double2 x) {
  double2 *o = P.C + (P.cm ? P.cm[m] : m * P.ldc) + (P.cn ? P.cn[n] : n);
  const double2 y = cmul(P.alpha, x);
  if (P.wmode == SW_ADD) {
    atomicAdd(&o->x, y.x);
    atomicAdd(&o->y, y.y);
  } else {
    *o = P.wmode == SW_STORE ? y : cadd(y, cmul(P.beta, *o));
  }
}

// one element by a warp, the lanes striding k
__device__ __forceinline__ void fix_element(const FixArgs &P, const FixPatch &q, int r, int c) {
  const long m = q.m0 + r, n = q.n0 + c;
  const double2 *pa = P.A.p + (P.A.rt ? P.A.rt[m] : m * P.A.ld);
  const double2 *pb = P.B.p + (P.B.rt ? P.B.rt[n] : n * P.B.ld);
  double2 s = make_double2(0.0, 0.0);
  for (long k = q.k0 + (threadIdx.x & 31); k < q.k1; k += 128) {
    double2 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const long kk = min(k + 32 * u, q.k1 - 1);
      a[u] = pa[P.A.kt ? P.A.kt[kk] : kk];
      b[u] = pb[P.B.kt ? P.B.kt[kk] : kk];
    }
    double2 x = make_double2(0.0, 0.0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (P.A.conj) a[u].y = -a[u].y;
      if (P.B.conj) b[u].y = -b[u].y;
      if (k + 32 * u < q.k1) x = cfma(a[u], b[u], x);
    }
    s = cadd(s, x);
  }
  for (int o = 16; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  if ((threadIdx.x & 31) == 0) fix_store(P, m, n, s);
}

// The elements slice_gemm_kernel has listed, over the K range of their split.
// Single ones (the usual case: near zeros of structured operands): a warp
// each. A unit of a patch with more: a block, its operands through shared
// memory; blocks draw the units from a queue. Sums run over 8 terms and over
// 512 / 8 such runs at a time, as short as those of the FP64 kernels' warps.
__global__ void __launch_bounds__(FIX_THREADS, FIX_BLOCKS) slice_fix_kernel(const FixArgs P) {
  __shared__ double2 As[FIX_K][PATCH_M + 1], Bs[FIX_K][PATCH_N + 1];
  __shared__ unsigned short el[FIX_UNIT];
  __shared__ int unit;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int n_el = P.fix.queue[0], n_units = P.fix.queue[1];
  if (*P.err) return;  // a wait has expired
  for (long f = blockIdx.x * (FIX_THREADS / 32L) + warp; f < n_el; f += gridDim.x * (FIX_THREADS / 32L)) {
    const unsigned long long e = P.fix.list[f];
    const int c = e & 0xffffu;
    fix_element(P, fix_patch(P, static_cast<long>(e >> 16)), c / PATCH_N, c % PATCH_N);
  }
  if (n_units) {
    for (;;) {
      if (t == 0) unit = atomicAdd(&P.fix.queue[2], 1);
      __syncthreads();
      if (unit >= n_units) break;
      const unsigned long long id = P.fix.list[P.fix.patches * FIX_FEW - 1 - unit];
      const long pt = static_cast<long>(id >> 16);
      const FixPatch q = fix_patch(P, pt);
      const int first = static_cast<int>(id & 0xffffu) * FIX_UNIT;
      int n = 0;
      for (int r = 0; r < PATCH_M; ++r) {
        const unsigned w = fix_mask(P, q, pt, r);
        const int at = n + __popc(w & ((1u << lane) - 1u)) - first;
        if (warp == 0 && ((w >> lane) & 1u) && at >= 0 && at < FIX_UNIT)
          el[at] = static_cast<unsigned short>(r * PATCH_N + lane);
        n += __popc(w);
      }
      __syncthreads();
      // two or four threads an element, each every second or fourth k
      const int m = min(n - first, FIX_UNIT), sl = m > FIX_THREADS / 4 ? 1 : 2, sp = 1 << sl;
      const int sub = t & (sp - 1);
      const bool on = (t >> sl) < m;
      const int e = on ? el[t >> sl] : 0, r = e / PATCH_N, c = e % PATCH_N;
      double2 s = make_double2(0.0, 0.0);
      FixTile<PATCH_M> ta;
      FixTile<PATCH_N> tb;
      ta.rows(P.A, q.m0, P.M);
      tb.rows(P.B, q.n0, P.N);
      for (long kc = q.k0; kc < q.k1; kc += FIX_CHUNK) {
        const long ke = min(q.k1, kc + FIX_CHUNK);
        double2 y = make_double2(0.0, 0.0);
        for (long k = kc; k < ke; k += FIX_K) {
          ta.load(P.A, k, q.k1);
          tb.load(P.B, k, q.k1);
          ta.store(P.A, k, q.k1, As);
          tb.store(P.B, k, q.k1, Bs);
          __syncthreads();
          if (on) {
            const double2 *a = &As[sub][r], *b = &Bs[sub][c];
            for (int g = 0; g < FIX_K >> sl; g += 8) {
              double2 x = make_double2(0.0, 0.0);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                x = cfma(*a, *b, x);
                a += sp * (PATCH_M + 1);
                b += sp * (PATCH_N + 1);
              }
              y = cadd(y, x);
            }
          }
          __syncthreads();
        }
        s = cadd(s, y);
      }
      for (int o = sp / 2; o > 0; o >>= 1) {
        s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
        s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
      }
      if (on && sub == 0) fix_store(P, q.m0 + r, q.n0 + c, s);
    }
  }
}

template <int STAGES, bool PAIR>  // STAGES slots of SKB K blocks for each operand
void launch_slices(SliceArgs &a, const SlicePlanes &A, const SlicePlanes &B, int units, int sms,
                   cudaStream_t st) {
  constexpr int STAGE_BYTES = SKB * (BM + (PAIR ? SBN / 2 : SBN)) * ROW_BYTES;
  constexpr int SMEM = STAGES * STAGE_BYTES + BAR_BYTES + EPI_WARPS * 1536 + 1024;
  static_assert((4 * STAGES + 2 * NBUF + 1) * 8 + 8 <= BAR_BYTES, "barrier block");
  static_assert(SMEM <= 232448, "shared memory budget");
  auto kern = slice_gemm_kernel<STAGES, PAIR>;
  static const bool attr = [&] {
    CUDA_CHECK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM));
    return true;
  }();
  (void)attr;
  a.mA = make_map(A.planes, SLICE_PLANES * A.plane_rows, A.Kp, BM, 2);
  a.mB = make_map(B.planes, SLICE_PLANES * B.plane_rows, B.Kp, PAIR ? SBN / 2 : SBN, 2);
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

// Work of one launch in tile-K-blocks per resident unit (29 products of a K
// block), the epilogue counted as 3 K blocks: what a split is chosen by.
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
// [exponents, norms, padded to 256 B][planes]
size_t slice_head(long rows) { return (sizeof(int) * 2 * rows + 255) / 256 * 256; }
}  // namespace

size_t slice_bytes(bool a_side, long rows, long K) {
  return slice_head(rows) + sizeof(__half) * SLICE_PLANES * (a_side ? 2 : 1) * rows * slice_kp(K);
}

SlicePlanes slice_planes(void *mem, bool a_side, long rows, long K) {
  SlicePlanes p;
  p.e = static_cast<int *>(mem);
  p.n2 = reinterpret_cast<float *>(p.e + rows);
  p.planes = static_cast<char *>(mem) + slice_head(rows);
  p.rows = rows;
  p.plane_rows = (a_side ? 2 : 1) * rows;
  p.Kp = slice_kp(K);
  return p;
}

void slice_pack(const SliceOperand *A, const SlicePlanes *pa, const SliceOperand *B,
                const SlicePlanes *pb, long K, void *scratch, cudaStream_t st, int num_sms) {
  SideArgs a = {}, b = {};
  long exp_a = 0, exp_b = 0, tiles_a = 0, tiles_b = 0, Kp = 0;
  auto setup = [&](const SliceOperand &x, const SlicePlanes &p, bool expand, SideArgs &s, long &ne,
                   long &nt) {
    s = side(x, p, expand);
    ne = x.rows_unit ? (x.rows + 31) / 32 * ((K + 15) / 16) : x.rows * ((K + 255) / 256);
    nt = (x.rows + 31) / 32 * (p.Kp / 64);
    Kp = p.Kp;
    CUDA_CHECK(cudaMemsetAsync(p.e, 0, sizeof(int) * 2 * x.rows, st));
  };
  if (A) setup(*A, *pa, true, a, exp_a, tiles_a);
  if (B) setup(*B, *pb, false, b, exp_b, tiles_b);
  const long ne = exp_a + exp_b, nt = tiles_a + tiles_b;
  if (nt == 0) return;
  slice_exp_kernel<<<static_cast<unsigned>(std::min<long>((ne + 7) / 8, 8L * num_sms)), 256, 0, st>>>(
      a, b, K, exp_a, ne, static_cast<int *>(scratch));
  LAUNCH_CHECK();
  slice_pack_kernel<<<static_cast<unsigned>(std::min<long>(nt, 32L * num_sms)), 256, 0, st>>>(
      a, b, K, Kp, tiles_a, nt);
  LAUNCH_CHECK();
  count_launch(2);
}

namespace {
// Tiles and K split of an M x N product over num_kb blocks of 64
struct SlicePlan {
  bool pair;
  int kb_per_split, k_splits, m_tiles, n_tiles;
  long units() const { return static_cast<long>(m_tiles) * n_tiles * k_splits; }
  long patches_m() const { return static_cast<long>(m_tiles) * ((pair ? BM : BM / 2) / PATCH_M); }
  long patches_n() const { return static_cast<long>(n_tiles) * (SBN / PATCH_N); }
  long patches() const { return patches_m() * patches_n() * k_splits; }
};

SlicePlan slice_plan(long M, long N, long num_kb, int num_sms) {
  // CTA pairs when they leave no more work to the slowest SM than single CTAs
  // (whose 128-row tiles pad less but stream a third more per product)
  const long nt = (N + SBN - 1) / SBN;
  const long t1 = (2 * M + BM - 1) / BM * nt, t2 = (2 * M + 2 * BM - 1) / (2 * BM) * nt;
  auto best_split = [&](long tiles, long P, double &cost) {
    long sp = 1;
    cost = makespan(tiles, num_kb, 1, P);
    if (tiles < 2 * P)
      for (long s = 2; s <= std::min<long>(num_kb, 64); ++s) {
        // a split adds its partial sums to the output in FP64: one more K
        // block's worth of epilogue
        const double c = makespan(tiles, num_kb, s, P) + 1.0;
        if (c < 0.95 * cost) {
          cost = c;
          sp = s;
        }
      }
    return sp;
  };
  double c1, c2;
  const long s1 = best_split(t1, num_sms, c1), s2 = best_split(t2, num_sms / 2, c2);
  SlicePlan p;
  p.pair = c2 <= 1.05 * c1;
  const long split = p.pair ? s2 : s1;
  p.kb_per_split = static_cast<int>((num_kb + split - 1) / split);
  p.k_splits = static_cast<int>((num_kb + p.kb_per_split - 1) / p.kb_per_split);
  p.n_tiles = static_cast<int>(nt);
  p.m_tiles = static_cast<int>((2 * M + (p.pair ? 2 * BM : BM) - 1) / (p.pair ? 2 * BM : BM));
  return p;
}
}  // namespace

size_t slice_scratch_bytes(long M, long N, long K, int num_sms) {
  if (M <= 0 || N <= 0) return 0;
  return SLICE_RESET_BYTES + (sizeof(unsigned) * PATCH_M + sizeof(unsigned long long) * FIX_FEW) *
                                 slice_plan(M, N, slice_kp(K) / 64, num_sms).patches();
}

void gemm_slices(const SliceGemm &g, cudaStream_t st, int *err, int num_sms) {
  if (g.M <= 0 || g.N <= 0) return;
  const SlicePlanes &A = g.A, &B = g.B;
  if (A.Kp != B.Kp || SLICE_PLANES * A.plane_rows > 0x7fffffffL || SLICE_PLANES * B.plane_rows > 0x7fffffffL)
    fail(CC_ERR_ARG, "gemm_slices: operand planes");
  SliceArgs a = {};
  a.M = g.M;
  a.N = g.N;
  a.K = g.src.K;
  a.rows_a = A.plane_rows;
  a.rows_b = B.plane_rows;
  a.a_row0 = 2 * g.a_row0;
  a.b_row0 = g.b_row0;
  a.ea = A.e;
  a.eb = B.e;
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
  const SlicePlan p = slice_plan(g.M, g.N, a.num_kb, num_sms);
  a.kb_per_split = p.kb_per_split;
  a.k_splits = p.k_splits;
  a.n_tiles = p.n_tiles;
  a.m_tiles = p.m_tiles;
  const double square = std::sqrt(static_cast<double>(p.pair ? num_sms / 2 : num_sms) * SBN / (p.pair ? 2 * BM : BM));
  a.group_m = std::max(1, std::min(a.m_tiles, static_cast<int>(square)));
  if (p.units() > 0x7fffffffL) fail(CC_ERR_ARG, "gemm_slices: too many tiles");
  if (!g.scratch || g.scratch_bytes < slice_scratch_bytes(g.M, g.N, g.src.K, num_sms) ||
      slice_kp(g.src.K) != A.Kp)
    fail(CC_ERR_ARG, "gemm_slices: scratch");
  a.fix.patches = p.patches();
  a.fix.queue = static_cast<int *>(g.scratch);
  a.fix.list = reinterpret_cast<unsigned long long *>(static_cast<char *>(g.scratch) + SLICE_RESET_BYTES);
  a.fix.mask = reinterpret_cast<unsigned *>(a.fix.list + p.patches() * FIX_FEW);
  a.wmode = (g.beta.x == 0.0 && g.beta.y == 0.0) ? SW_STORE
            : (g.beta.x == 1.0 && g.beta.y == 0.0) ? SW_ADD
                                                   : SW_BETA;
  if (a.k_splits > 1) {
    scale_2d(g.C, g.cm, g.cn, g.ldc, g.M, g.N, g.beta, st);
    a.wmode = SW_ADD;
  }
  // (the rule of gemm_f64 for outputs that warps sum, in short chains; its
  // tiles sum K terms one after another)
  const long tiles = (g.M + 63) / 64 * ((g.N + 63) / 64);
  a.least = tiles < num_sms && g.M * g.N <= 65535L * 8 ? 0x1p-7f : 0x1.6ap-9f;
  const int u = static_cast<int>(p.units());
  if (p.pair) launch_slices<4, true>(a, A, B, u, num_sms, st);
  else launch_slices<3, false>(a, A, B, u, num_sms, st);
  // the elements left out, on the FP64 pipe
  FixArgs f = {};
  f.M = g.M;
  f.N = g.N;
  f.K = g.src.K;
  f.k_per_split = 32L * p.kb_per_split;
  f.pm = p.patches_m();
  f.pn = p.patches_n();
  f.fix = a.fix;
  f.err = err;
  f.A = FixSide{g.src.A, g.src.am, g.src.ak, g.src.lda, g.src.conjA, g.a_rows};
  f.B = FixSide{g.src.B, g.src.bn, g.src.bk, g.src.ldb, g.src.conjB, g.b_rows};
  f.C = g.C;
  f.cm = g.cm;
  f.cn = g.cn;
  f.ldc = g.ldc;
  f.alpha = g.alpha;
  f.beta = g.beta;
  f.wmode = a.wmode;
  const long blocks = std::min<long>(f.fix.patches, static_cast<long>(FIX_BLOCKS) * num_sms);
  slice_fix_kernel<<<static_cast<unsigned>(blocks), FIX_THREADS, 0, st>>>(f);
  LAUNCH_CHECK();
  count_launch();
}

// Estimated times (s) of an M x N x K product here and on the FP64 pipe. The
// tensor side: 29 products of every 128 x 128 x 64 block at about 1
// PF/s, an epilogue of three K blocks per tile, the planes written and read,
// five launches per block of 65536 k (8 x 64 x 300000, five blocks: 1.87 ms,
// 1.21 on the FP64 pipe). The FP64 side: 1 TF/s or its operands at 5 TB/s, on whole
// 64 x 64 tiles where the tiled kernel takes the product (a tile's rows cost
// the same empty: 5 x 64000 x 160 took 4.5 ms there).
bool slices_pay(long M, long N, long K) {
  const double m = (2 * M + 127) / 128 * 128.0, n = (N + 127) / 128 * 128.0;
  const double kb = static_cast<double>((2 * K + 63) / 64);
  const double mma = 2.0 * m * n * 64.0 * 29.0 * (kb + 3.0) / 1.04e15;
  const double pack = (static_cast<double>(M) * K * (32 + 128) + static_cast<double>(N) * K * (32 + 64)) / 5.5e12;
  const double out = 32.0 * M * N / 5e12;
  // (few outputs: K is split over many SMs, whose additions to the output cost
  // 10 us more; 30 x 30 x 10000 95 us, 85 on the FP64 pipe)
  const double few = M * N <= 4096 ? 10e-6 : 0.0;
  const double t_slices = 20e-6 * ((K + 65535) / 65536) + few + std::max(mma, 20e-6) + pack + out;
  const long tm = (M + 63) / 64, tn = (N + 63) / 64;
  const bool skinny = K <= SKINNY64_MAX_K && std::min(M, N) <= 256 && std::max(M, N) >= 1024;
  const bool tiled = M > 1 && N > 1 && !skinny && tm * tn >= 152;
  const double mn = tiled ? 4096.0 * tm * tn : static_cast<double>(M) * N;
  const double t_f64 = 4e-6 + std::max(8.0 * mn * K / 1e12, 16.0 * (static_cast<double>(M) * K + static_cast<double>(N) * K) / 5e12);
  return t_slices < 0.8 * t_f64;
}

}  // namespace cdfns
