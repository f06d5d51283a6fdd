// FP64-accurate complex GEMM on the FP16 tensor cores by exact integer slicing.
//
// GB300 runs FP64 FMA at 1.25 TFLOP/s; its tensor cores run FP16 about 1500 times faster.
// The FP64 products of the update (the FP64 H_eff.theta, theta, the environments, the SVD's
// Gram matrices and projections) are therefore computed as sums of exact integer products
// (the Ozaki splitting):
//   * every row i of A has a power of two 2^a_i > max_k |A_ik| (re and im), every column j
//     of B a power 2^b_j;
//   * A_ik 2^-a_i is rounded to the 55-bit fixed-point value F 2^-55 and written in balanced
//     base-128 digits, F = sum_p d_p 128^(8-p), -64 <= d_p <= 64: eight slices of integers
//     that FP16 holds exactly; likewise B;
//   * a product of digits is an integer of at most 2^12, and the sum over a K chunk of 256
//     and over all pairs (p, q) of one level p + q = l (at most 8 pairs, two terms each of
//     a complex part) is at most 2^24: FP32 accumulation gives the level's sum exactly;
//   * the level sums are integers, combined in 64-bit integer arithmetic: the four top
//     levels H = sum_{l=2..5} 128^(5-l) S_l and the four others L = sum_{l=6..9} 128^(9-l) S_l
//     are exact over all of K; C = (2^28 H + L) 2^(a_i + b_j - 61), rounded once, by a
//     second kernel (in the MMA kernel's eight epilogue warps that conversion took 25 to
//     60 us a tile, more than the tile's MMAs).
// The pairs left out (p + q > 9) and the digits' rounding are below 3 K 2^-53 2^(a_i + b_j) in
// the worst case and of random sign; the result does not depend on tiling or K splits.
// No FP64-pipe instruction runs in these kernels: an SM retires two FP64 operations per
// clock, and combining the level sums in FP64 (with TF32 operands, six-bit digits and 45
// pairs) took longer than the MMAs.  Measured: H_eff.theta at chi = 256, d = 4 (two products
// of 1.07 G complex multiply-adds) 5.71 -> 0.67 ms; theta and its gate at chi = 512, d = 5 7.3 ->
// 0.94 ms.  What bounds it: operand reads from
// shared memory (an N = 128 MMA takes about 90 clocks for 64 clocks of arithmetic).
//
// Kernel: persistent, one CTA per SM over items (output tile 128 x 64, level group, K
// split).  A complex multiply-add is two MMAs of N = 128: A_re with the rows [B_re; B_im] of
// the B tile gives the real and the imaginary part side by side, A_im with [-B_im; B_re]
// adds the rest (the B tile keeps three planes, -im, re, im).  The group's four levels
// accumulate at once in the 512 TMEM columns, so a slice tile is loaded once per 32 of K
// and group instead of once per pair: 28 KB per 1024 MMA clocks, which the L2 can feed.
// Within a block of 32 of K, A's slices p stream through a ring; slice q of B stays in its
// own ring from its first to its last pair.  The slice kernel writes the tiles in the
// shared-memory order (64-byte rows, 64-byte swizzle), so a load is one bulk copy and no
// tensor map is built.  Warp 0 loads, warp 1 issues, warps 2..9 convert the level sums.
// All waits bounded.
#include <algorithm>
#include <cmath>
#include <vector>

#include "heff_plan.cuh"
#include "tc_common.cuh"
#include "f32conv.cuh"
#include "oz.cuh"

namespace tnt {

namespace {
using namespace tc;

constexpr int OZ_S = 8;                         // slices per operand
constexpr int OZ_KB = 32;                       // K of one slice tile (64 bytes of FP16)
constexpr int OZ_CHUNK = 8;                     // K blocks per exact FP32 accumulation
constexpr int OZ_BM = 128, OZ_BN = 64;          // output tile
constexpr int OZ_TA = 2 * OZ_BM * 64;           // A slice tile: re, im
constexpr int OZ_TB = 3 * OZ_BN * 64;           // B slice tile: -im, re, im
constexpr int OZ_NA = 6, OZ_NB = 10;            // ring stages
constexpr int OZ_SMEM = OZ_NA * OZ_TA + OZ_NB * OZ_TB + 1024 + 512;
constexpr int OZ_EPI = 8;                       // epilogue warps
constexpr int OZ_THREADS = 64 + 32 * OZ_EPI;
constexpr int OZ_SPLIT_LEVEL = 5;               // group 0: levels 2..5, group 1: 6..9
constexpr int OZ_PAIRS0 = 10, OZ_PAIRS1 = 26;   // slice pairs of the two groups
static_assert(2LL * OZ_S * OZ_CHUNK * OZ_KB * 64 * 64 <= (1LL << 24),
              "a level sum over one K chunk must stay exact in FP32");
static_assert(OZ_SMEM <= 227 * 1024, "rings fit the shared memory of an SM");

// one product of a launch; offsets are bytes into the launch's buffer
struct OzTask {
  const z *A, *B;
  z* C;
  int64_t a_rs, a_ks, b_rs, b_ks, c_rs;  // A(i, k) = A[i a_rs + k a_ks], B(k, j) = B[j b_rs + k b_ks]
  int64_t offA, offB, offE, offP;        // slice tiles, exponent fields (M then N), partial sums
  int64_t atom0[2];                      // first slice atom among all tasks', per side
  int M, N, K;
  int ntm, ntn, nkb;                     // tiles along M and N, K blocks of 32
  int ks, both;                          // K splits; an item runs both level groups, or one
  int conj_a, conj_b;
  int herm;  // C = A B is Hermitian: tiles strictly above the diagonal are mirrored, not computed
  int sub;   // C -= A B
  int item0, scale0[2], fin0;            // first item / scale block (per side) / finish block
  int grp0[2];                           // first group of eight rows, per side
};
// The products of one launch travel as a kernel argument (no table upload), or, for a plan
// whose products repeat, in device memory (CAP = 0).
constexpr int OZ_MAXT = 40;
struct OzHead {
  int n, items, fin_blocks;
  int scale_blocks[2];  // per side (A, B)
  int groups[2];        // of eight rows, padding to whole tiles included
  int64_t atoms[2];
  int sides;            // the sides to scale and slice: bit 0 A, bit 1 B
  int64_t add_b;        // bytes added to every task's B
  uint8_t* buf;
  int* status;
};
template <int CAP>
struct OzTasks {
  OzHead h;
  OzTask t[CAP];
  __device__ __forceinline__ const OzTask& at(int i) const { return t[i]; }
};
template <>
struct OzTasks<0> {
  OzHead h;
  const OzTask* t;
  __device__ __forceinline__ const OzTask& at(int i) const { return t[i]; }
};
// the last task whose first index (by FIRST) is at most w
template <int CAP, typename F>
__device__ __forceinline__ int oz_find(const OzTasks<CAP>& T, F first, int64_t w) {
  if (CAP == 1) return 0;
  int lo = 0, hi = T.h.n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if ((int64_t)first(T.at(mid)) <= w) lo = mid;
    else hi = mid;
  }
  return lo;
}

struct OzItem {
  int task, mt, nt, g0, g1, kb0, kb1, sp;  // groups g0..g1, K blocks [kb0, kb1)
};
// item w of the launch; a task's heavier groups come first.  false: a tile left out
template <int CAP>
__device__ __forceinline__ bool oz_item(const OzTasks<CAP>& T, int w, OzItem* it) {
  it->task = oz_find(T, [](const OzTask& t) { return t.item0; }, w);
  const OzTask& g = T.at(it->task);
  w -= g.item0;
  const int ntiles = g.ntm * g.ntn;
  const int t = w % ntiles, r = w / ntiles;
  it->mt = t / g.ntn;
  it->nt = t % g.ntn;
  if (g.both) {
    it->g0 = 0;
    it->g1 = 1;
  } else {
    it->g0 = it->g1 = r < g.ks ? 1 : 0;
  }
  it->sp = r % g.ks;
  it->kb0 = (int)((int64_t)it->sp * g.nkb / g.ks);
  it->kb1 = (int)((int64_t)(it->sp + 1) * g.nkb / g.ks);
  return !(g.herm && it->mt * OZ_BM + OZ_BM <= it->nt * OZ_BN);
}
// pairs (p, q) of group levels l0..l1 at slice p of A: q in [qlo, qhi]
__device__ __forceinline__ void oz_levels(int grp, int* l0, int* l1) {
  *l0 = grp ? OZ_SPLIT_LEVEL + 1 : 2;
  *l1 = grp ? OZ_S + 1 : OZ_SPLIT_LEVEL;
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          su32(dst)),
      "l"(src), "r"(bytes), "r"(su32(bar))
      : "memory");
}
// instruction descriptor: D = F32, A = B = F16, both K-major, M = 128, N = 128
constexpr uint32_t OZ_IDESC = (1u << 4) | ((uint32_t)(128 >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
__device__ __forceinline__ void mma_f16(uint32_t tmem, uint32_t alo, uint32_t blo, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "mov.b64 a, {%1, %5};\n\t"
      "mov.b64 b, {%2, %5};\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}\n" ::"r"(tmem),
      "r"(alo), "r"(blo), "r"(OZ_IDESC), "r"(acc), "r"(DESC_SW64_HI)
      : "memory");
}

// The MMAs of one K block of group GRP: the loop over the pairs is unrolled, so that the one
// issuing thread spends about ten instructions per MMA (with the ring slots and descriptors
// computed in a rolled loop it took about 200 clocks per 64-clock MMA, 450 us for a
// 1024 x 1024 x 1024 product that is 142 us of MMAs).  sa / sb: ring slots of the block's
// first A and B slice, with the phases of their barriers in pa / pb.
struct OzIssue {
  uint32_t a0, b0;  // descriptor low words of the rings
  uint64_t *fa, *ea, *fb, *eb;
  uint64_t* acce;  // set: a level's first MMA waits until its last sums have been read
  uint32_t pacc;
  uint32_t sa, pa, sb, pb;
};
template <int GRP>
__device__ __forceinline__ bool oz_issue_block(OzIssue& r, uint32_t tmem, bool first, int* status) {
  constexpr int L0 = GRP ? OZ_SPLIT_LEVEL + 1 : 2, L1 = GRP ? OZ_S + 1 : OZ_SPLIT_LEVEL;
  constexpr int QM = L1 - 1;  // slices of either operand
  uint32_t blo[QM];
  uint32_t sq = r.sb, pq = r.pb;  // slot and phase of the next slice of B (descending q)
#pragma unroll
  for (int p = 1; p <= QM; ++p) {
    constexpr int LL0 = L0;
    const int qlo = LL0 - p > 1 ? LL0 - p : 1, qhi = L1 - p < QM ? L1 - p : QM;
    const int qprev = p == 1 ? QM + 1 : (LL0 - p + 1 > 1 ? LL0 - p + 1 : 1);  // lowest slice seen before
    if (!mbar_wait(&r.fa[r.sa], r.pa, status)) return false;
    const uint32_t alo = r.a0 + r.sa * (uint32_t)(OZ_TA >> 4);
#pragma unroll
    for (int q = qhi; q >= qlo; --q) {
      if (q < qprev) {
        if (!mbar_wait(&r.fb[sq], pq, status)) return false;
        blo[q - 1] = r.b0 + sq * (uint32_t)(OZ_TB >> 4);
        if (++sq == OZ_NB) {
          sq = 0;
          pq ^= 1;
        }
      }
      if (p == 1 && r.acce && !mbar_wait(&r.acce[q + 1 - L0], r.pacc, status)) return false;
      if (q == qhi || q < qprev) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d = tmem + (uint32_t)(p + q - L0) * 128u, bq = blo[q - 1];
      // every level's first pair has p = 1
      mma_f16(d, alo, bq + (OZ_BN * 64 >> 4), p == 1 ? (first ? 0u : 1u) : 1u);
      mma_f16(d, alo + (OZ_BM * 64 >> 4), bq, 1u);
      mma_f16(d, alo + 2, bq + (OZ_BN * 64 >> 4) + 2, 1u);
      mma_f16(d, alo + (OZ_BM * 64 >> 4) + 2, bq + 2, 1u);
    }
    mma_commit(&r.ea[r.sa]);
    if (++r.sa == OZ_NA) {
      r.sa = 0;
      r.pa ^= 1;
    }
    mma_commit(&r.eb[r.sb]);  // the last pair of slice q = L1 - p, the oldest in its ring
    if (++r.sb == OZ_NB) {
      r.sb = 0;
      r.pb ^= 1;
    }
  }
  return true;
}

// one group's loads of an item, in the order of first use
struct OzRings {
  uint8_t *a, *b;
  uint64_t *fa, *ea, *fb, *eb;
};

// 32 pairs of one row to memory (nc of them exist), two per 32-byte store where o allows it
__device__ __forceinline__ void oz_put(longlong2* o, int nc, const long long* re, const long long* im) {
  if (nc == 32 && ((uintptr_t)o & 31) == 0) {
#pragma unroll
    for (int j = 0; j < 32; j += 2)
      asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(o + j), "l"(re[j]), "l"(im[j]), "l"(re[j + 1]),
                   "l"(im[j + 1])
                   : "memory");
    return;
  }
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (j < nc) o[j] = make_longlong2(re[j], im[j]);
}

template <int CAP>
__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz_gemm(const __grid_constant__ OzTasks<CAP> T) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  OzRings R;
  R.a = smem;
  R.b = smem + OZ_NA * OZ_TA;
  R.fa = (uint64_t*)(R.b + OZ_NB * OZ_TB);
  R.ea = R.fa + OZ_NA;
  R.fb = R.ea + OZ_NA;
  R.eb = R.fb + OZ_NB;
  uint64_t* accf = R.eb + OZ_NB;
  uint64_t* acce = accf + 1;
  uint32_t* tmem_slot = (uint32_t*)(acce + 4);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nitems = T.h.items;

  if (threadIdx.x == 0) {
    for (int s = 0; s < OZ_NA; ++s) {
      mbar_init(&R.fa[s], 1);
      mbar_init(&R.ea[s], 1);
    }
    for (int s = 0; s < OZ_NB; ++s) {
      mbar_init(&R.fb[s], 1);
      mbar_init(&R.eb[s], 1);
    }
    mbar_init(accf, 1);
    for (int l = 0; l < 4; ++l) mbar_init(&acce[l], OZ_EPI);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------ loads
    uint32_t ia = 0, ib = 0;
    bool stop = false;
    auto load = [&](uint8_t* ring, uint64_t* full, uint64_t* empty, uint32_t& i, int n, uint32_t bytes,
                    const uint8_t* src) {
      const int s = (int)(i % (uint32_t)n);
      if (i >= (uint32_t)n && !mbar_wait(&empty[s], ((i / n) & 1) ^ 1, T.h.status)) *abort_flag = 1;
      if (*abort_flag) {
        stop = true;
        return;
      }
      mbar_expect_tx(&full[s], bytes);
      bulk_load(ring + (size_t)s * bytes, src, bytes, &full[s]);
      ++i;
    };
    for (int w = blockIdx.x; w < nitems && !stop; w += gridDim.x) {
      OzItem it;
      if (!oz_item(T, w, &it)) continue;
      const OzTask& g = T.at(it.task);
      for (int grp = it.g0; grp <= it.g1 && !stop; ++grp) {
        int l0, l1;
        oz_levels(grp, &l0, &l1);
        const int pmax = min(OZ_S, l1 - 1);
        for (int kb = it.kb0; kb < it.kb1 && !stop; ++kb) {
          const uint8_t* A = T.h.buf + g.offA + ((int64_t)it.mt * g.nkb + kb) * (OZ_S * OZ_TA);
          const uint8_t* B = T.h.buf + g.offB + ((int64_t)it.nt * g.nkb + kb) * (OZ_S * OZ_TB);
          int qnext = min(OZ_S, l1 - 1);  // next slice of B to load (descending)
          for (int p = 1; p <= pmax && !stop; ++p) {
            const int qlo = max(1, l0 - p);
            for (; qnext >= qlo && !stop; --qnext)
              load(R.b, R.fb, R.eb, ib, OZ_NB, OZ_TB, B + (qnext - 1) * OZ_TB);
            if (!stop) load(R.a, R.fa, R.ea, ia, OZ_NA, OZ_TA, A + (p - 1) * OZ_TA);
          }
        }
      }
    }
    // copies in flight land before the CTA may exit
    for (uint32_t i = (ia > (uint32_t)OZ_NA ? ia - OZ_NA : 0u); i < ia; ++i)
      mbar_wait(&R.fa[i % OZ_NA], (i / OZ_NA) & 1, T.h.status);
    for (uint32_t i = (ib > (uint32_t)OZ_NB ? ib - OZ_NB : 0u); i < ib; ++i)
      mbar_wait(&R.fb[i % OZ_NB], (i / OZ_NB) & 1, T.h.status);
  } else if (warp == 1 && lane == 0) {
    // ------------------------------------------------ MMA issue
    uint32_t sub = 0;
    bool stop = false;
    OzIssue r{desc_lo(su32(R.a)), desc_lo(su32(R.b)), R.fa, R.ea, R.fb, R.eb, nullptr, 0, 0, 0, 0, 0};
    for (int w = blockIdx.x; w < nitems && !stop; w += gridDim.x) {
      OzItem it;
      if (!oz_item(T, w, &it)) continue;
      for (int grp = it.g0; grp <= it.g1 && !stop; ++grp) {
        for (int kb = it.kb0; kb < it.kb1; ++kb) {
          const bool first = ((kb - it.kb0) % OZ_CHUNK) == 0;
          bool ok = *abort_flag == 0;
          r.acce = first && sub > 0 ? acce : nullptr;
          r.pacc = (sub - 1) & 1;
          if (ok) ok = grp ? oz_issue_block<1>(r, tmem, first, T.h.status) : oz_issue_block<0>(r, tmem, first, T.h.status);
          if (!ok) {
            *abort_flag = 1;
            stop = true;
            break;
          }
          if (kb + 1 == it.kb1 || (kb + 1 - it.kb0) % OZ_CHUNK == 0) {
            mma_commit(accf);
            ++sub;
          }
        }
      }
    }
  } else if (warp >= 2) {
    // ------------------------------------------------ level sums into 64-bit integers
    const int q4 = warp & 3, half = (warp - 2) >> 2;
    const int row = q4 * 32 + lane;
    const uint32_t taddr = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(half * 32);
    uint32_t sub = 0;
    bool stop = false;
    for (int w = blockIdx.x; w < nitems && !stop; w += gridDim.x) {
      OzItem it;
      if (!oz_item(T, w, &it)) continue;
      const OzTask& g = T.at(it.task);
      const int64_t gm = (int64_t)it.mt * OZ_BM + row;
      const int64_t gn0 = (int64_t)it.nt * OZ_BN + half * 32;
      for (int grp = it.g0; grp <= it.g1 && !stop; ++grp) {
        long long re[32], im[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) re[j] = im[j] = 0;
        for (int kb = it.kb0; kb < it.kb1; kb += OZ_CHUNK) {
          if (*abort_flag || !mbar_wait(accf, sub & 1, T.h.status)) {
            *abort_flag = 1;
            stop = true;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
          for (int l = 3; l >= 0; --l) {  // the order in which the next chunk needs them
            const int wt = 1 << (7 * (3 - l));
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              uint32_t r[16];
              tmem_ld16(taddr + l * 128 + h * 16, r);
#pragma unroll
              for (int j = 0; j < 16; ++j)
                re[16 * h + j] += (long long)__float2int_rn(__uint_as_float(r[j])) * wt;
              tmem_ld16(taddr + l * 128 + 64 + h * 16, r);
#pragma unroll
              for (int j = 0; j < 16; ++j)
                im[16 * h + j] += (long long)__float2int_rn(__uint_as_float(r[j])) * wt;
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&acce[l]);
          }
          ++sub;
        }
        if (stop || gm >= g.M) continue;
        const int nc = (int)min((int64_t)32, (int64_t)g.N - gn0);  // columns of this half tile
        if (nc <= 0) continue;
        oz_put((longlong2*)(T.h.buf + g.offP) + ((int64_t)(2 * it.sp + grp) * g.M + gm) * g.N + gn0, nc, re, im);
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
}

// C from the partial sums of the K splits (integers: any order gives the same value); one
// element per thread, a block's 256 elements in one task.  Hermitian results: the lower
// triangle, mirrored.
template <int CAP>
__global__ void __launch_bounds__(256, 5) k_oz_finish(const __grid_constant__ OzTasks<CAP> T) {
  for (int fb = blockIdx.x; fb < T.h.fin_blocks; fb += gridDim.x) {
    const OzTask& g = T.at(oz_find(T, [](const OzTask& t) { return t.fin0; }, fb));
    const int64_t total = (int64_t)g.M * g.N, e0 = (int64_t)(fb - g.fin0) * 256, e = e0 + threadIdx.x;
    if (e >= total) continue;
    // row and column from the block's first element, in 32 bits (a 64-bit division a thread
    // cost as much as both conversions)
    const unsigned N = (unsigned)g.N;
    int64_t i = e < (1ll << 32) ? (unsigned)e0 / N : e0 / N;
    unsigned j = (unsigned)(e0 - i * N) + threadIdx.x;
    if (N > 256) {
      if (j >= N) j -= N, ++i;
    } else {
      i += j / N;
      j %= N;
    }
    if (g.herm && j > i) continue;
    const longlong2* P = (const longlong2*)(T.h.buf + g.offP) + e;
    longlong2 h = make_longlong2(0, 0), l = h;
#pragma unroll 2
    for (int s = 0; s < g.ks; ++s) {
      const longlong2 a = P[(int64_t)(2 * s) * total], b = P[(int64_t)(2 * s + 1) * total];
      h.x += a.x;
      h.y += a.y;
      l.x += b.x;
      l.y += b.y;
    }
    const int* ex = (const int*)(T.h.buf + g.offE);
    const int ea = ex[i], eb = ex[g.M + j];
    z v = zmk(oz_value(h.x, l.x, ea, eb), oz_value(h.y, l.y, ea, eb));
    z* o = g.C + i * g.c_rs + j;
    if (g.sub) v = zsub(*o, v);
    *o = v;
    if (g.herm && j < i) g.C[j * g.c_rs + i] = zconj(v);
  }
}

// ---------------------------------------------------------------- scales and slices
// one operand of a product seen as rows of K entries: X[i * rs + k * cs]
struct OzOp {
  const z* X;
  int64_t rows, rs, cs;
  int conj;
  int* e;        // per row: largest exponent field of the re and im parts
  uint8_t* out;  // slice tiles
};
// B enters as rows n with K along the row
__device__ __forceinline__ OzOp oz_operand(const OzTask& g, const OzHead& h, bool isb) {
  uint8_t* buf = h.buf;
  OzOp o;
  o.X = isb ? (const z*)((const char*)g.B + h.add_b) : g.A;
  o.rows = isb ? g.N : g.M;
  o.rs = isb ? g.b_rs : g.a_rs;
  o.cs = isb ? g.b_ks : g.a_ks;
  o.conj = isb ? g.conj_b : g.conj_a;
  o.e = (int*)(buf + g.offE) + (isb ? g.M : 0);
  o.out = buf + (isb ? g.offB : g.offA);
  return o;
}

// largest exponent field of every row.  Entries contiguous along K: one warp per row;
// otherwise 8 rows by up to OZ_SCALE_K of K per CTA, eight neighbouring lanes on neighbouring
// rows, one 128-byte line (a longer K combines its parts with an atomic maximum, e zeroed
// before).  Latency-bound: with 32 rows a CTA there were 64 of them for 2048 rows, and each
// thread had 64 loads to make.
constexpr int OZ_SCALE_K = 512;
__device__ __forceinline__ unsigned oz_exp(z v) {
  return max(((unsigned)__double2hiint(v.x) >> 20) & 0x7ffu, ((unsigned)__double2hiint(v.y) >> 20) & 0x7ffu);
}
__host__ __device__ inline int64_t oz_scale_blocks(int64_t rows, int64_t ks, int64_t K) {
  return ((rows + 7) / 8) * (ks == 1 ? 1 : (K + OZ_SCALE_K - 1) / OZ_SCALE_K);
}
template <int CAP>
__global__ void __launch_bounds__(256) k_oz_scale(const __grid_constant__ OzTasks<CAP> T) {
  const int na = (T.h.sides & 1) ? T.h.scale_blocks[0] : 0;
  const bool isb = (int)blockIdx.x >= na;
  const int w = (int)blockIdx.x - (isb ? na : 0);
  const OzTask& g = T.at(isb ? oz_find(T, [](const OzTask& t) { return t.scale0[1]; }, w)
                             : oz_find(T, [](const OzTask& t) { return t.scale0[0]; }, w));
  const int64_t K = g.K, blk = w - g.scale0[isb];
  const OzOp o = oz_operand(g, T.h, isb);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (o.cs == 1) {
    const int64_t i = blk * 8 + warp;
    if (i >= o.rows) return;
    unsigned mx = 0;
    const z* x = o.X + i * o.rs;
#pragma unroll 8
    for (int64_t k = lane; k < K; k += 32) mx = max(mx, oz_exp(x[k]));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) o.e[i] = (int)mx;
    return;
  }
  __shared__ unsigned s_mx[8];
  if (threadIdx.x < 8) s_mx[threadIdx.x] = 0;
  __syncthreads();
  const int64_t nk = (K + OZ_SCALE_K - 1) / OZ_SCALE_K, k0 = (blk % nk) * OZ_SCALE_K, i = (blk / nk) * 8 + (lane & 7);
  unsigned mx = 0;
  if (i < o.rows) {
    const int64_t k1 = min(K, k0 + OZ_SCALE_K);
    const z* x = o.X + i * o.rs;
#pragma unroll 8
    for (int64_t k = k0 + (threadIdx.x >> 3); k < k1; k += 32) mx = max(mx, oz_exp(x[k * o.cs]));
  }
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
  mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
  if (mx && lane < 8) atomicMax(&s_mx[lane], mx);
  __syncthreads();
  if (threadIdx.x < 8 && i < o.rows) {
    if (nk == 1) o.e[i] = (int)s_mx[lane];
    else atomicMax((unsigned*)o.e + i, s_mx[lane]);
  }
}

// slices of 8 rows by 32 of K per warp: lane = (row, 8 of K), so every plane's 512-byte
// swizzle atom is written whole.  Rows and K beyond the operand are zero.
template <int PLANES>
__device__ __forceinline__ void oz_slice_atom(const OzOp& o, int64_t K, int nkb, int64_t i8, int kb, int lane, int e) {
  constexpr int ROWS = PLANES == 2 ? OZ_BM : OZ_BN, TILE = PLANES == 2 ? OZ_TA : OZ_TB;
  const int r = lane >> 2, c8 = lane & 3;
  const int64_t i = i8 * 8 + r, k0 = (int64_t)kb * OZ_KB + c8 * 8;
  uint64_t fr[8], fi[8];
  uint32_t sr[4], si[4];  // signs of the eight entries, as bits 15 and 31 of a word per pair
  const z* x = o.X + i * o.rs + k0 * o.cs;
  z v[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) v[t] = (i < o.rows && k0 + t < K) ? x[t * o.cs] : zmk(0, 0);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const uint32_t cj = o.conj ? 0x80008000u : 0u;
    sr[t] = oz_signs(v[2 * t].x, v[2 * t + 1].x);
    si[t] = oz_signs(v[2 * t].y, v[2 * t + 1].y) ^ cj;
  }
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    fr[t] = oz_fixed(v[t].x, e) + OZ_BIAS;
    fi[t] = oz_fixed(v[t].y, e) + OZ_BIAS;
  }
  const int64_t rt = (i8 * 8) / ROWS;
  const int ra = (int)((i8 * 8) % ROWS) / 8;
  uint8_t* base = o.out + (rt * nkb + kb) * (int64_t)(OZ_S * TILE) + ra * 512 + r * 64 + ((c8 ^ ((r >> 1) & 3)) << 4);
#pragma unroll
  for (int p = 0; p < OZ_S; ++p) {
    uint32_t wr[4], wi[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      wr[t] = oz_digit2(fr[2 * t], fr[2 * t + 1], p, sr[t]);
      wi[t] = oz_digit2(fi[2 * t], fi[2 * t + 1], p, si[t]);
    }
    uint8_t* q = base + p * TILE;
    if (PLANES == 3) {
      *(uint4*)q = make_uint4(wi[0] ^ 0x80008000u, wi[1] ^ 0x80008000u, wi[2] ^ 0x80008000u, wi[3] ^ 0x80008000u);
      q += ROWS * 64;
    }
    *(uint4*)q = make_uint4(wr[0], wr[1], wr[2], wr[3]);
    *(uint4*)(q + ROWS * 64) = make_uint4(wi[0], wi[1], wi[2], wi[3]);
  }
}
template <int PLANES>
__device__ __forceinline__ void oz_slice_at(const OzOp& o, int64_t K, int nkb, int64_t atom, int lane) {
  const int64_t i8 = atom / nkb, i = i8 * 8 + (lane >> 2);
  oz_slice_atom<PLANES>(o, K, nkb, i8, (int)(atom % nkb), lane, i < o.rows ? o.e[i] : 0);
}
template <int CAP>
__global__ void __launch_bounds__(256) k_oz_slice(const __grid_constant__ OzTasks<CAP> T) {
  const int lane = threadIdx.x & 31;
  const int64_t na = (T.h.sides & 1) ? T.h.atoms[0] : 0, all = na + ((T.h.sides & 2) ? T.h.atoms[1] : 0);
  for (int64_t w = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); w < all; w += (int64_t)gridDim.x * 8) {
    if (w < na) {
      const OzTask& g = T.at(oz_find(T, [](const OzTask& t) { return t.atom0[0]; }, w));
      oz_slice_at<2>(oz_operand(g, T.h, false), g.K, g.nkb, w - g.atom0[0], lane);
    } else {
      const OzTask& g = T.at(oz_find(T, [](const OzTask& t) { return t.atom0[1]; }, w - na));
      oz_slice_at<3>(oz_operand(g, T.h, true), g.K, g.nkb, w - na - g.atom0[1], lane);
    }
  }
}

// Scales and slices of K up to OZ_SCALE_K in one launch: a CTA takes eight rows, their
// maxima first, then their slices (the second read hits L1 or L2).  Small products are bound by
// the launches (scale and slice 5 to 7 us each); oz_one_prep says where.
template <int CAP>
__global__ void __launch_bounds__(256) k_oz_prep(const __grid_constant__ OzTasks<CAP> T) {
  __shared__ unsigned s_mx[8];
  const int na = (T.h.sides & 1) ? T.h.groups[0] : 0;
  const bool isb = (int)blockIdx.x >= na;
  const int w = (int)blockIdx.x - (isb ? na : 0);
  const OzTask& g = T.at(isb ? oz_find(T, [](const OzTask& t) { return t.grp0[1]; }, w)
                             : oz_find(T, [](const OzTask& t) { return t.grp0[0]; }, w));
  const OzOp o = oz_operand(g, T.h, isb);
  const int K = g.K, nkb = g.nkb, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t i8 = w - g.grp0[isb];
  if (o.cs == 1) {
    const int64_t i = i8 * 8 + warp;
    unsigned mx = 0;
    if (i < o.rows) {
      const z* x = o.X + i * o.rs;
#pragma unroll 8
      for (int k = lane; k < K; k += 32) mx = max(mx, oz_exp(x[k]));
    }
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) s_mx[warp] = mx;
  } else {
    if (threadIdx.x < 8) s_mx[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = i8 * 8 + (lane & 7);
    unsigned mx = 0;
    if (i < o.rows) {
      const z* x = o.X + i * o.rs;
#pragma unroll 8
      for (int k = threadIdx.x >> 3; k < K; k += 32) mx = max(mx, oz_exp(x[k * o.cs]));
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    if (mx && lane < 8) atomicMax(&s_mx[lane], mx);
  }
  __syncthreads();
  if (threadIdx.x < 8 && i8 * 8 + threadIdx.x < o.rows) o.e[i8 * 8 + threadIdx.x] = (int)s_mx[threadIdx.x];
  const int e = (int)s_mx[lane >> 2];
  for (int kb = warp; kb < nkb; kb += 8) {
    if (isb) oz_slice_atom<3>(o, K, nkb, i8, kb, lane, e);
    else oz_slice_atom<2>(o, K, nkb, i8, kb, lane, e);
  }
}

int64_t cdiv(int64_t a, int64_t b) { return (a + b - 1) / b; }

// How a product of `tiles` output tiles and nkb K blocks is dealt to nsm SMs: K splits, and
// whether an item takes both level groups (one CTA then loads the rings once) or one.  In
// units of one slice pair over one K block (about 330 clocks) an item costs its pairs times
// its blocks plus about 8 per group for reading the level sums out; the partial sums of one
// tile and split cost about 0.4 to write and read back (0.5 MB), spread over the GPU.
struct OzDeal {
  int ks, both;
};
OzDeal oz_deal(int64_t tiles, int64_t nkb, int nsm) {
  OzDeal best{1, 1};
  double cost = 1e300;
  for (int ks = 1; ks <= 16 && ks <= nkb; ++ks) {
    if (ks > 1 && tiles * (ks - 1) >= nsm) break;
    const double kb = (double)cdiv(nkb, ks), heavy = OZ_PAIRS1 * kb + 8.0, light = OZ_PAIRS0 * kb + 8.0;
    const int64_t n = tiles * ks;
    const double sums = 0.4 * (double)n;
    for (int both = 1; both >= 0; --both) {
      double c;
      if (both) {
        c = (double)cdiv(n, nsm) * (heavy + light);
      } else {
        // items w, w + nsm, ... of one CTA; the n heavy ones come first
        c = 0;
        for (int64_t b : {(int64_t)0, n % nsm, (2 * n) % nsm, (int64_t)nsm - 1}) {
          const int64_t all = 2 * n > b ? cdiv(2 * n - b, nsm) : 0, h = n > b ? cdiv(n - b, nsm) : 0;
          c = std::max(c, (double)h * heavy + (double)(all - h) * light);
        }
      }
      c += sums;
      if (c < cost * 0.98) {
        cost = c;
        best = OzDeal{ks, both};
      }
    }
  }
  return best;
}

}  // namespace

// Where the slice product is the faster one.  The FP64 kernel's 16 x 16 tiles take 0.27 us per
// K entry and round of one tile per SM (512 FMAs of 256 threads at two per clock), down to a
// quarter of that for tiles four rows high when there are few; the launches here take about
// 30 us however small the product.  Measured with 16 x 16 tiles (FP64 / slices, us):
// 128 x 512 x 32 35 / 30, 64 x 512 x 64 18 / 27, 256 x 256 x 64 36 / 30,
// 256 x 1024 x 64 125 / 32, 64 x 64 x 1024 280 / 39.
// Accuracy, rms error against extended precision relative to the rms result (FP64 units /
// slices), Gaussian entries: 512 x 4096 x 16 1.8e-16 / 1.4e-16, 256 x 1024 x 64 2.5e-16 / 2.1e-16,
// 128 x 512 x 128 1.9e-16 / 2.7e-16 (the low tiles' partial sums), 2048 x 512 x 512 1.0e-15 / 3.7e-16;
// one operand falling by four decades along K: 3.4e-16 / 5.3e-16 at K = 64, 1.3e-15 / 7.6e-16 at
// K = 512.  Entries far below their row's largest keep fewer bits (see tnt_set_fp64_gemm): with
// operands that fall and rise against each other by four decades 2e-16 / 5e-13; FP64 H_eff of MPO
// environments, whose channels differ by decades, at chi = 64: 2e-16 / 6e-15 of the largest entry.
// Over the range of use (bonds of 12 to 512) the errors of matvecs, solves, environments, theta
// and SVDs agree between the engines within their references' own (1e-15, SVDs 1e-13).
static double fma_rounds(const Ctx* c, double k, double tiles) { return k * std::max(0.3, tiles / c->nsm); }
bool ozgemm_eligible(const Ctx* c, const ZGemm& g) {
  if (c->oz_mode == 0 || g.batch != 1 || g.alpha.x != 1.0 || g.alpha.y != 0.0 || g.beta.x != 0.0 ||
      g.beta.y != 0.0 || g.M < 16 || g.N < 16 || g.K < 16 || g.M >= (1LL << 31) || g.N >= (1LL << 31))
    return false;
  const double tiles = (double)cdiv(g.M, 16) * (double)cdiv(g.N, 16) * (g.lower_only ? 0.5 : 1.0);
  return fma_rounds(c, (double)g.K, tiles) >= 110.0;
}

namespace {
int oz_setup(Ctx* c) {
  TNT_TRY(func_smem(c, (const void*)k_oz_gemm<1>, OZ_SMEM));
  TNT_TRY(func_smem(c, (const void*)k_oz_gemm<OZ_MAXT>, OZ_SMEM));
  return func_smem(c, (const void*)k_oz_gemm<0>, OZ_SMEM);
}

// tables of the products tk[0..n): T's head and tasks, and the bytes of buffer they use
size_t oz_layout(const GemmTask* const* tk, int n, int sm, OzHead* h, OzTask* t, double* flop, double* bytes) {
  size_t off = 0;
  int64_t items = 0, scale[2] = {0, 0}, groups[2] = {0, 0}, fin = 0, rows = 0;
  double work = 0, wflop = 0, wbytes = 0;
  *h = OzHead{};
  h->n = n;
  h->sides = 3;
  for (int i = 0; i < n; ++i) {
    const ZGemm& g = tk[i]->g;
    OzTask& o = t[i];
    o.A = g.A; o.B = g.B; o.C = g.C;
    o.a_rs = g.a_rs; o.a_ks = g.a_cs; o.b_rs = g.b_cs; o.b_ks = g.b_rs; o.c_rs = g.c_rs;
    o.conj_a = g.conj_a; o.conj_b = g.conj_b;
    o.herm = tk[i]->herm; o.sub = tk[i]->sub;
    o.M = (int)g.M; o.N = (int)g.N; o.K = (int)g.K;
    o.ntm = (int)cdiv(g.M, OZ_BM);
    o.ntn = (int)cdiv(g.N, OZ_BN);
    o.nkb = (int)cdiv(g.K, OZ_KB);
    work += 36.0 * o.nkb * o.ntm * o.ntn;
    wflop += (o.herm ? 4.0 : 8.0) * (double)g.M * (double)g.N * (double)g.K;
  }
  for (int i = 0; i < n; ++i) {
    OzTask& o = t[i];
    const double mn = (double)o.M * (double)o.N;
    OzDeal deal{1, 1};
    if (n == 1) {
      deal = oz_deal((int64_t)o.ntm * o.ntn, o.nkb, sm);
    } else if (work < 4.0 * sm * 36.0 * o.nkb) {
      // few items per SM: none longer than half of an SM's share, nor shorter than two blocks
      const double share = std::max(work / sm * 0.5, 72.0);
      deal.ks = (int)std::min<int64_t>(std::max(1, o.nkb / 2), (int64_t)std::ceil(36.0 * o.nkb / share));
    }
    while (deal.ks > 1 && 32.0 * deal.ks * mn > 256e6) --deal.ks;
    o.ks = deal.ks;
    o.both = deal.both;
    o.offA = (int64_t)off;
    off += ws_round((size_t)o.ntm * o.nkb * OZ_S * OZ_TA);
    o.offB = (int64_t)off;
    off += ws_round((size_t)o.ntn * o.nkb * OZ_S * OZ_TB);
    o.offP = (int64_t)off;
    off += ws_round(sizeof(longlong2) * 2 * (size_t)o.ks * (size_t)mn);
    wbytes += 16.0 * ((double)o.M + o.N) * o.K + (double)(o.offP - o.offA);
    o.item0 = (int)items;
    items += (int64_t)o.ntm * o.ntn * o.ks * (o.both ? 1 : 2);
    o.scale0[0] = (int)scale[0];
    o.scale0[1] = (int)scale[1];
    scale[0] += oz_scale_blocks(o.M, o.a_ks, o.K);
    scale[1] += oz_scale_blocks(o.N, o.b_ks, o.K);
    o.atom0[0] = h->atoms[0];
    o.atom0[1] = h->atoms[1];
    o.grp0[0] = h->groups[0];
    o.grp0[1] = h->groups[1];
    groups[0] += (int64_t)o.ntm * (OZ_BM / 8);
    groups[1] += (int64_t)o.ntn * (OZ_BN / 8);
    h->groups[0] = (int)groups[0];
    h->groups[1] = (int)groups[1];
    h->atoms[0] += (int64_t)o.ntm * (OZ_BM / 8) * o.nkb;
    h->atoms[1] += (int64_t)o.ntn * (OZ_BN / 8) * o.nkb;
    o.fin0 = (int)fin;
    fin += cdiv((int64_t)o.M * o.N, 256);
  }
  for (int i = 0; i < n; ++i) {  // the exponent fields are the buffer's end
    t[i].offE = (int64_t)(off + sizeof(int) * (size_t)rows);
    rows += t[i].M + t[i].N;
  }
  off += ws_round(sizeof(int) * (size_t)rows);
  if (items > INT32_MAX || scale[0] + scale[1] > INT32_MAX || groups[0] + groups[1] > INT32_MAX || fin > INT32_MAX) return 0;
  h->items = (int)items;
  h->scale_blocks[0] = (int)scale[0];
  h->scale_blocks[1] = (int)scale[1];
  h->fin_blocks = (int)fin;
  *flop = wflop;
  *bytes = wbytes;
  return off;
}
template <int CAP>
unsigned oz_scale_grid(const OzTasks<CAP>& T) {
  return (unsigned)(((T.h.sides & 1) ? T.h.scale_blocks[0] : 0) + ((T.h.sides & 2) ? T.h.scale_blocks[1] : 0));
}
template <int CAP>
unsigned oz_slice_grid(const OzTasks<CAP>& T) {
  const int64_t a = ((T.h.sides & 1) ? T.h.atoms[0] : 0) + ((T.h.sides & 2) ? T.h.atoms[1] : 0);
  return (unsigned)std::min<int64_t>(cdiv(a, 8), 152 * 16);
}
template <int CAP>
unsigned oz_prep_grid(const OzTasks<CAP>& T) {
  return (unsigned)(((T.h.sides & 1) ? T.h.groups[0] : 0) + ((T.h.sides & 2) ? T.h.groups[1] : 0));
}
// Whether the scales and slices of t[0..n) take one launch (k_oz_prep): rows of one CTA's
// share of K, and no more row groups than about two CTAs for every SM; more of them are
// bound by throughput, and the separate slice kernel keeps more loads in flight.  Whole
// products, separate / one launch, us: 256 x 256 x 128 63.5 / 58.6, 1024 x 1024 x 64 86.7 / 81.8,
// 1024 x 1024 x 512 189.7 / 186.1 (256 groups), 1024 x 4096 x 256 333.6 / 333.8 (640),
// 2048 x 2048 x 512 536.7 / 539.1 (512), 256 x 8192 x 512 356.5 / 364.2 (1056).
bool oz_one_prep(const OzHead& h, const OzTask* t, int n, int sm) {
  if (h.groups[0] + h.groups[1] > 2 * sm) return false;
  for (int i = 0; i < n; ++i)
    if (t[i].K > OZ_SCALE_K) return false;
  return true;
}

bool oz_capturing(Ctx* c) {
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(c->stream, &st) != cudaSuccess) {
    cudaGetLastError();  // the legacy stream beside another stream's capture
    return false;
  }
  return st != cudaStreamCaptureStatusNone;
}

// products tk[0..n) in one set of launches; slices and partial sums live in the context's own
// buffer, grown between calls, never inside a capture; a buffer that a captured graph refers to
// is kept until the context goes.  OZ_NOROOM: the buffer cannot grow as needed
template <int CAP>
int oz_launch(Ctx* c, const GemmTask* const* tk, int n, int sm) {
  OzTasks<CAP> T;
  double flop = 0, bytes = 0;
  const size_t need = oz_layout(tk, n, sm, &T.h, T.t, &flop, &bytes);
  if (!need) return set_err(c, TNT_E_UNSUPPORTED, "FP64 products too large for one launch");
  T.h.status = c->d_status;
  const bool capture = oz_capturing(c);
  if (capture && need > c->oz_cap) return OZ_NOROOM;
  if (capture) c->oz_captured = true;
  if (need > c->oz_cap) {
    TNT_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
    if (c->oz_captured) c->oz_kept.push_back(c->oz_buf);
    else dev_free(c->dalloc, c->oz_buf);
    c->oz_captured = false;
    c->oz_buf = nullptr;
    c->oz_cap = 0;
    if (dev_alloc(c->dalloc, &c->oz_buf, need) != 0) return OZ_NOROOM;
    c->oz_cap = need;
  }
  T.h.buf = (uint8_t*)c->oz_buf;
  {
    ProfScope ps(c, "oz_slice", bytes);
    if (oz_one_prep(T.h, T.t, n, sm)) {
      k_oz_prep<CAP><<<oz_prep_grid(T), 256, 0, c->stream>>>(T);
      c->launches++;
    } else {
      for (int i = 0; i < n; ++i) {  // maxima combined from several CTAs start from zero
        const OzTask& o = T.t[i];
        if (o.K > OZ_SCALE_K && (o.a_ks != 1 || o.b_ks != 1))
          TNT_CUDA_TRY(c, cudaMemsetAsync(T.h.buf + o.offE, 0, sizeof(int) * (size_t)(o.M + o.N), c->stream));
      }
      k_oz_scale<CAP><<<oz_scale_grid(T), 256, 0, c->stream>>>(T);
      k_oz_slice<CAP><<<oz_slice_grid(T), 256, 0, c->stream>>>(T);
      c->launches += 2;
    }
  }
  {
    ProfScope ps(c, "oz_gemm", flop);
    k_oz_gemm<CAP><<<(unsigned)std::min(T.h.items, sm), OZ_THREADS, OZ_SMEM, c->stream>>>(T);
    k_oz_finish<CAP><<<(unsigned)std::min(T.h.fin_blocks, 152 * 8), 256, 0, c->stream>>>(T);
  }
  c->launches += 2;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}
}  // namespace

// ---------------------------------------------------------------- repeated products
size_t oz_plan_bytes(Ctx* c, const std::vector<GemmTask>& tasks) {
  if (tasks.empty()) return 0;
  const int sm = c->nsm;
  std::vector<const GemmTask*> tk;
  for (const GemmTask& t : tasks) tk.push_back(&t);
  std::vector<OzTask> t(tasks.size());
  OzHead h;
  double f, b;
  const size_t need = oz_layout(tk.data(), (int)tk.size(), sm, &h, t.data(), &f, &b);
  return need ? need + ws_round(sizeof(OzTask) * t.size()) : 0;
}

int oz_plan_build(Ctx* c, const std::vector<GemmTask>& tasks, int fixed_sides, OzPlan* p) {
  TNT_TRY(oz_setup(c));
  const int sm = c->nsm;
  std::vector<const GemmTask*> tk;
  for (const GemmTask& t : tasks) {
    tk.push_back(&t);
    if (t.g.K > OZ_SCALE_K && (t.g.a_cs != 1 || t.g.b_rs != 1))
      return set_err(c, TNT_E_UNSUPPORTED, "planned FP64 product with a strided K of %lld", (long long)t.g.K);
  }
  std::vector<OzTask> t(tasks.size());
  static_assert(sizeof(OzTasks<0>) <= sizeof(p->args), "the plan's argument block holds the kernels' argument");
  OzTasks<0> T;
  double f, b;
  const size_t need = oz_layout(tk.data(), (int)tk.size(), sm, &T.h, t.data(), &f, &b);
  uint8_t* buf = (uint8_t*)ws_alloc(c, need);
  OzTask* dt = (OzTask*)ws_alloc(c, ws_round(sizeof(OzTask) * t.size()));
  if (!need || !buf || !dt) return set_err(c, TNT_E_ALLOC, "scratch exhausted (planned FP64 products)");
  TNT_TRY(to_device(c, dt, t.data(), sizeof(OzTask) * t.size()));
  T.h.buf = buf;
  T.h.status = c->d_status;
  T.t = dt;
  const bool one = oz_one_prep(T.h, t.data(), (int)t.size(), sm);
  auto inputs = [&](OzNode* node) {  // the launches that read the operands of T.h.sides
    if (one) {
      node[0] = OzNode{(void*)k_oz_prep<0>, oz_prep_grid(T), 256, 0};
      return 1;
    }
    node[0] = OzNode{(void*)k_oz_scale<0>, oz_scale_grid(T), 256, 0};
    node[1] = OzNode{(void*)k_oz_slice<0>, oz_slice_grid(T), 256, 0};
    return 2;
  };
  p->fixed = 0;
  if (fixed_sides) {
    T.h.sides = fixed_sides;
    p->fixed = inputs(p->fix);
    memcpy(p->fix_args, &T, sizeof(T));
  }
  T.h.sides = 3 & ~fixed_sides;
  memcpy(p->args, &T, sizeof(T));
  p->flop = f;
  p->inputs = inputs(p->node);
  p->node[p->inputs] = OzNode{(void*)k_oz_gemm<0>, (unsigned)std::min(T.h.items, sm), OZ_THREADS, OZ_SMEM};
  p->node[p->inputs + 1] = OzNode{(void*)k_oz_finish<0>, (unsigned)std::min(T.h.fin_blocks, 152 * 8), 256, 0};
  p->nodes = p->inputs + 2;
  return TNT_OK;
}

int oz_plan_fix(Ctx* c, OzPlan& p) {
  void* args[] = {p.fix_args};
  for (int i = 0; i < p.fixed; ++i) {
    const OzNode& n = p.fix[i];
    TNT_CUDA_TRY(c, cudaLaunchKernel(n.fn, dim3(n.grid), dim3(n.block), args, n.smem, c->stream));
    c->launches++;
  }
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

void oz_plan_args(const OzPlan& p, const z* add_b, void* out) {
  OzTasks<0> T;
  memcpy(&T, p.args, sizeof(T));
  T.h.add_b = (int64_t)(intptr_t)add_b;
  memcpy(out, &T, sizeof(T));
}

int oz_plan_run(Ctx* c, const OzPlan& p, const z* add_b) {
  alignas(16) unsigned char a[sizeof(p.args)];
  oz_plan_args(p, add_b, a);
  void* args[] = {a};
  for (int i = 0; i < p.nodes; ++i) {
    const OzNode& n = p.node[i];
    TNT_CUDA_TRY(c, cudaLaunchKernel(n.fn, dim3(n.grid), dim3(n.block), args, n.smem, c->stream));
    c->launches++;
  }
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int ozgemm(Ctx* c, const ZGemm& g) {
  TNT_TRY(oz_setup(c));
  const int sm = c->nsm;
  const GemmTask t{g, 0, 0};
  const GemmTask* p = &t;
  return oz_launch<1>(c, &p, 1, sm);
}

// The products of `tasks` (alpha = 1, beta = 0, batch = 1; independent of one another) with as
// few launches as their number allows.  They go to the slice kernels together when their
// FP64 tiles, dealt to the SMs, would take longer than the slice launches' 30 us (the rule of
// ozgemm_eligible for the whole set); products with a side below 16 stay on FP64 units.
int zgemm_tasks(Ctx* c, const std::vector<GemmTask>& tasks) {
  TNT_TRY(oz_setup(c));
  const int sm = c->nsm;
  double rounds = 0, longest = 0;
  for (const GemmTask& t : tasks) {
    const double k = (double)t.g.K;
    rounds += k * (double)cdiv(t.g.M, 16) * (double)cdiv(t.g.N, 16) * (t.herm ? 0.5 : 1.0) / sm;
    longest = std::max(longest, fma_rounds(c, k, 0.0));
  }
  const bool slices = c->oz_mode != 0 && std::max(rounds, longest) >= 110.0;
  std::vector<const GemmTask*> oz, fma;
  for (const GemmTask& t : tasks) {
    const ZGemm& g = t.g;
    if (g.M <= 0 || g.N <= 0) continue;
    if (c->oz_mode == 0 && cdiv(g.M, 64) * cdiv(g.N, 64) >= sm && (!t.herm || g.c_rs == g.M)) {
      // FP64 units alone: a large product fills the GPU by itself with 64 x 64 tiles
      ZGemm h = g;
      h.lower_only = t.herm;
      if (t.sub) {
        h.alpha = zmk(-1, 0);
        h.beta = zmk(1, 0);
      }
      TNT_TRY(zgemm(c, h));
      if (t.herm) TNT_TRY(herm_mirror(c, g.C, g.M));
      continue;
    }
    if (g.K <= 0 || g.batch != 1) return set_err(c, TNT_E_INVALID, "grouped FP64 product with K = %lld", (long long)g.K);
    (slices && std::min(g.M, std::min(g.N, g.K)) >= 16 && std::max(g.M, g.N) < (1LL << 31) ? oz : fma).push_back(&t);
  }
  // longest items first
  std::stable_sort(oz.begin(), oz.end(), [](const GemmTask* a, const GemmTask* b) { return a->g.K > b->g.K; });
  for (size_t i = 0; i < oz.size(); i += OZ_MAXT) {
    const int n = (int)std::min<size_t>(OZ_MAXT, oz.size() - i);
    const int r = n == 1 ? oz_launch<1>(c, oz.data() + i, 1, sm) : oz_launch<OZ_MAXT>(c, oz.data() + i, n, sm);
    if (r == OZ_NOROOM) fma.insert(fma.end(), oz.begin() + (long)i, oz.begin() + (long)i + n);
    else TNT_TRY(r);
  }
  return fma.empty() ? TNT_OK : zgemm_fma_tasks(c, fma.data(), (int)fma.size());
}

}  // namespace tnt
