// Leading eigenpairs of a large Hermitian FP64 matrix (the Gram matrix of one charge block
// of the truncated SVD, App. B.1.2): k largest eigenvalues and their eigenvectors.
//
//   1. Householder reduction to real tridiagonal form G = Q T Q^H: for each column j the
//      reflector H_j = I - tau v v^H maps the part below the diagonal to beta e_1 (beta
//      real), and the trailing block is updated as A <- H_j^H A H_j through
//      p = tau A v, w = p - (tau/2)(p^H v) v, A <- A - v w^H - w v^H.
//   2. Multisection on Sturm counts of T for eigenvalues n-1, ..., n-k (one warp each),
//      to full precision.
//   3. Inverse iteration on T - lambda_i I (pivoted tridiagonal LU, three sweeps), each
//      eigenvalue its own shift; the iterates of a cluster of eigenvalues closer than
//      1e3 eps |T| are re-orthogonalised against the cluster's earlier vectors.
//   4. Back-transformation U = H_0 H_1 ... H_{n-2} Y.
//   5. Two Newton-Schulz steps U <- U (3 I - U^H U) / 2 in FP64 to restore orthonormality
//      lost to close eigenvalues.
// All arithmetic is FP64.  The cost is O(n^3) once, against O(sweeps n^3) for a Jacobi
// eigensolver.  Blocks of up to 1216 rows go through every stage together (heig_blocks).
#include <algorithm>
#include <cmath>

#include "heff_plan.cuh"
#include "f32conv.cuh"
#include "tri_deal.cuh"

namespace tnt {

namespace {
constexpr double EPS = 2.220446049250313e-16;
constexpr double SPLIT_TOL = 1e3 * EPS;  // negligible against |T| (k_split)

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ int hi_exp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// x -= a conj(b) as four FMAs (the FP64 pipe is the bottleneck of these kernels on GB300)
__device__ __forceinline__ void zsub_mul_conj(z& x, z a, z b) {
  x.x = fma(-a.x, b.x, fma(-a.y, b.y, x.x));
  x.y = fma(-a.y, b.x, fma(a.x, b.y, x.y));
}

// block-wide sum; valid in every thread on return.  The warp sums are combined by a
// butterfly over one warp's lanes (every warp the same order, so every thread gets the
// same bits): five FP64 adds per thread, where a loop over the warp sums in every thread
// cost one add per warp per thread (the FP64 pipe is the scarce unit on GB300)
__device__ double block_sum_all(double v, double* sh) {
  v = warp_sum_d(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

// block-wide maximum; valid in every thread on return
__device__ double block_max_all(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r = fmax(r, __shfl_xor_sync(0xffffffffu, r, o));
  return r;
}

// ---------------------------------------------------------------- persistent reduction
// All columns in one cooperative launch, one grid barrier per column.  Entering column j
// every block holds the reflector (v_j, tau_j) in its workspace and p_j = tau_j T_j v_j is
// complete in global memory (T_j: the trailing block after column j-1).  Then:
//   every block: s_j = p_j^H v_j (from the per-block partials, same order everywhere),
//     w_j = p_j - (tau_j s_j / 2) v_j, the updated row j+1 of A, and from it reflector
//     j+1 (block 0 also stores it for the back-transformation);
//   each warp: for the rows it owns, T <- T - v_j w_j^H - w_j v_j^H, and in the same pass
//     the row's entry of p_{j+1} = tau_{j+1} T_{j+1} v_{j+1} and its share of s_{j+1};
//   grid barrier.
// Row g belongs to block g mod nb and, within it, to warp (g / nb) mod 16, so the rows
// left at every column stay spread over all blocks.  p and the
// partial sums are double-buffered by column parity.  The grid barrier spins on a
// generation counter with a %globaltimer limit; if any wait expires, an abort flag makes
// every block leave at its next barrier.
struct TriArgs {
  z* G;
  int64_t n;
  z* Hv;
  z* tau;
  double* d;
  double* e;
  z* p;                // 2 x n: p of even / odd columns
  z* part;             // 2 x nb partial sums of p^H v
  unsigned* bar;       // [0] arrivals, [1] generation
  int* abort_flag;
  int* status;
  z* gws;              // per-block workspace (4 n) when n exceeds the shared cache
};

__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// returns false if the CTA must stop (a wait expired here or elsewhere)
__device__ bool grid_barrier(const TriArgs& a) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile unsigned* gen = a.bar + 1;
    const unsigned g = *gen;
    __threadfence();
    const unsigned arrived = atomicAdd(a.bar, 1u);
    int ok = 1;
    if (arrived == gridDim.x - 1) {
      a.bar[0] = 0;
      __threadfence();
      atomicAdd(a.bar + 1, 1u);
    } else {
      const uint64_t t0 = gtime();
      while (*gen == g) {
        if (*(volatile int*)a.abort_flag) { ok = 0; break; }
        if (gtime() - t0 > 2000000000ull) {
          atomicOr(a.status, 2);
          atomicExch(a.abort_flag, 1);
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    if (*(volatile int*)a.abort_flag) ok = 0;
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Block-wide sum, valid in thread 0 only (warp 0 combines the warp sums).
__device__ double block_sum0(double v, double* sh) {
  v = warp_sum_d(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0;
  if (w == 0) r = warp_sum_d((l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0);
  return r;
}

// Householder reflector of a row x (the part below the diagonal of a column of a Hermitian
// matrix, conjugated): alpha = conj(x_0), xn2 = sum_{r>0} |x_r|^2.  H = I - tau v v^H with
// v = (1, conj(x_r) scale, ...) maps conj(x) to beta e_1, beta real.  Computed by one thread:
// a full-block FP64 square root and three divisions cost more FP64-pipe issue slots on
// GB300 than the vector work of a short column.
// A row whose squares sum to less than 2^-900 counts as zero (no reflection): the blocks are
// scaled to a largest entry of about one, and a matrix of low rank leaves trailing blocks of
// 1e-16, 1e-32, 1e-48, ... whose squares would underflow after a few columns.
struct Refl {
  z tau, scale;
  double beta;
};
__device__ __forceinline__ bool refl_none(z alpha, double xn2) {
  return hi_exp(fma(alpha.x, alpha.x, fma(alpha.y, alpha.y, xn2))) < 1023 - 900 || (xn2 == 0.0 && alpha.y == 0.0);
}
__device__ Refl refl_params(z alpha, double xn2, bool empty) {
  Refl R;
  if (empty || refl_none(alpha, xn2)) {
    R.tau = zmk(0, 0);
    R.beta = alpha.x;
    R.scale = zmk(0, 0);
  } else {
    const double nrm = sqrt(alpha.x * alpha.x + alpha.y * alpha.y + xn2);
    R.beta = alpha.x >= 0 ? -nrm : nrm;
    R.tau = zmk((R.beta - alpha.x) / R.beta, -alpha.y / R.beta);
    const z den = zmk(alpha.x - R.beta, alpha.y);  // scale = 1 / (alpha - beta)
    const double dd = den.x * den.x + den.y * den.y;
    R.scale = zmk(den.x / dd, -den.y / dd);
  }
  return R;
}

// Reflector from x_r = conj(row[r]), r < m (row already in the workspace): v (length m,
// v[0] = 1), tau, beta with H^H x = beta e_1.  Every thread of the block returns the same
// tau and beta.
__device__ void make_reflector(const z* row, int64_t m, z* v, z* tau_out, double* beta_out,
                               double* sh) {
  __shared__ Refl s_refl;
  double acc = 0;
  for (int64_t r = 1 + threadIdx.x; r < m; r += blockDim.x) {
    const z x = row[r];
    acc = fma(x.x, x.x, fma(x.y, x.y, acc));
  }
  acc = block_sum0(acc, sh);
  if (threadIdx.x == 0) s_refl = refl_params(m > 0 ? zconj(row[0]) : zmk(0, 0), acc, m == 0);
  __syncthreads();
  const Refl R = s_refl;
  for (int64_t r = threadIdx.x; r < m; r += blockDim.x)
    v[r] = (r == 0) ? zmk(1, 0) : zmul(zconj(row[r]), R.scale);
  *tau_out = R.tau;
  *beta_out = R.beta;
  __syncthreads();
}

constexpr int TRI_THREADS = 512;
constexpr int TRI_WARPS = TRI_THREADS / 32;
constexpr int64_t TRI_CACHE = 2048;  // workspace in shared memory up to this n

__global__ void __launch_bounds__(TRI_THREADS) k_tridiag_persistent(TriArgs a) {
  extern __shared__ z sm_tri[];
  __shared__ double sh[32];
  __shared__ double shr[TRI_WARPS], shi[TRI_WARPS];
  __shared__ z s_cf;
  const int64_t n = a.n;
  const int nb = gridDim.x, b = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // row g belongs to block g mod nb, warp (g / nb) mod TRI_WARPS: consecutive rows land on
  // different SMs, so every SM's FP64 units share each column's work
  const int64_t nwarps = (int64_t)nb * TRI_WARPS, own0 = (int64_t)b + (int64_t)nb * warp;
  z* ws = (n <= TRI_CACHE) ? sm_tri : a.gws + (int64_t)b * 4 * n;
  z* sv = ws;           // v_j
  z* sw = ws + n;       // w_j
  z* srow = ws + 2 * n; // updated row j+1
  z* sv2 = ws + 3 * n;  // v_{j+1}
  // reflector 0 from row 0, and p_0 = tau_0 T_0 v_0 over the owned rows
  z t;
  double beta;
  {
    const int64_t m = n - 1;
    for (int64_t c = threadIdx.x; c < m; c += blockDim.x) srow[c] = __ldcg(a.G + 1 + c);
    __syncthreads();
    make_reflector(srow, m, sv, &t, &beta, sh);
    if (b == 0) {
      for (int64_t c = threadIdx.x; c < m; c += blockDim.x) a.Hv[c] = sv[c];
      if (threadIdx.x == 0) {
        a.tau[0] = t;
        a.d[0] = __ldcg(a.G).x;
        if (m > 0) a.e[0] = beta;
      }
    }
    double pr = 0, pi = 0;
    for (int64_t g = own0; g < n; g += nwarps) {  // global row g = local row g - 1
      if (g < 1) continue;
      const z* row = a.G + g * n + 1;
      double sr = 0, si = 0;
#pragma unroll 4
      for (int64_t c = lane; c < m; c += 32) {
        const z x = __ldcg(row + c), y = sv[c];
        sr = fma(x.x, y.x, fma(-x.y, y.y, sr));
        si = fma(x.x, y.y, fma(x.y, y.x, si));
      }
      sr = warp_sum_d(sr);
      si = warp_sum_d(si);
      if (lane == 0) {
        const z pv = zmul(t, zmk(sr, si));
        a.p[g - 1] = pv;
        const z vr = sv[g - 1];
        pr += pv.x * vr.x + pv.y * vr.y;
        pi += pv.x * vr.y - pv.y * vr.x;
      }
    }
    if (lane == 0) { shr[warp] = pr; shi[warp] = pi; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double sa = 0, sb = 0;
      for (int q = 0; q < TRI_WARPS; ++q) { sa += shr[q]; sb += shi[q]; }
      a.part[b] = zmk(sa, sb);
    }
  }
  for (int64_t j = 0; j + 1 < n; ++j) {
    if (!grid_barrier(a)) return;
    const int64_t m = n - j - 1;          // size of T_j (local rows/cols 0..m-1 = global j+1..)
    const z* pj = a.p + (j & 1) * n;
    z* pn = a.p + ((j + 1) & 1) * n;
    const z* partj = a.part + (j & 1) * nb;
    z* partn = a.part + ((j + 1) & 1) * nb;
    if (warp == 0) {  // the nb partials, loaded by 32 lanes at once and summed by shuffles
      double sa = 0, sb = 0;
      for (int q = lane; q < nb; q += 32) {
        const z pq = __ldcg(partj + q);
        sa += pq.x;
        sb += pq.y;
      }
      sa = warp_sum_d(sa);
      sb = warp_sum_d(sb);
      if (lane == 0) {
        const z ts = zmul(t, zmk(sa, sb));
        s_cf = zmk(-0.5 * ts.x, -0.5 * ts.y);
      }
    }
    __syncthreads();
    const z cf = s_cf;
    for (int64_t c = threadIdx.x; c < m; c += blockDim.x) {
      const z pv = __ldcg(pj + c), vv = sv[c];
      sw[c] = zmk(fma(cf.x, vv.x, fma(-cf.y, vv.y, pv.x)), fma(cf.x, vv.y, fma(cf.y, vv.x, pv.y)));
    }
    __syncthreads();
    // updated row j+1 (local row 0), then reflector j+1 from its entries 1..m-1
    const z v0 = sv[0], w0 = sw[0];
    {
      const z* row = a.G + (j + 1) * n + j + 1;
      for (int64_t c = threadIdx.x; c < m; c += blockDim.x) {
        z x = __ldcg(row + c);
        zsub_mul_conj(x, v0, sw[c]);
        zsub_mul_conj(x, w0, sv[c]);
        srow[c] = x;
      }
    }
    __syncthreads();
    const int64_t m2 = m - 1;  // size of T_{j+1}
    z t2;
    make_reflector(srow + 1, m2, sv2, &t2, &beta, sh);
    if (b == 0) {
      for (int64_t c = threadIdx.x; c < m2; c += blockDim.x) a.Hv[(j + 1) * n + c] = sv2[c];
      if (threadIdx.x == 0) {
        a.tau[j + 1] = t2;
        a.d[j + 1] = srow[0].x;
        if (m2 > 0) a.e[j + 1] = beta;
      }
    }
    // owned rows r >= 1 of T_j: update, and dot with v_{j+1} for p_{j+1}
    double pr = 0, pi = 0;
    for (int64_t g = own0 + ((j + 2 > own0) ? ((j + 2 - own0 + nwarps - 1) / nwarps) * nwarps : 0);
         g < n; g += nwarps) {
      const int64_t r = g - (j + 1);  // local row in T_j
      z* row = a.G + g * n + j + 1;
      const z vr = sv[r], wr = sw[r];
      double sr = 0, si = 0;
#pragma unroll 4
      for (int64_t c = 1 + lane; c < m; c += 32) {
        z x = __ldcg(row + c);
        zsub_mul_conj(x, vr, sw[c]);
        zsub_mul_conj(x, wr, sv[c]);
        row[c] = x;
        const z q = sv2[c - 1];
        sr = fma(x.x, q.x, fma(-x.y, q.y, sr));
        si = fma(x.x, q.y, fma(x.y, q.x, si));
      }
      sr = warp_sum_d(sr);
      si = warp_sum_d(si);
      if (lane == 0) {
        const z pv = zmul(t2, zmk(sr, si));
        pn[r - 1] = pv;
        const z vv = sv2[r - 1];
        pr += pv.x * vv.x + pv.y * vv.y;
        pi += pv.x * vv.y - pv.y * vv.x;
      }
    }
    if (lane == 0) { shr[warp] = pr; shi[warp] = pi; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double sa = 0, sb = 0;
      for (int q = 0; q < TRI_WARPS; ++q) { sa += shr[q]; sb += shi[q]; }
      partn[b] = zmk(sa, sb);
    }
    // v_{j+1} becomes the current reflector
    for (int64_t c = threadIdx.x; c < m2; c += blockDim.x) sv[c] = sv2[c];
    t = t2;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- rows in shared memory
// The same column-by-column reduction for blocks of n <= TRI_ROWS_NMAX rows, several blocks
// (the charge blocks of one truncated SVD) in one cooperative launch.  A block gets a group of
// CTAs in proportion to its work (tri_deal); row g of the block belongs to CTA g mod nb of
// its group and stays in that CTA's shared memory for the whole reduction: the trailing
// update and the product with the next reflector touch shared memory only, and per column
// the global memory carries p (n entries), the per-CTA partial sums and the one row that is
// the source of the next reflector.  The group's own barrier, once per column; a group of
// one CTA needs none, and keeps p in shared memory.
// Reflector j is v_j = (1, conj(x_c) s_j for c > j+1) with x row j of the updated matrix
// and s_j its scale; p_j = tau_j T_j v_j is formed without v_j as
// tau_j (T(g, j+1) + s_j sum_{c > j+1} T(g, c) conj(x_c)), so that the reflector's scalars are
// computed by a warp of their own (TRI_WARPS) while the others update the rows.
// K_j = v_j^H T_j v_j is real, and with it w_j = p_j + c_j v_j, c_j = -|tau_j|^2 K_j / 2, and the
// next source row x'(c) = T_j(j+1, c) - conj(p_j(c)) - (p_j(j+1) + 2 c_j) conj(v_j(c)).
// Entering column j every CTA holds x (in sx, the entry j+1 zeroed), tau_j and s_j, and p_j
// with the per-CTA parts of K_j is in global memory:
//   the scalar warp: c_j from the parts; the others: v_j(c), and x'(c) but for its c_j term;
//   x' (into sx) and w_j, with the sum of |x'(c)|^2 over c > j+2;
//   the scalar warp: reflector j+1; the others, the CTA's rows g > j+1 of T_j, flattened over
//     (row, column) and split evenly over the warps: T <- T - v_j w_j^H - w_j v_j^H and
//     sum_c T(g, c) conj(x'(c)); the owner of row j+2 also stores it in global memory;
//   warp 0: p_{j+1}(g) for the CTA's rows and its part of K_{j+1};
//   group barrier.
// Reflector j replaces row j of the block in global memory (columns 0 .. n-j-2), the layout
// the back-transformation reads: no CTA reads row j after its barrier j.
// A Gram matrix is positive semidefinite, so its trailing block is bounded by that block's
// trace.  Once an entry and the trace of what follows are both at most SPLIT_TOL / 4 times the
// largest entry, so is the coupling (the square root of their product), and the reduction
// stops: the rest is the negligible range that k_split takes off (d = e = 0, no reflectors).
// What the entries found so far leave of the whole trace is only the hint: where many entries
// are of the largest one's size that difference is off by thousands of eps of them (its own
// rounding, and the drift of the trace under the reflectors).  At a hint the group sums the
// trailing diagonal as it stands, with a barrier of its own (as a rule once per block).  A 5 : 1
// block of a centre move has a fifth of its columns left to do, theta of a truncated state about half.
// Vectors are indexed by row of the block.  Per column a CTA spends 16 FP64 operations per
// trailing entry on the shared vectors and 12 per entry of its rows: that work bounds large
// blocks (two operations per SM and clock); small ones are bound by the sequence of about 60
// dependent FP64 instructions at 100 to 200 clocks each, the barrier and the loads.  The
// barrier is one release-add and an acquire-poll of a counter (an atomic with its old value, a
// generation word and a timer read per poll took 9000 to 13000 clocks); square root and
// reciprocal are Newton steps from FP32 seeds (library calls: 5000 clocks).
// Before, blocks of up to 256 rows were reduced on one SM each (a 200-row block: 3.8 ms,
// the FP64 pipe of one SM) and larger ones one after the other across the GPU (500 rows
// 4.5 ms, 1024 rows 24.4 ms).
static_assert(TRI_WARPS == 16, "the flattened row split divides by 16 with shifts");
constexpr int TRI_VEC = 3;              // vector entries per thread
static_assert(TRI_ROWS_NMAX <= TRI_VEC * TRI_THREADS, "every vector entry has a thread");
constexpr int TRI_GTHREADS = TRI_THREADS + 32;

struct TriBlk {
  z* G;          // the block, n x n; its rows become the reflectors
  z* tau;
  double* d;
  double* e;
  z* p;          // 2 x n: p of even / odd columns
  double* part;  // 2 x nb parts of v^H T v (even / odd columns), then nb of the trailing trace
  int n, c0, nb; // CTAs [c0, c0 + nb)
};
struct TriGroup {
  int nblk;
  unsigned* bar;   // 32 words per block: arrivals (words 0 and 16, zero before the launch)
  int* status;
  TriBlk b[TRI_MAXB];
};

// Barrier j of a group of nb CTAs on its counter `word` (0: columns, 16: hints): each adds one
// (release: its threads' stores before the CTA barrier are visible to whoever sees the sum) and
// waits until all have.  false: the wait expired, the CTA must stop (and so will the others of
// its group).
__device__ bool group_barrier(const TriGroup& t, int grp, int nb, int j, int word) {
  __shared__ int s_ok;
  __syncthreads();
  if (nb == 1) return true;
  if (threadIdx.x == 0) {
    unsigned* bar = t.bar + 32 * grp + word;
    const unsigned want = (unsigned)nb * (unsigned)(j + 1);
    unsigned seen;
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(bar), "r"(1u) : "memory");
    uint64_t t0 = 0;
    for (unsigned polls = 0;; ++polls) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      if (seen >= want) break;
      if ((polls & 1023u) == 1023u) {
        const uint64_t now = gtime();
        if (!t0) t0 = now;
        if (now - t0 > 2000000000ull) {
          atomicOr(t.status, 2);
          ok = 0;
          break;
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// (a, b) summed over the warp with five FP64 adds (the two sums share each step); every
// lane returns both
__device__ __forceinline__ void warp_sum_pair(double& a, double& b) {
  const bool up = (threadIdx.x & 16) != 0;
  double v = (up ? b : a) + __shfl_xor_sync(0xffffffffu, up ? a : b, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  a = __shfl_sync(0xffffffffu, v, 0);
  b = __shfl_sync(0xffffffffu, v, 16);
}

// four values summed over the warp with seven FP64 adds: lane l returns the total of s[l & 3]
__device__ __forceinline__ double warp_sum4(double* s) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int o = 2; o >= 1; o >>= 1) {
    const bool up = (l & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double give = up ? s[i] : s[i + o], keep = up ? s[i + o] : s[i];
      s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double r = s[0];
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  return r;
}

struct GroupRefl {
  z tau, scale;
  double beta, c;  // c = -|tau|^2 / 2
};
struct RowsShared {
  double b4[TRI_WARPS][4];       // few rows: per warp, sum T conj(x) of its two row segments
  z q0[TRI_RMAX], q1[TRI_RMAX];  // many rows: per row, from its start / its second warp
  double nrm[TRI_WARPS];         // per warp: sum |x|^2
  GroupRefl rf[2];               // reflectors of even / odd columns
  z alpha;
  double cf, part;
  double left, dmax;             // what is left of the trace; largest diagonal entry so far
  double entry, tailp;           // the column's diagonal entry; at a hint: one CTA's trace
  int done, hints;               // the rest of the block may be, and then is, negligible; hints so far
};

// Reflector parameters (refl_params) by one warp
__device__ GroupRefl refl_warp(z alpha, double xn2, bool empty) {
  GroupRefl R;
  R.tau = R.scale = zmk(0, 0);
  R.beta = alpha.x;
  R.c = 0;
  if (empty || refl_none(alpha, xn2)) return R;
  const double s = fma(alpha.x, alpha.x, fma(alpha.y, alpha.y, xn2));
  double nrm, inv;
  if (hi_exp(s) < 1946) {  // not below 2^-900
    inv = rsqrt_newton(s);
    nrm = s * inv;
  } else {
    nrm = sqrt(s);
    inv = 1.0 / nrm;
  }
  R.beta = alpha.x >= 0 ? -nrm : nrm;
  const z den = zmk(alpha.x - R.beta, alpha.y);  // scale = 1 / (alpha - beta), |den| >= nrm
  const double dd = fma(den.x, den.x, den.y * den.y);
  const double rd = hi_exp(dd) < 1946 ? rcp_newton(dd) : 1.0 / dd;  // dd >= s
  const double rb = alpha.x >= 0 ? inv : -inv;  // -1 / beta
  R.tau = zmk(den.x * rb, alpha.y * rb);
  R.scale = zmk(den.x * rd, -den.y * rd);
  R.c = -0.5 * fma(R.tau.x, R.tau.x, R.tau.y * R.tau.y);
  return R;
}

// one segment of a row: T(g, c) -= v(g) conj(w(c)) + w(g) conj(v(c)) (with UPD; also to gout)
// for c0 <= c < c1, and the lane's sum of T(g, c) conj(x(c)) to sr, si
template <bool UPD>
__device__ __forceinline__ void row_segment(z* rw, int c0, int c1, z vr, z wr, const z* v, const z* w, const z* x,
                                            z* gout, double& sr, double& si) {
  sr = si = 0;
#pragma unroll 2
  for (int c = c0 + (threadIdx.x & 31); c < c1; c += 32) {
    z t = rw[c];
    if (UPD) {
      zsub_mul_conj(t, vr, w[c]);
      zsub_mul_conj(t, wr, v[c]);
      rw[c] = t;
      if (gout) gout[c] = t;
    }
    const z y = x[c];  // t conj(y)
    sr = fma(t.x, y.x, fma(t.y, y.y, sr));
    si = fma(t.y, y.x, fma(-t.x, y.y, si));
  }
}

// The row warps a column's work is split over, as a power of two: at least 64 entries each
// (their sums are added one after the other afterwards, at 150 to 200 clocks an addition).
__device__ __forceinline__ int row_warps_log2(unsigned total) {
  return total >= 1024u ? 4 : total >= 512u ? 3 : total >= 256u ? 2 : total >= 128u ? 1 : 0;
}
// Rows g >= lo of this CTA (rows[i] = row b + nb i, R of them) over W = 2^s row warps: warp w
// covers [f0, f1) of the flattened (row, column) range, f0 = ract L w / W, and starts in row
// floor(ract w / W) (exact: floor(floor(x) / L) = floor(x / L)).  Fewer than W rows: a warp
// meets at most two rows, a row several warps.  W and more: a row meets at most two warps.
template <bool UPD>
__device__ void rows_update(z* rows, int R, int b, int nb, int n, int lo, const z* v, const z* w, const z* x,
                            z* grow, RowsShared& S) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = (lo > b) ? (lo - b + nb - 1) / nb : 0;
  const int ract = R - i0 > 0 ? R - i0 : 0;
  const unsigned L = (unsigned)(n - lo), total = (unsigned)ract * L;
  const int ws = row_warps_log2(total);
  if (warp >> ws) return;
  const unsigned f0 = (total * (unsigned)warp) >> ws, f1 = (total * (unsigned)(warp + 1)) >> ws;
  const int r0 = (ract * warp) >> ws;
  if (ract < (1 << ws)) {
    double s4[4] = {0, 0, 0, 0};
#pragma unroll
    for (int seg = 0; seg < 2; ++seg) {
      const int ri = r0 + seg;  // row of this segment
      const int s0 = (seg == 0) ? (int)f0 - ri * (int)L : 0;
      const int s1 = min((int)L, (int)f1 - ri * (int)L);
      if (ri < ract && s0 < s1) {
        const int i = i0 + ri, g = b + nb * i;
        row_segment<UPD>(rows + (int64_t)i * n, lo + s0, lo + s1, UPD ? v[g] : zmk(0, 0), UPD ? w[g] : zmk(0, 0), v,
                         w, x, (UPD && g == lo) ? grow : nullptr, s4[2 * seg], s4[2 * seg + 1]);
      }
    }
    if (f0 < f1) {
      const double s = warp_sum4(s4);
      if (lane < 4) S.b4[warp][lane] = s;
    }
    return;
  }
  for (int ri = r0; ri < ract && (unsigned)ri * L < f1; ++ri) {
    const int s0 = max(0, (int)f0 - ri * (int)L), s1 = min((int)L, (int)f1 - ri * (int)L);
    if (s0 >= s1) continue;
    const int i = i0 + ri, g = b + nb * i;
    double sr, si;
    row_segment<UPD>(rows + (int64_t)i * n, lo + s0, lo + s1, UPD ? v[g] : zmk(0, 0), UPD ? w[g] : zmk(0, 0), v, w, x,
                     (UPD && g == lo) ? grow : nullptr, sr, si);
    warp_sum_pair(sr, si);
    if (lane == 0) {
      if (s0 == 0) S.q0[ri] = zmk(sr, si);
      else S.q1[ri] = zmk(sr, si);
    }
  }
}

// Warp 0 after rows_update, with reflector rf of the column whose trailing block starts at lo:
// q = T(g, lo) + s sum and p(g) = tau q for the CTA's rows g >= lo into pout, the CTA's part
// of v^H T v, the sum of Re(conj(v(g)) q) (v(lo) = 1, v(c) = conj(x(c)) s), into *partout.
__device__ void rows_finish(const z* rows, int R, int b, int nb, int n, int lo, const z* x, const GroupRefl& rf,
                            z* pout, double* partout, RowsShared& S) {
  const int lane = threadIdx.x & 31;
  const int i0 = (lo > b) ? (lo - b + nb - 1) / nb : 0;
  const int ract = R - i0 > 0 ? R - i0 : 0;
  const unsigned L = (unsigned)(n - lo), total = (unsigned)ract * L;
  const int ws = row_warps_log2(total);
  double part = 0;
  for (int r = lane; r < ract; r += 32) {
    const int g = b + nb * (i0 + r);
    const z t0 = rows[(int64_t)(i0 + r) * n + lo];
    const z vg = (g == lo) ? zmk(1, 0) : zmul(zconj(x[g]), rf.scale);
    double sr = 0, si = 0;
    if (ract < (1 << ws)) {
      for (int w = 0; w < (1 << ws); ++w) {  // the warps whose range meets row r, in order
        const unsigned f0 = (total * (unsigned)w) >> ws, f1 = (total * (unsigned)(w + 1)) >> ws;
        const int r0 = (ract * w) >> ws;
        if (f0 < f1 && r0 == r) {
          sr += S.b4[w][0];
          si += S.b4[w][1];
        } else if (f0 < f1 && r0 + 1 == r && f1 > (unsigned)r * L) {
          sr += S.b4[w][2];
          si += S.b4[w][3];
        }
      }
    } else {
      sr = S.q0[r].x;
      si = S.q0[r].y;
      // the first warp boundary after the row's start, if it falls inside the row
      const unsigned rl = (unsigned)r * L, w = (((rl + 1u) << ws) + total - 1u) / total;
      if (w < (1u << ws) && ((total * w) >> ws) < rl + L) {
        sr += S.q1[r].x;
        si += S.q1[r].y;
      }
    }
    const z q = zmk(fma(rf.scale.x, sr, fma(-rf.scale.y, si, t0.x)), fma(rf.scale.x, si, fma(rf.scale.y, sr, t0.y)));
    pout[g] = zmul(rf.tau, q);
    part = fma(vg.x, q.x, fma(vg.y, q.y, part));
  }
  for (int o = ract > 16 ? 16 : ract > 8 ? 8 : ract > 4 ? 4 : ract > 2 ? 2 : ract > 1 ? 1 : 0; o > 0; o >>= 1)
    part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) *partout = part;
}

// the 16 row warps' sums of |x|^2, in every lane of the scalar warp
__device__ __forceinline__ double nrm_total(const RowsShared& S) {
  const int lane = threadIdx.x & 31;
  double nr = S.nrm[lane & 15];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) nr += __shfl_xor_sync(0xffffffffu, nr, o);
  return nr;
}

// Column j of a group's CTA after its scalars and vectors: reflector j+1, the update of the rows,
// p_{j+1} and the CTA's part of K_{j+1}
__device__ __forceinline__ void column_update(const TriBlk& a, z* rows, int R, int b, int j, const z* sv, const z* sw,
                                              const z* sx, z* pn, double* partn, RowsShared& S) {
  const int n = a.n, nb = a.nb, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool empty = n - j - 2 <= 0;  // length of reflector j+1
  if (warp == TRI_WARPS) {
    const GroupRefl rf = refl_warp(empty ? zmk(0, 0) : S.alpha, nrm_total(S), empty);
    if (lane == 0) {
      S.rf[(j + 1) & 1] = rf;
      if (b == 0) {
        a.tau[j + 1] = rf.tau;
        if (!empty) a.e[j + 1] = rf.beta;
      }
    }
  } else {
    rows_update<true>(rows, R, b, nb, n, j + 2, sv, sw, sx, nb == 1 ? nullptr : a.G + (int64_t)(j + 2) * n, S);
  }
  __syncthreads();
  if (warp == 0) rows_finish(rows, R, b, nb, n, j + 2, sx, S.rf[(j + 1) & 1], pn, partn, S);
}

// Column j at a hint: the trace of rows j+1 and on, summed over the group before the column's update,
// which leaves it, says whether the reduction ends.  If not, the column goes on as usual.
// true: the CTA is done (or the wait expired).  A call outside the loop over the columns, which
// keeps its registers so: a flat block of 1024 / 300 / 100 rows takes 19.56 / 2.46 / 0.69 ms, with
// the sum inside the loop 19.74 / 2.50 / 0.71, without any (the hint alone) 19.28 / 2.46 / 0.71.
__device__ __noinline__ bool hint_column(const TriGroup& T, int grp, z* rows, z* sv, int j, RowsShared& S) {
  const TriBlk& a = T.b[grp];
  const int n = a.n, nb = a.nb, b = (int)blockIdx.x - a.c0, R = (b < n) ? (n - b + nb - 1) / nb : 0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool one = nb == 1;
  double* tails = one ? &S.tailp : a.part + 2 * nb;
  if (warp == 0) {
    double tr = 0;
    for (int i = lane; i < R; i += 32)
      if (b + nb * i > j) tr += rows[(int64_t)i * n + b + nb * i].x;
    tr = warp_sum_d(tr);
    if (lane == 0) tails[b] = tr;
  }
  if (!group_barrier(T, grp, nb, S.hints, 16)) return true;
  if (warp == 0) {
    double tr = 0;
    for (int q = lane; q < nb; q += 32) tr += one ? tails[q] : __ldcg(tails + q);
    tr = warp_sum_d(tr);
    if (lane == 0) {
      S.done = tr - S.entry <= 0.25 * SPLIT_TOL * S.dmax;
      ++S.hints;
    }
  }
  __syncthreads();
  if (!S.done) {
    column_update(a, rows, R, b, j, sv, sv + n, sv + 2 * n, one ? sv + 3 * n : a.p + ((j + 1) & 1) * n,
                  one ? &S.part : a.part + ((j + 1) & 1) * nb + b, S);
    return false;
  }
  if (b == 0)
    for (int i = j + 1 + tid; i < n; i += TRI_GTHREADS) {
      a.tau[i] = zmk(0, 0);
      a.e[i] = 0.0;
      if (i > j + 1) a.d[i] = 0.0;
    }
  return true;
}

__global__ void __launch_bounds__(TRI_GTHREADS, 1) k_tridiag_group(const __grid_constant__ TriGroup T) {
  extern __shared__ z sm_tri[];
  __shared__ RowsShared S;
  int grp = 0;
  while (grp + 1 < T.nblk && T.b[grp + 1].c0 <= (int)blockIdx.x) ++grp;
  const TriBlk& a = T.b[grp];
  const int n = a.n, nb = a.nb, b = (int)blockIdx.x - a.c0;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const bool scalar = warp == TRI_WARPS;  // the warp of the scalars
  const int rmax = (n + nb - 1) / nb;
  const int R = (b < n) ? (n - b + nb - 1) / nb : 0;
  z* rows = sm_tri;
  z* sv = rows + (int64_t)rmax * n;  // v_j
  z* sw = sv + n;                    // w_j
  z* sx = sw + n;                    // x of the next reflector (its first entry zeroed)
  z* sp = sx + n;                    // p, in a group of one CTA
  const bool one = nb == 1;
  if (scalar) {  // the trace, in the same order in every CTA
    double s = 0;
    for (int i = lane; i < n; i += 32) s += __ldcg(a.G + (int64_t)i * n + i).x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const double d0 = __ldcg(a.G).x;
      S.left = s - d0;
      S.dmax = d0;
      S.done = S.hints = 0;
    }
  }
  for (int i = 0; i < R; ++i) {
    const z* src = a.G + (b + (int64_t)nb * i) * n;
    for (int c = tid; c < n; c += TRI_GTHREADS) rows[(int64_t)i * n + c] = __ldcg(src + c);
  }
  {  // reflector 0 from row 0 (columns 1..n-1), and p_0
    double acc = 0;
    if (!scalar) {
#pragma unroll
      for (int k = 0; k < TRI_VEC; ++k) {
        const int c = 1 + tid + k * TRI_THREADS;
        if (c < n) {
          const z xc = __ldcg(a.G + c);
          if (c == 1) S.alpha = zconj(xc);
          else acc = fma(xc.x, xc.x, fma(xc.y, xc.y, acc));
          sx[c] = (c == 1) ? zmk(0, 0) : xc;
        }
      }
      acc = warp_sum_d(acc);
      if (lane == 0) S.nrm[warp] = acc;
    }
    __syncthreads();
    if (scalar) {
      const GroupRefl rf = refl_warp(n > 1 ? S.alpha : zmk(0, 0), nrm_total(S), n < 2);
      if (lane == 0) {
        S.rf[0] = rf;
        if (b == 0) {
          a.tau[0] = rf.tau;
          a.d[0] = __ldcg(a.G).x;
          if (n > 1) a.e[0] = rf.beta;
        }
      }
    } else {
      rows_update<false>(rows, R, b, nb, n, 1, sv, sw, sx, nullptr, S);
    }
    __syncthreads();
    if (warp == 0) rows_finish(rows, R, b, nb, n, 1, sx, S.rf[0], one ? sp : a.p, one ? &S.part : a.part + b, S);
  }
  for (int j = 0;; ++j) {  // (a hint leaves the inner loop, which then goes on)
    for (; j + 1 < n; ++j) {
      if (!group_barrier(T, grp, nb, j, 0)) return;
      const z* pj = one ? sp : a.p + (j & 1) * n;
      z* pn = one ? sp : a.p + ((j + 1) & 1) * n;
      const double* partj = one ? &S.part : a.part + (j & 1) * nb;
      double* partn = one ? &S.part : a.part + ((j + 1) & 1) * nb + b;
      const z* grow = one ? rows + (int64_t)(j + 1) * n : a.G + (int64_t)(j + 1) * n;
      z pc[TRI_VEC], tc[TRI_VEC], vc[TRI_VEC];
      if (scalar) {  // c_j: the group's parts of K, by 32 lanes at once
        double s[5], k = 0;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          const int q = lane + 32 * i;
          s[i] = q < nb ? (one ? partj[q] : __ldcg(partj + q)) : 0.0;
        }
        k = s[0];
        if (nb > 64) k = (s[0] + s[1]) + ((s[2] + s[3]) + s[4]);
        else if (nb > 32) k = s[0] + s[1];
        for (int q = lane + 160; q < nb; q += 32) k += __ldcg(partj + q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
        if (lane == 0) S.cf = S.rf[j & 1].c * k;
      } else {
        const z scale = S.rf[j & 1].scale;
        const z p1 = one ? pj[j + 1] : __ldcg(pj + j + 1);
#pragma unroll
        for (int k = 0; k < TRI_VEC; ++k) {
          const int c = j + 1 + tid + k * TRI_THREADS;
          if (c < n) {
            pc[k] = one ? pj[c] : __ldcg(pj + c);
            tc[k] = one ? grow[c] : __ldcg(grow + c);
          }
        }
#pragma unroll
        for (int k = 0; k < TRI_VEC; ++k) {  // v_j, written out for the back-transformation
          const int c = j + 1 + tid + k * TRI_THREADS;
          if (c < n) {
            vc[k] = (c == j + 1) ? zmk(1, 0) : zmul(zconj(sx[c]), scale);
            sv[c] = vc[k];
            if (b == 0) a.G[(int64_t)j * n + (c - j - 1)] = vc[k];
            tc[k].x -= pc[k].x;  // T(j+1, c) - conj(p(c)) - p(j+1) conj(v(c))
            tc[k].y += pc[k].y;
            zsub_mul_conj(tc[k], p1, vc[k]);
          }
        }
      }
      __syncthreads();
      if (!scalar) {
        const double cf = S.cf, cf2 = 2.0 * cf;
        double acc = 0;
#pragma unroll
        for (int k = 0; k < TRI_VEC; ++k) {
          const int c = j + 1 + tid + k * TRI_THREADS;
          if (c < n) {
            const z xn = zmk(fma(-cf2, vc[k].x, tc[k].x), fma(cf2, vc[k].y, tc[k].y));
            sw[c] = zmk(fma(cf, vc[k].x, pc[k].x), fma(cf, vc[k].y, pc[k].y));
            if (c == j + 1) {  // thread 0
              if (b == 0) a.d[j + 1] = xn.x;
              const double left = S.left - xn.x, top = fmax(S.dmax, xn.x), tol = 0.25 * SPLIT_TOL * top;
              S.left = left;
              S.dmax = top;
              S.done = xn.x <= tol && left <= tol;
              S.entry = xn.x;
            } else if (c == j + 2) {
              S.alpha = zconj(xn);
              sx[c] = zmk(0, 0);
            } else {
              acc = fma(xn.x, xn.x, fma(xn.y, xn.y, acc));
              sx[c] = xn;
            }
          }
        }
        if (j + 1 + 32 * warp < n) acc = warp_sum_d(acc);
        if (lane == 0) S.nrm[warp] = acc;
      }
      __syncthreads();
      if (S.done) break;  // the same in every CTA of the group
      column_update(a, rows, R, b, j, sv, sw, sx, pn, partn, S);
    }
    if (j + 1 >= n || hint_column(T, grp, rows, sv, j, S)) return;
  }
}

// Reflectors as the columns of V: column i of a panel starting at reflector j0 is element
// (rho, i) = Hv[j0 n + i (n - 1) + rho], which for rho < i falls in the part of row j0 + i - 1
// right of its reflector.  That part is zeroed here, and so is a reflector with tau = 0.
struct CleanBlk {
  z* G;
  z* tau;  // a zero becomes 1 (the inverse of T's diagonal entry)
  int n;
};
struct CleanGroup {
  int nblk;
  CleanBlk b[TRI_MAXB];
};
__global__ void __launch_bounds__(256) k_clean_reflectors(const __grid_constant__ CleanGroup T) {
  const CleanBlk& a = T.b[blockIdx.y];
  for (int j = blockIdx.x; j + 1 < a.n; j += gridDim.x) {
    const z t = a.tau[j];
    const bool none = t.x == 0.0 && t.y == 0.0;
    z* row = a.G + (int64_t)j * a.n;
    for (int c = (none ? 0 : a.n - j - 1) + threadIdx.x; c < a.n; c += 256) row[c] = zmk(0, 0);
    __syncthreads();
    if (none && threadIdx.x == 0) a.tau[j] = zmk(1, 0);
  }
}

// T of a panel of reflectors, H_0 ... H_{b-1} = I - V T V^H: T^-1 is the strict upper triangle
// of V^H V plus diag(1 / tau).  One CTA per diagonal sub-block of up to WY_SUB reflectors,
// four threads per column of T: T(i, i) = tau_i, then T(r, i) = -tau_r sum_q S(r, q) T(q, i)
// upwards.  The off-diagonal blocks, -T_1 S_12 T_2, come from products (32 -> 64 -> 128).
constexpr int WY_SUB = 32, WY_PANEL = 4 * WY_SUB;
struct WySub {
  const z* S;   // the sub-block's diagonal block of V^H V
  const z* tau;
  z* T;         // zero before
  int n, ld;
};
__global__ void __launch_bounds__(4 * WY_SUB) k_wy_t(const WySub* __restrict__ subs) {
  __shared__ z s_t[WY_SUB][WY_SUB + 1];  // column i in s_t[i]
  const WySub a = subs[blockIdx.x];
  const int i = threadIdx.x >> 2, part = threadIdx.x & 3;
  if (part == 0 && i < a.n) s_t[i][i] = a.tau[i];
  for (int r = a.n - 2; r >= 0; --r) {
    __syncthreads();
    double sr = 0, si = 0;
    if (i > r && i < a.n)
      for (int q = r + 1 + part; q <= i; q += 4) {
        const z s = a.S[(int64_t)r * a.ld + q], t = s_t[i][q];
        sr = fma(s.x, t.x, fma(-s.y, t.y, sr));
        si = fma(s.x, t.y, fma(s.y, t.x, si));
      }
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      sr += __shfl_xor_sync(0xffffffffu, sr, o);
      si += __shfl_xor_sync(0xffffffffu, si, o);
    }
    if (part == 0 && i > r && i < a.n) {
      const z t = a.tau[r];
      s_t[i][r] = zmk(fma(-t.x, sr, t.y * si), fma(-t.x, si, -t.y * sr));
    }
  }
  __syncthreads();
  if (i < a.n)
    for (int r = part; r <= i; r += 4) a.T[(int64_t)r * a.ld + i] = s_t[i][r];
}

// Number of eigenvalues of T below x from the signs of the leading principal minors
// p_i = det(T_i - x I), p_i = (d_i - x) p_{i-1} - e_{i-1}^2 p_{i-2} (Sturm sequence of the
// characteristic polynomials, Givens' bisection): a sign change between p_{i-1} and p_i
// marks an eigenvalue below x.  Each step is one subtraction and two products; rounding in
// a step perturbs only d_i and e_{i-1} by O(eps) relative, so the count is that of a
// matrix within O(eps |T|).  Division-free: a full-warp FP64 division costs several times
// the FP64-pipe issue slots of these three operations.  The pair (p_{i-1}, p_i) is
// rescaled by an exact power of two when its exponent leaves [-400, 400]; e2 = e^2; signs and
// exponents are read as integers.  A zero minor is replaced by 2^-60 |p_{i-1}| with the
// sign opposite to its predecessor (the tiny negative pivot of the ratio form).  det(T - x I)
// itself is *last times 2^*lastex.
__device__ int sturm_lt(const double* d, const double* e2, int64_t n, double x, double* last,
                        int* lastex) {
  double pm2 = 1.0, pm1 = d[0] - x;
  int neg_prev = 0;  // sign of p_0 = 1
  int cnt = 0, total = 0;
  if (pm1 == 0.0) pm1 = -0x1p-60;
  int neg = __double2hiint(pm1) < 0;
  cnt += neg != neg_prev;
  neg_prev = neg;
  for (int64_t i = 1; i < n; ++i) {
    double p = fma(d[i] - x, pm1, -e2[i - 1] * pm2);
    if (((__double2hiint(p) << 1) | __double2loint(p)) == 0) p = neg_prev ? 0x1p-60 * fabs(pm1) : -0x1p-60 * fabs(pm1);
    neg = __double2hiint(p) < 0;
    cnt += neg != neg_prev;
    neg_prev = neg;
    pm2 = pm1;
    pm1 = p;
    const int ex = hi_exp(p);
    if (ex > 1023 + 400 || ex < 1023 - 400) {  // keep the pair in range: exact scaling
      const double f = __hiloint2double((2046 - ex) << 20, 0);
      pm1 *= f;
      pm2 *= f;
      total += ex - 1023;
    }
  }
  *last = pm1;
  *lastex = total;
  return cnt;
}
// the same in FP32, for T scaled to entries of at most about one
__device__ int sturm_lt32(const float* d, const float* e2, int64_t n, float x) {
  float pm2 = 1.f, pm1 = d[0] - x;
  int neg_prev = 0, cnt = 0;
  if (pm1 == 0.f) pm1 = -0x1p-30f;
  int neg = __float_as_int(pm1) < 0;
  cnt += neg != neg_prev;
  neg_prev = neg;
  for (int64_t i = 1; i < n; ++i) {
    float p = fmaf(d[i] - x, pm1, -e2[i - 1] * pm2);
    if (p == 0.f) p = neg_prev ? 0x1p-30f * fabsf(pm1) : -0x1p-30f * fabsf(pm1);
    neg = __float_as_int(p) < 0;
    cnt += neg != neg_prev;
    neg_prev = neg;
    pm2 = pm1;
    pm1 = p;
    const int ex = (__float_as_int(p) >> 23) & 0xff;
    if (ex > 127 + 40 || ex < 127 - 40) {
      const float f = __int_as_float((254 - ex) << 23);
      pm1 *= f;
      pm2 *= f;
    }
  }
  return cnt;
}

// One eigenproblem of the eigen phase, several of which share each launch (the charge
// blocks of one truncated SVD): the tridiagonal T (d, e, tau at off; n entries), its
// reflectors (row j = v_j of Hv at hoff, row stride n), and the k wanted eigenpairs, whose
// eigenvalues sit at ev[evo ..], iterates at Y[yo ..] (n k), first eigenvectors at
// U0[yo ..] (n x k, leading dimension k), inverse-iteration factors at gwork[wo ..] (6 n k).
struct EBlk {
  int64_t n, k;
  int64_t off, hoff, evo, yo, wo;
};

// Split of T at a negligible trailing block (the deflation LAPACK's tridiagonal solvers
// apply at negligible off-diagonals): the longest trailing range [s, n) whose diagonal and
// off-diagonal entries, its coupling e_{s-1} included, are all at most SPLIT_TOL |T|.  A
// rank-deficient Gram block reduces to such a T: once the reflectors have spanned the
// block's range, the trailing matrix is rounding noise (a few eps |T| and more where the
// Gram matrix itself carries the rounding of a long sum); 1e3 eps |T| catches it.  The
// split also absorbs real eigenvalues below that level (singular values under ~5e-7
// sigma_max): the canonical vectors span their subspace exactly, and the truncated SVD
// resolves its singular values in a second pass over that subspace.  The eigenvalues of that range are
// zero to within SPLIT_TOL |T|, and any orthonormal basis of its coordinates is an
// eigenbasis to that accuracy: the canonical vectors e_s, ..., e_{n-1} are taken, exactly
// orthonormal to each other and (zero beyond s) to the iterates of T[0, s), with no
// inverse iteration.  One warp per problem: |T| (Gershgorin) to tnorm, s to nr.
__global__ void k_split(const double* __restrict__ dAll, const double* __restrict__ eAll,
                        const EBlk* __restrict__ blks, double* __restrict__ tnorm,
                        int64_t* __restrict__ nr) {
  const int lane = threadIdx.x & 31;
  const EBlk B = blks[blockIdx.x];
  const int64_t n = B.n;
  const double* d = dAll + B.off;
  const double* e = eAll + B.off;
  double tn = 0;
  for (int64_t r = lane; r < n; r += 32)
    tn = fmax(tn, fabs(d[r]) + (r > 0 ? fabs(e[r - 1]) : 0.0) + (r < n - 1 ? fabs(e[r]) : 0.0));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tn = fmax(tn, __shfl_xor_sync(0xffffffffu, tn, o));
  const double tol = SPLIT_TOL * tn;
  int64_t s = 0;  // one past the last row that is not negligible
  for (int64_t r = lane; r < n; r += 32)
    if (!(fabs(d[r]) <= tol && (r == 0 || fabs(e[r - 1]) <= tol))) s = r + 1;
  s = __reduce_max_sync(0xffffffffu, (int)s);
  if (lane == 0) {
    tnorm[blockIdx.x] = tn;
    nr[blockIdx.x] = s;
  }
}

// eigenvalue of ascending index n-1-i for i < k; ev[i] descending.  One warp per
// eigenvalue: the 32 lanes evaluate Sturm counts at 32 interior points, shrinking the
// bracket 33-fold per step, to full precision.  The values serve only as
// shifts (singular values are taken later as FP64 projection norms), and each SM's few
// FP64 units favour short dependent chains over many of them.  Warp g works on eigenvalue
// eig[g].y of problem eig[g].x, on the leading block T[0, s) of the split; indices from s
// on belong to the negligible block and take its diagonal entry.
// The first four steps, down to 8e-7 of the Gershgorin interval, run on FP32 counts of T
// scaled to that interval: such a count is exact for a matrix within a few FP32 roundings of
// T, so the bracket is widened by 2e-6 of the interval and holds the eigenvalue (FP64 steps
// cost a full FP64-pipe pass over T each, 3 instructions of 64 clocks per row).
// The FP64 steps after the first are guided: where the counts at the bracket's ends differ
// by one, the determinants there change sign, and the line through them meets zero near the
// eigenvalue (off by about bracket^2 / gap).  The 32 points then lie on both sides of that
// estimate at distances width 2^(-1.5 j), j = 0..15: an estimate good to 2^-13 shrinks the
// bracket 8192-fold where even spacing shrinks it 33-fold.  The counts decide in either form,
// so a poor estimate costs that step only, and the next one is evenly spaced.  Three or four
// FP64 steps in place of seven: the launches of a TEBD run at L = 10, chi = 128 took 104 us on
// average with even spacing alone, 77 us guided, and 35 us since small eigenvalues stop at
// half a last bit of |T| too (before, at 4 eps of their own size, up to a dozen steps).
__global__ void __launch_bounds__(32) k_bisect(const double* __restrict__ dAll, const double* __restrict__ eAll,
                         const EBlk* __restrict__ blks, const int2* __restrict__ eig,
                         const int64_t* __restrict__ nrAll, double* __restrict__ evAll) {
  extern __shared__ double sm_bis[];  // e^2 (n), then the FP32 copies (2 n floats)
  const int lane = threadIdx.x & 31;
  const int2 gi = eig[blockIdx.x];
  const EBlk B = blks[gi.x];
  const int64_t n = nrAll[gi.x], i = gi.y;
  const double* d = dAll + B.off;
  const double* e = eAll + B.off;
  if (i >= n) {
    if (lane == 0) evAll[B.evo + i] = d[i];
    return;
  }
  double lo = INFINITY, hi = -INFINITY;
  for (int64_t r = lane; r < n; r += 32) {
    const double er = r < n - 1 ? e[r] : 0.0;
    const double rad = (r > 0 ? fabs(e[r - 1]) : 0.0) + fabs(er);
    lo = fmin(lo, d[r] - rad);
    hi = fmax(hi, d[r] + rad);
    sm_bis[r] = er * er;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const int64_t idx = n - 1 - i;
  const double pad = 2 * EPS * fmax(fabs(lo), fabs(hi)) + 1e-300;
  lo -= pad;
  hi += pad;
  const double w0 = hi - lo;
  if (n > 1 && w0 > 1e-200 && w0 < 1e200) {
    float* fd = (float*)(sm_bis + n);
    float* fe = fd + n;
    const double inv = 1.0 / w0;
    for (int64_t r = lane; r < n; r += 32) {
      fd[r] = (float)((d[r] - lo) * inv);
      fe[r] = (float)(sm_bis[r] * inv * inv);
    }
    __syncwarp();
    float fl = 0.f, fw = 1.f;
    for (int it = 0; it < 4; ++it) {
      const float x = fl + fw * (float)(lane + 1) * (1.f / 33.f);
      const int p = __popc(__ballot_sync(0xffffffffu, sturm_lt32(fd, fe, n, x) <= (int)idx));
      fl += fw * (float)p * (1.f / 33.f);
      fw *= 1.f / 33.f;
    }
    const double l2 = lo + w0 * ((double)fl - 2e-6), h2 = lo + w0 * ((double)fl + (double)fw + 2e-6);
    lo = fmax(lo, l2);
    hi = fmin(hi, h2);
  }
  __syncwarp();
  // full precision, the shifts must resolve close eigenvalues: 4 eps |lambda|, but no more than
  // the last bit of the largest ones, which T itself does not hold
  const double tol = fmax(1e-300, 0.5 * EPS * w0);
  double guess = 0;
  bool guided = false;
  for (int it = 0; it < 64; ++it) {
    const double width = hi - lo;
    if (width <= fmax(tol, 4 * EPS * fmax(fabs(lo), fabs(hi)))) break;
    double x;
    if (guided) {
      const int j = lane < 16 ? lane : 31 - lane;
      const float off = exp2f(-1.5f * (float)j);
      x = fma(lane < 16 ? -width : width, (double)off, guess);
      x = fmin(fmax(x, lo), hi);
    } else {
      x = lo + width * (double)(lane + 1) / 33.0;
    }
    double det;
    int dex;
    const int cnt = sturm_lt(d, sm_bis, n, x, &det, &dex);
    const unsigned below = __ballot_sync(0xffffffffu, cnt <= idx);
    const int p = __popc(below);  // points left of eigenvalue idx (counts are monotone)
    const int pl = p > 0 ? p - 1 : 0, pr = p < 32 ? p : 31;
    const double xl = __shfl_sync(0xffffffffu, x, pl), xr = __shfl_sync(0xffffffffu, x, pr);
    if (p > 0) lo = xl;
    if (p < 32) hi = xr;
    const double nw = hi - lo;
    // the next estimate: lo + (hi - lo) / (1 + |det(hi) / det(lo)|), for a single eigenvalue
    // between, above the level where the determinants are rounding
    const int cl = __shfl_sync(0xffffffffu, cnt, pl), cr = __shfl_sync(0xffffffffu, cnt, pr);
    const int el = __shfl_sync(0xffffffffu, dex + hi_exp(det), pl), er = __shfl_sync(0xffffffffu, dex + hi_exp(det), pr);
    const float m = (float)__hiloint2double((__double2hiint(det) & 0xfffff) | (1023 << 20), 0);  // in [1, 2)
    const float ml = __shfl_sync(0xffffffffu, m, pl), mr = __shfl_sync(0xffffffffu, m, pr);
    const bool slow = guided && nw * 33.0 > width;
    guided = !slow && p > 0 && p < 32 && cl == idx && cr == idx + 1 && nw > 16 * EPS * w0;
    if (guided) {
      const int de = max(-120, min(120, er - el));
      const float q = mr / ml * __int_as_float((127 + de) << 23);
      guess = fma(nw, (double)(1.f / (1.f + q)), lo);
    }
  }
  if (lane == 0) evAll[B.evo + i] = 0.5 * (lo + hi);
}

// Inverse iteration on T - lambda_i I, one shift per eigenvalue.  Eigenvalues whose
// consecutive gaps are below IV_ORTOL |T| = 1e3 eps |T| form a cluster (in a truncated
// SVD's Gram block, typically the rounding-level eigenvalues of a rank-deficient block),
// handled by one CTA: each member's thread factors T - lambda_i I with its
// own eigenvalue as the shift (pivoted tridiagonal LU in the member's slice of gwork), every
// sweep solves all members at once (one thread per member, the recurrences are serial) and
// re-orthogonalises the members in order (classical Gram-Schmidt, twice, then a max-scaled
// normalisation), so coincident eigenvalues still give independent vectors.  With its own
// shift a member's iterate is dominated by its own eigenvector after each solve; a shared
// shift (the cluster head's) left the members far from it dominated by the eigenvector
// just outside the cluster, nearly parallel to that vector's own iterate, and Newton-Schulz
// cannot restore a basis that far from orthonormal.  Outside a cluster an iterate is
// accurate to about eps |T| / gap <= eps / IV_ORTOL, which the final Newton-Schulz steps
// absorb.  The iterates are the output columns Y[i * n ...] themselves.
constexpr int IV_THREADS = 128;
constexpr int IV_CHUNK = 1024;   // earlier cluster members handled per Gram-Schmidt chunk
constexpr double IV_ORTOL = 1e3 * 2.220446049250313e-16;

// |a| as an integer that orders like it (an FP64 comparison holds the FP64 pipe as long as an
// FMA)
__device__ __forceinline__ long long mag(double a) { return __double_as_longlong(a) & 0x7fffffffffffffffll; }
// 1 / p, |p| raised to small
__device__ __forceinline__ double pivot_rcp(double p, double small) {
  if (mag(p) < mag(small)) p = __double2hiint(p) < 0 ? -small : small;
  return hi_exp(p) < 1946 ? rcp_newton(p) : 1.0 / p;
}

// LU with partial pivoting of T - lam I (tridiagonal, textbook); factors in w[0 .. 5n):
// dl, 1 / dm, du, du2 (n each), then n pivot bytes.  Pivots are floored at +-small in both
// branches so that the solve never multiplies by more than 1 / (eps |T|).  The pivots'
// reciprocals are kept (one reciprocal a row instead of one division here and one in each
// of three solves), and the row in progress stays in registers: what counts is the chain
// from one row to the next (the launches of a TEBD run at L = 10, chi = 128: 62 us on average
// with divisions and the rows in memory, 40 us so).
__device__ void iv_factor(const double* __restrict__ d, const double* __restrict__ e, int64_t n, double lam,
                          double small, double* __restrict__ w) {
  double* dl = w;
  double* dm = w + n;
  double* du = w + 2 * n;
  double* du2 = w + 3 * n;
  int8_t* piv = (int8_t*)(w + 4 * n);
  double a = d[0] - lam, u = n > 1 ? e[0] : 0.0, b = u;
  for (int64_t r = 0; r < n - 1; ++r) {
    const double an = d[r + 1] - lam, un = r + 1 < n - 1 ? e[r + 1] : 0.0;
    const bool keep = mag(a) >= mag(b);
    const double inv = pivot_rcp(keep ? a : b, small);
    const double f = (keep ? b : a) * inv;
    const double top = keep ? u : an;
    dm[r] = inv;
    dl[r] = f;
    du[r] = top;
    du2[r] = keep ? 0.0 : un;
    piv[r] = !keep;
    a = fma(-f, top, keep ? an : u);
    u = keep ? un : -f * un;
    b = un;
  }
  dm[n - 1] = pivot_rcp(a, small);
  du[n - 1] = du2[n - 1] = 0.0;
}

// solve (T - lambda I) y = y in place from the factors of iv_factor; the vector is scaled
// down whenever an entry passes 2^500 (compounding pivots of near-degenerate eigenvalues:
// the solution of a scaled system is the scaled solution)
__device__ void iv_solve(double* __restrict__ y, int64_t n, const double* __restrict__ w) {
  const double* dl = w;
  const double* dm = w + n;
  const double* du = w + 2 * n;
  const double* du2 = w + 3 * n;
  const int8_t* piv = (const int8_t*)(w + 4 * n);
  double cur = y[0];
#pragma unroll 4
  for (int64_t r = 0; r < n - 1; ++r) {
    const double nx = y[r + 1], f = dl[r];
    const bool keep = piv[r] == 0;
    y[r] = keep ? cur : nx;
    cur = fma(-f, keep ? cur : nx, keep ? nx : cur);
  }
  y[n - 1] = cur;
  double y1 = 0, y2 = 0;
#pragma unroll 4
  for (int64_t r = n - 1; r >= 0; --r) {
    const double t = fma(-du2[r], y2, y[r]);
    const double v = fma(-du[r], y1, t) * dm[r];
    y[r] = v;
    y2 = y1;
    y1 = v;
    if (hi_exp(v) >= 1023 + 500 && hi_exp(v) < 2047) {  // (nothing to save in an infinity or NaN)
      for (int64_t q = 0; q < n; ++q) y[q] *= 0x1p-500;
      y1 *= 0x1p-500;
      y2 *= 0x1p-500;
    }
  }
}

__global__ void __launch_bounds__(IV_THREADS) k_inviter(
    const double* __restrict__ dAll, const double* __restrict__ eAll,
    const EBlk* __restrict__ blks, const int2* __restrict__ eig,
    const int64_t* __restrict__ nrAll, const double* __restrict__ evAll,
    const double* __restrict__ tnorm, double* __restrict__ gworkAll, double* __restrict__ YAll) {
  __shared__ double sdot[IV_CHUNK];
  __shared__ double sh[32];
  const int2 gi = eig[blockIdx.x];
  const EBlk B = blks[gi.x];
  const int64_t nfull = B.n, i0 = gi.y;
  const int64_t n = nrAll[gi.x];          // the leading block of the split
  const int64_t k = min(B.k, n);          // eigenpairs of the leading block
  const double* d = dAll + B.off;
  const double* e = eAll + B.off;
  const double* ev = evAll + B.evo;
  double* gwork = gworkAll + B.wo;
  double* Y = YAll + B.yo;
  if (i0 >= n) {  // an index of the negligible trailing block: the canonical vector e_i0
    for (int64_t r = threadIdx.x; r < nfull; r += blockDim.x) Y[i0 * nfull + r] = (r == i0) ? 1.0 : 0.0;
    return;
  }
  // |T| floored well inside the normal range: a zero block (a charge sector of theta with
  // no weight) has T = 0, and pivots of eps |T| would then be denormal and the solves
  // would overflow; with the floor its eigenvectors come out as orthonormal start vectors
  const double tn = fmax(tnorm[gi.x], 1e-200);
  const double ortol = IV_ORTOL * tn;
  if (i0 > 0 && ev[i0 - 1] - ev[i0] < ortol) return;  // not the head of its cluster
  int64_t i1 = i0 + 1;
  while (i1 < k && ev[i1 - 1] - ev[i1] < ortol) ++i1;
  const double small = EPS * tn;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nwarps = IV_THREADS / 32;
  // each member's own factorisation, in its own 6n-double slice of gwork
  for (int64_t i = i0 + tid; i < i1; i += IV_THREADS) iv_factor(d, e, n, ev[i], small, gwork + i * (6 * n));
  // deterministic start vectors, free of structure, distinct per member
  for (int64_t i = i0; i < i1; ++i)
    for (int64_t r = tid; r < nfull; r += IV_THREADS) {
      uint32_t h = 2166136261u ^ (uint32_t)(i * 2654435761u) ^ (uint32_t)(r * 2246822519u);
      h *= 16777619u;
      h ^= h >> 15;
      h *= 2654435761u;
      Y[i * nfull + r] = r < n ? 0.5 + (double)(h & 0xffff) / 65536.0 : 0.0;
    }
  __syncthreads();
  for (int sweep = 0; sweep < 3; ++sweep) {
    for (int64_t i = i0 + tid; i < i1; i += IV_THREADS) iv_solve(Y + i * nfull, n, gwork + i * (6 * n));
    __syncthreads();
    for (int64_t i = i0; i < i1; ++i) {
      double* y = Y + i * nfull;
      for (int pass = 0; pass < 2 && i > i0; ++pass) {
        for (int64_t q0 = i0; q0 < i; q0 += IV_CHUNK) {
          const int64_t q1 = min(i, q0 + IV_CHUNK);
          for (int64_t q = q0 + warp; q < q1; q += nwarps) {  // one warp per dot product
            const double* yq = Y + q * nfull;
            double acc = 0;
            for (int64_t r = lane; r < n; r += 32) acc = fma(y[r], yq[r], acc);
            acc = warp_sum_d(acc);
            if (lane == 0) sdot[q - q0] = acc;
          }
          __syncthreads();
          for (int64_t r = tid; r < n; r += IV_THREADS) {
            double v = y[r];
            for (int64_t q = q0; q < q1; ++q) v = fma(-sdot[q - q0], Y[q * nfull + r], v);
            y[r] = v;
          }
          __syncthreads();
        }
      }
      // norm of y / max|y|: the solve can return entries near 1 / (eps |T|), whose squares
      // would overflow
      double mx = 0;
      for (int64_t r = tid; r < n; r += IV_THREADS) mx = fmax(mx, fabs(y[r]));
      mx = block_max_all(mx, sh);
      const double sc = mx > 0 ? 1.0 / mx : 0.0;
      double acc = 0;
      for (int64_t r = tid; r < n; r += IV_THREADS) {
        const double v = y[r] * sc;
        acc = fma(v, v, acc);
      }
      acc = block_sum_all(acc, sh);
      const double inv = acc > 0 ? sc / sqrt(acc) : 0.0;
      for (int64_t r = tid; r < n; r += IV_THREADS) y[r] *= inv;
      __syncthreads();
    }
  }
}

// U[:, i] = H_0 ... H_{n-2} y_i; one CTA per BT_COLS eigenvectors of one problem
// (bt[g] = (problem, first column)), held in shared memory.  Each reflector is read once
// per CTA for all its columns, and the CTA's reduction of the BT_COLS dot products is one
// pass: the FP64 pipe, not the reflector loads or the synchronisation, sets the pace.
constexpr int BT_COLS = 2;
__global__ void __launch_bounds__(256) k_backtransform(const double* __restrict__ YAll,
                                                       const z* __restrict__ HvAll,
                                                       const z* __restrict__ tauAll,
                                                       const EBlk* __restrict__ blks,
                                                       const int2* __restrict__ bt, int cols,
                                                       z* __restrict__ U0All) {
  extern __shared__ double sm_bt[];
  z* y = (z*)sm_bt;  // cols x n (cols = BT_COLS, or 1 when two vectors do not fit)
  __shared__ double shw[8][4];
  __shared__ z s_ts[BT_COLS];
  static_assert(BT_COLS == 2, "four sums per reflector");
  const int2 gb = bt[blockIdx.x];
  const EBlk B = blks[gb.x];
  const int64_t n = B.n, k = B.k, i0 = gb.y;
  const double* Y = YAll + B.yo;
  const z* Hv = HvAll + B.hoff;
  const z* tau = tauAll + B.off;
  z* U = U0All + B.yo;  // n x k, leading dimension k
  const int ncol = (k - i0 < cols) ? (int)(k - i0) : cols;
  for (int q = 0; q < cols; ++q)
    for (int64_t r = threadIdx.x; r < n; r += blockDim.x)
      y[q * n + r] = zmk(q < ncol ? Y[(i0 + q) * n + r] : 0.0, 0);
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t j = n - 2; j >= 0; --j) {
    const z t = tau[j];
    if (t.x == 0.0 && t.y == 0.0) continue;
    const int64_t m = n - j - 1;
    const int nw = (int)(m < 256 ? (m + 31) >> 5 : 8);  // warps that have entries
    const z* v = Hv + j * n;
    double s4[2 * BT_COLS] = {0, 0, 0, 0};  // s = v^H y[j+1:] per column, (re, im) pairs
    for (int64_t r = threadIdx.x; r < m; r += blockDim.x) {
      const z a = v[r];
#pragma unroll
      for (int q = 0; q < BT_COLS; ++q) {
        if (q >= cols) break;
        const z b = y[q * n + j + 1 + r];
        s4[2 * q] = fma(a.x, b.x, fma(a.y, b.y, s4[2 * q]));
        s4[2 * q + 1] = fma(a.x, b.y, fma(-a.y, b.x, s4[2 * q + 1]));
      }
    }
    if (warp < nw) {  // the four sums: seven adds per warp, then a butterfly over the warps' sums
      const double s = warp_sum4(s4);
      if (lane < 4) shw[warp][lane] = s;
    }
    __syncthreads();
    if (warp == 0) {  // lane = (warp's sum, value): lane l holds value l & 3 of warp l >> 2
      double s = (lane >> 2) < nw ? shw[lane >> 2][lane & 3] : 0.0;
      for (int o = 4; o < 4 * nw; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const double im = __shfl_down_sync(0xffffffffu, s, 1);
      if (lane < 4 && (lane & 1) == 0) s_ts[lane >> 1] = zmul(t, zmk(s, im));
    }
    __syncthreads();
    for (int64_t r = threadIdx.x; r < m; r += blockDim.x) {
      const z a = v[r];
#pragma unroll
      for (int q = 0; q < BT_COLS; ++q) {
        if (q >= cols) break;
        z* p = y + q * n + j + 1 + r;
        const z ts = s_ts[q];
        z x = *p;
        x.x = fma(-ts.x, a.x, fma(ts.y, a.y, x.x));
        x.y = fma(-ts.x, a.y, fma(-ts.y, a.x, x.y));
        *p = x;
      }
    }
    __syncthreads();
  }
  for (int q = 0; q < ncol; ++q)
    for (int64_t r = threadIdx.x; r < n; r += blockDim.x) U[r * k + i0 + q] = y[q * n + r];
}

// per eigenproblem: U0 (n x k) = Y as complex numbers (U0 at Y's offset)
__global__ void __launch_bounds__(256) k_complex_cols(const double* __restrict__ YAll, const EBlk* __restrict__ blks,
                                                      z* __restrict__ U0All) {
  __shared__ double s[32][33];
  const EBlk B = blks[blockIdx.y];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t nt = (B.n + 31) / 32, kt = (B.k + 31) / 32;
  for (int64_t w = blockIdx.x; w < nt * kt; w += gridDim.x) {
    const int64_t r0 = (w % nt) * 32, i0 = (w / nt) * 32;
    for (int q = ty; q < 32; q += 8)
      if (i0 + q < B.k && r0 + tx < B.n) s[q][tx] = YAll[B.yo + (i0 + q) * B.n + r0 + tx];
    __syncthreads();
    for (int q = ty; q < 32; q += 8)
      if (r0 + q < B.n && i0 + tx < B.k) U0All[B.yo + (r0 + q) * B.k + i0 + tx] = zmk(s[tx][q], 0);
    __syncthreads();
  }
}

// S <- 1.5 I - 0.5 S for every problem's k x k block (at so[problem])
__global__ void k_ns_coef_all(z* __restrict__ SAll, const EBlk* __restrict__ blks, const int64_t* __restrict__ so) {
  const int64_t k = blks[blockIdx.y].k;
  z* S = SAll + so[blockIdx.y];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < k * k; e += (int64_t)gridDim.x * blockDim.x) {
    z v = zscale(S[e], -0.5);
    if (e / k == e % k) v.x += 1.5;
    S[e] = v;
  }
}

// S <- 1.5 I - 0.5 S  (k x k)
__global__ void k_ns_coef(z* S, int64_t k) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < k * k;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / k, c = e % k;
    z v = zscale(S[e], -0.5);
    if (r == c) v.x += 1.5;
    S[e] = v;
  }
}

__global__ void k_copy_cols(const z* __restrict__ src, int64_t n, int64_t k, int64_t lds,
                            z* __restrict__ dst, int64_t ldd) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * k;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = e / k, c = e % k;
    dst[r * ldd + c] = src[r * lds + c];
  }
}

unsigned gsz(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  if (b < 1) b = 1;
  return (unsigned)b;
}
}  // namespace

constexpr int TRI_MAX_BLOCKS = 1216;

size_t heig_scratch_bound(int64_t n, int64_t k) {
  const size_t gws = n > TRI_CACHE ? ws_round(sizeof(z) * 4 * n * TRI_MAX_BLOCKS) : 0;
  return ws_round(sizeof(z) * n * n) + 3 * ws_round(sizeof(z) * n) + 3 * ws_round(sizeof(double) * n) +
         gws + ws_round(sizeof(z) * 2 * TRI_MAX_BLOCKS) + ws_round(sizeof(double) * k) +
         ws_round(sizeof(double) * (6 * n * k + k)) +
         ws_round(sizeof(double) * n * k) + 2 * ws_round(sizeof(z) * n * k) + 2 * ws_round(sizeof(z) * k * k) +
         (size_t)(1 << 20);
}

constexpr int64_t EIG_NMAX = 8192;  // rows of the largest eigenproblem
constexpr size_t BT_SMEM = 200 * 1024;

// one warp per eigenvalue, the largest problem of n rows
static int launch_bisect(Ctx* c, int64_t n, int64_t kt, const double* d, const double* e, const EBlk* dblk,
                         const int2* deig, const int64_t* nr, double* ev) {
  const size_t smem = sizeof(double) * 2 * (size_t)n;
  TNT_TRY(func_smem(c, (const void*)k_bisect, sizeof(double) * 2 * EIG_NMAX));
  k_bisect<<<(unsigned)kt, 32, smem, c->stream>>>(d, e, dblk, deig, nr, ev);
  return TNT_OK;
}

// Second half of the eigensolve: from the tridiagonal form (d, e) and its reflectors
// (Hv, row j = v_j, row stride n; tau) to the eigenvectors of the k largest eigenvalues
// in U (n x k, leading dimension ldu), descending; ev (device, k).
int heig_finish(Ctx* c, int64_t n, int64_t k, const z* Hv, const z* tau, const double* d,
                const double* e, z* U, int64_t ldu, double* ev) {
  const size_t top = c->ws.top;
  double* tn = (double*)ws_alloc(c, ws_round(sizeof(double)));
  int64_t* nr = (int64_t*)ws_alloc(c, ws_round(sizeof(int64_t)));
  double* work = (double*)ws_alloc(c, ws_round(sizeof(double) * (6 * n * k + k)));
  double* Y = (double*)ws_alloc(c, ws_round(sizeof(double) * n * k));
  z* U0 = (z*)ws_alloc(c, ws_round(sizeof(z) * n * k));
  z* S = (z*)ws_alloc(c, ws_round(sizeof(z) * k * k));
  EBlk* dblk = (EBlk*)ws_alloc(c, ws_round(sizeof(EBlk)));
  int2* deig = (int2*)ws_alloc(c, ws_round(sizeof(int2) * (size_t)(2 * k + 2)));
  if (!tn || !nr || !work || !Y || !U0 || !S || !dblk || !deig) {
    c->ws.top = top;
    return set_err(c, TNT_E_ALLOC, "scratch exhausted (eigenvectors n=%lld k=%lld)", (long long)n, (long long)k);
  }
  cudaStream_t st = c->stream;
  const int cols = (sizeof(z) * n * BT_COLS <= BT_SMEM) ? BT_COLS : 1;
  const int64_t nbt = (k + cols - 1) / cols;
  {  // one problem: the block table and the (eigenvalue, back-transformation) index tables
    const EBlk hb{n, k, 0, 0, 0, 0, 0};
    std::vector<int2> he((size_t)(k + nbt));
    for (int64_t i = 0; i < k; ++i) he[(size_t)i] = make_int2(0, (int)i);
    for (int64_t q = 0; q < nbt; ++q) he[(size_t)(k + q)] = make_int2(0, (int)(q * cols));
    TNT_TRY(to_device(c, dblk, &hb, sizeof(EBlk)));
    TNT_TRY(to_device(c, deig, he.data(), sizeof(int2) * he.size()));
  }
  {
    ProfScope ps(c, "heig_tridiag_eig");
    k_split<<<1, 32, 0, st>>>(d, e, dblk, tn, nr);
    TNT_TRY(launch_bisect(c, n, k, d, e, dblk, deig, nr, ev));
    k_inviter<<<(unsigned)k, IV_THREADS, 0, st>>>(d, e, dblk, deig, nr, ev, tn, work, Y);
    c->launches += 2;
    TNT_CHECK_LAUNCH(c);
  }
  {
    ProfScope ps(c, "heig_backtransform", 8.0 * (double)n * (double)n * (double)k);
    const size_t smem = sizeof(z) * n * cols;
    TNT_TRY(func_smem(c, (const void*)k_backtransform, BT_SMEM));
    k_backtransform<<<(unsigned)nbt, 256, smem, st>>>(Y, Hv, tau, dblk, deig + k, cols, U0);
    c->launches++;
    TNT_CHECK_LAUNCH(c);
  }
  // two Newton-Schulz steps: S = X^H X; S <- 1.5 I - 0.5 S; X <- X S  (U0 -> U -> U0 -> U)
  int r = TNT_OK;
  z* src = U0;
  int64_t lds = k;
  for (int step = 0; step < 2 && r == TNT_OK; ++step) {
    z* dst = (step == 0) ? U : U0;
    const int64_t ldd = (step == 0) ? ldu : k;
    ZGemm g{};
    g.M = k; g.N = k; g.K = n;
    g.A = src; g.a_rs = 1; g.a_cs = lds; g.conj_a = 1;
    g.B = src; g.b_rs = lds; g.b_cs = 1;
    g.C = S; g.c_rs = k;
    g.alpha = zmk(1, 0); g.beta = zmk(0, 0); g.batch = 1;
    r = zgemm(c, g);
    if (r != TNT_OK) break;
    k_ns_coef<<<gsz(k * k), 256, 0, st>>>(S, k);
    c->launches++;
    ZGemm h{};
    h.M = n; h.N = k; h.K = k;
    h.A = src; h.a_rs = lds; h.a_cs = 1;
    h.B = S; h.b_rs = k; h.b_cs = 1;
    h.C = dst; h.c_rs = ldd;
    h.alpha = zmk(1, 0); h.beta = zmk(0, 0); h.batch = 1;
    r = zgemm(c, h);
    src = dst;
    lds = ldd;
  }
  if (r == TNT_OK) {
    k_copy_cols<<<gsz(n * k), 256, 0, st>>>(U0, n, k, k, U, ldu);
    c->launches++;
  }
  c->ws.top = top;
  return r;
}

// G (n x n, row-major, Hermitian, destroyed); U (n x k, leading dimension ldu): the
// eigenvectors of the k largest eigenvalues, in descending order; ev (device, k).
int heig_top(Ctx* c, z* G, int64_t n, int64_t k, z* U, int64_t ldu, double* ev) {
  if (k < 1 || k > n) return set_err(c, TNT_E_INVALID, "heig_top: k = %lld of n = %lld", (long long)k, (long long)n);
  if (n > EIG_NMAX) return set_err(c, TNT_E_UNSUPPORTED, "heig_top: n = %lld > %lld", (long long)n, (long long)EIG_NMAX);
  const size_t top = c->ws.top;
  z* Hv = (z*)ws_alloc(c, ws_round(sizeof(z) * n * n));
  z* tau = (z*)ws_alloc(c, ws_round(sizeof(z) * n));
  z* p = (z*)ws_alloc(c, ws_round(sizeof(z) * 2 * n));
  double* d = (double*)ws_alloc(c, ws_round(sizeof(double) * n));
  double* e = (double*)ws_alloc(c, ws_round(sizeof(double) * n));
  z* part = (z*)ws_alloc(c, ws_round(sizeof(z) * 2 * TRI_MAX_BLOCKS));
  z* gws = n > TRI_CACHE ? (z*)ws_alloc(c, ws_round(sizeof(z) * 4 * n * TRI_MAX_BLOCKS)) : nullptr;
  unsigned* bar = (unsigned*)ws_alloc(c, 256);
  if (!Hv || !tau || !p || !d || !e || !part || !bar || (n > TRI_CACHE && !gws)) {
    c->ws.top = top;
    return set_err(c, TNT_E_ALLOC, "scratch exhausted (heig_top n=%lld k=%lld)", (long long)n, (long long)k);
  }
  cudaStream_t st = c->stream;
  {
    const double nn = (double)n;
    // Hermitian reduction to tridiagonal form: (16/3) n^3 real FLOPs (4 per complex
    // multiply-add, two rank-2 updates of the trailing block and its matrix-vector product)
    ProfScope ps(c, "heig_tridiag", 16.0 / 3.0 * nn * nn * nn);
    const size_t tri_smem = 4 * TRI_CACHE * sizeof(z);
    int occ = 0;
    TNT_TRY(func_smem(c, (const void*)k_tridiag_persistent, tri_smem));
    TNT_CUDA_TRY(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_tridiag_persistent, TRI_THREADS, tri_smem));
    if (occ < 1) return set_err(c, TNT_E_UNSUPPORTED, "tridiagonal kernel cannot be resident");
    TNT_CUDA_TRY(c, cudaMemsetAsync(bar, 0, 256, st));
    TriArgs ta{G, n, Hv, tau, d, e, p, part, (unsigned*)bar, (int*)(bar + 16), c->d_status,
               gws};
    void* args[] = {&ta};
    const int nb = std::min(c->nsm, TRI_MAX_BLOCKS);
    TNT_CUDA_TRY(c, cudaLaunchCooperativeKernel((void*)k_tridiag_persistent, dim3(nb),
                                                dim3(TRI_THREADS), args, tri_smem, st));
    c->launches += 1;
  }
  {
    int h_status = 0;
    TNT_CUDA_TRY(c, cudaMemcpyAsync(&h_status, c->d_status, sizeof(int), cudaMemcpyDeviceToHost, st));
    TNT_CUDA_TRY(c, cudaStreamSynchronize(st));
    if (h_status & 2) {
      cudaMemsetAsync(c->d_status, 0, sizeof(int), st);
      c->ws.top = top;
      return set_err(c, TNT_E_TIMEOUT, "tridiagonal reduction: a grid barrier wait expired");
    }
  }
  const int r = heig_finish(c, n, k, Hv, tau, d, e, U, ldu, ev);
  c->ws.top = top;
  return r;
}

// Above this many rows the panels' products are the faster back-transformation: a set of
// grouped products costs about 35 us, so a 128-reflector panel about 70 and the T factors
// 150 in all, where the one-CTA form takes about 2.5 us per reflector (two vectors a CTA:
// 200 rows 0.5 ms, 500 rows 2.2 ms, 1024 rows and 256 vectors 5.6 ms).
constexpr int64_t WY_MIN = 192;

// U0 <- H_0 ... H_{n-2} Y for the first nl blocks, by panels of WY_PANEL reflectors:
// U0 <- (I - V T V^H) U0 from the last panel to the first, all blocks' panels of one index
// together.  V is read from the reflector rows through its strides (k_clean_reflectors).
static int wy_backtransform(Ctx* c, z* G, const std::vector<SmallEig>& blocks, int nl, const std::vector<EBlk>& he,
                            const std::vector<int64_t>& po, const std::vector<int64_t>& vo,
                            const std::vector<int64_t>& wo, int64_t npan, z* tau, const EBlk* dblk,
                            const WySub* dsub, int nsub, const double* Y, z* U0, z* PS, z* PT, z* PX, z* VT, z* W) {
  cudaStream_t st = c->stream;
  const size_t pp = (size_t)WY_PANEL * WY_PANEL;
  for (int i0 = 0; i0 < nl; i0 += TRI_MAXB) {
    CleanGroup T;
    T.nblk = std::min(TRI_MAXB, nl - i0);
    for (int i = 0; i < T.nblk; ++i) {
      const SmallEig& b = blocks[(size_t)(i0 + i)];
      T.b[i] = CleanBlk{G + b.goff, tau + he[(size_t)(i0 + i)].off, (int)b.n};
    }
    k_clean_reflectors<<<dim3(64, (unsigned)T.nblk), 256, 0, st>>>(T);
    c->launches++;
  }
  k_complex_cols<<<dim3(64, (unsigned)nl), 256, 0, st>>>(Y, dblk, U0);
  TNT_CUDA_TRY(c, cudaMemsetAsync(PT, 0, sizeof(z) * pp * (size_t)npan, st));
  c->launches++;
  auto task = [](int64_t M, int64_t N, int64_t K, const z* A, int64_t a_rs, int64_t a_cs, int conj_a, const z* B,
                 int64_t b_rs, z* C, int64_t c_rs, int herm, int sub) {
    GemmTask t{};
    t.g.batch = 1;
    t.g.alpha = zmk(1, 0);
    t.g.M = M; t.g.N = N; t.g.K = K;
    t.g.A = A; t.g.a_rs = a_rs; t.g.a_cs = a_cs; t.g.conj_a = conj_a;
    t.g.B = B; t.g.b_rs = b_rs; t.g.b_cs = 1;
    t.g.C = C; t.g.c_rs = c_rs;
    t.herm = herm; t.sub = sub;
    return t;
  };
  struct Panel {
    int blk;
    int64_t j0, b, m, s;
  };
  std::vector<Panel> pan;
  int64_t steps = 0;
  for (int i = 0; i < nl; ++i)
    for (int64_t j0 = 0, s = 0; j0 < blocks[(size_t)i].n - 1; j0 += WY_PANEL, ++s) {
      const int64_t n = blocks[(size_t)i].n;
      pan.push_back(Panel{i, j0, std::min<int64_t>(WY_PANEL, n - 1 - j0), n - 1 - j0, s});
      steps = std::max(steps, s + 1);
    }
  std::vector<GemmTask> t;
  for (const Panel& q : pan) {  // V^H V
    const SmallEig& b = blocks[(size_t)q.blk];
    const z* V = G + b.goff + q.j0 * b.n;
    GemmTask g = task(q.b, q.b, q.m, V, b.n - 1, 1, 1, V, 1, PS + pp * (size_t)(po[(size_t)q.blk] + q.s), WY_PANEL, 1, 0);
    g.g.b_cs = b.n - 1;
    t.push_back(g);
  }
  TNT_TRY(zgemm_tasks(c, t));
  k_wy_t<<<(unsigned)nsub, 4 * WY_SUB, 0, st>>>(dsub);
  c->launches++;
  for (int64_t h = WY_SUB; h < WY_PANEL; h *= 2) {  // off-diagonal blocks of T, -T_1 (S_12 T_2)
    std::vector<GemmTask> ta, tb;
    for (const Panel& q : pan) {
      const size_t o = pp * (size_t)(po[(size_t)q.blk] + q.s);
      for (int64_t r = 0; r + h < q.b; r += 2 * h) {
        const int64_t n2 = std::min(h, q.b - r - h);
        const size_t d12 = o + (size_t)(r * WY_PANEL + r + h), d11 = o + (size_t)(r * (WY_PANEL + 1)),
                     d22 = o + (size_t)((r + h) * (WY_PANEL + 1));
        ta.push_back(task(h, n2, n2, PS + d12, WY_PANEL, 1, 0, PT + d22, WY_PANEL, PX + d12, WY_PANEL, 0, 0));
        tb.push_back(task(h, n2, h, PT + d11, WY_PANEL, 1, 0, PX + d12, WY_PANEL, PT + d12, WY_PANEL, 0, 1));
      }
    }
    TNT_TRY(zgemm_tasks(c, ta));
    TNT_TRY(zgemm_tasks(c, tb));
  }
  t.clear();
  for (const Panel& q : pan) {  // V T (m x b, at the panel's columns of the block's n x n area)
    const SmallEig& b = blocks[(size_t)q.blk];
    GemmTask g = task(q.m, q.b, q.b, G + b.goff + q.j0 * b.n, 1, b.n - 1, 0,
                      PT + pp * (size_t)(po[(size_t)q.blk] + q.s), WY_PANEL, VT + vo[(size_t)q.blk] + q.j0, b.n, 0, 0);
    t.push_back(g);
  }
  TNT_TRY(zgemm_tasks(c, t));
  for (int64_t s = steps - 1; s >= 0; --s) {
    std::vector<GemmTask> ta, tb;
    for (const Panel& q : pan) {
      if (q.s != s) continue;
      const SmallEig& b = blocks[(size_t)q.blk];
      z* Us = U0 + he[(size_t)q.blk].yo + (q.j0 + 1) * b.k;
      z* Wq = W + wo[(size_t)q.blk];
      ta.push_back(task(q.b, b.k, q.m, G + b.goff + q.j0 * b.n, b.n - 1, 1, 1, Us, b.k, Wq, b.k, 0, 0));
      tb.push_back(task(q.m, b.k, q.b, VT + vo[(size_t)q.blk] + q.j0, b.n, 1, 0, Wq, b.k, Us, b.k, 0, 1));
    }
    TNT_TRY(zgemm_tasks(c, ta));
    TNT_TRY(zgemm_tasks(c, tb));
  }
  return TNT_OK;
}

size_t heig_blocks_scratch(int64_t n, int64_t k) {
  const size_t nn = (size_t)n, kk = (size_t)k;
  return sizeof(z) * (nn * nn + 2 * nn * kk + kk * kk + 5 * (nn + WY_PANEL) * WY_PANEL + WY_PANEL * kk) +
         sizeof(double) * 7 * nn * kk + 64 * (2 * nn + 4096) + 256 * nn + (size_t)(2 << 20);
}

// Eigenvectors of the k largest eigenvalues of many Hermitian blocks: every stage of the
// eigensolve is one launch (or a few) over all blocks that a group of CTAs can hold (tri_holds:
// 1216 rows on 152 SMs); larger ones take heig_top one after the other.
// blocks[i] = {offset of the n x n block in G (and of its eigenvector columns in U, leading
// dimension n), n, k}; the reflectors replace the blocks' rows.  ev (device) receives the
// eigenvalues: of the blocks that no group holds in the order given, then of the others, largest
// block first.
int heig_blocks(Ctx* c, z* G, const std::vector<SmallEig>& all, z* U, double* ev) {
  if (all.empty()) return TNT_OK;
  const size_t top = c->ws.top;
  cudaStream_t st = c->stream;
  if (!c->tri_smem) {
    int optin = 0;
    cudaFuncAttributes fa{};
    TNT_CUDA_TRY(c, cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device));
    TNT_CUDA_TRY(c, cudaFuncGetAttributes(&fa, k_tridiag_group));
    const size_t most = (size_t)optin - fa.sharedSizeBytes;
    TNT_TRY(func_smem(c, (const void*)k_tridiag_group, most));
    c->tri_smem = most;
  }
  const int nsm = c->nsm;
  const size_t smem_max = c->tri_smem;
  std::vector<SmallEig> blocks;
  for (const SmallEig& b : all) {
    if (b.n < 1 || b.k < 1 || b.k > b.n)
      return set_err(c, TNT_E_INVALID, "eigensolve block n=%lld k=%lld", (long long)b.n, (long long)b.k);
    if (tri_holds(b.n, nsm, smem_max)) {
      blocks.push_back(b);
      continue;
    }
    TNT_TRY(heig_top(c, G + b.goff, b.n, b.k, U + b.goff, b.n, ev));
    ev += b.k;
  }
  if (blocks.empty()) return TNT_OK;
  std::stable_sort(blocks.begin(), blocks.end(), [](const SmallEig& a, const SmallEig& b) { return a.n > b.n; });
  const int nb = (int)blocks.size();
  // large blocks (the first nl): back-transformation by panels of reflectors
  int nl = 0;
  while (nl < nb && blocks[(size_t)nl].n > WY_MIN) ++nl;
  int64_t tot = 0, nk = 0, k2 = 0, nn = 0, npan = 0, kt = 0, kw = 0;
  std::vector<EBlk> he((size_t)nb);
  std::vector<int64_t> so((size_t)nb), vo((size_t)nb), po((size_t)nb), wo2((size_t)nb);
  std::vector<int2> heig, hbt;
  const int cols = BT_COLS;
  for (int i = 0; i < nb; ++i) {
    const SmallEig& b = blocks[(size_t)i];
    he[(size_t)i] = EBlk{b.n, b.k, tot, b.goff, kt, nk, 6 * nk};
    so[(size_t)i] = k2;
    for (int64_t q = 0; q < b.k; ++q) heig.push_back(make_int2(i, (int)q));
    if (i >= nl)
      for (int64_t q = 0; q < b.k; q += cols) hbt.push_back(make_int2(i, (int)q));
    tot += b.n;
    kt += b.k;
    nk += b.n * b.k;
    k2 += b.k * b.k;
    if (i < nl) {
      vo[(size_t)i] = nn;
      po[(size_t)i] = npan;
      wo2[(size_t)i] = kw;
      nn += b.n * b.n;
      npan += (b.n - 2 + WY_PANEL) / WY_PANEL;
      kw += WY_PANEL * b.k;
    }
  }
  const size_t pp = (size_t)WY_PANEL * WY_PANEL;
  double* d = (double*)ws_alloc(c, ws_round(sizeof(double) * tot));
  double* e = (double*)ws_alloc(c, ws_round(sizeof(double) * tot));
  z* tau = (z*)ws_alloc(c, ws_round(sizeof(z) * tot));
  z* p = (z*)ws_alloc(c, ws_round(sizeof(z) * 2 * tot));
  double* part = (double*)ws_alloc(c, ws_round(sizeof(double) * 3 * (size_t)nsm));
  unsigned* bar = (unsigned*)ws_alloc(c, ws_round(sizeof(unsigned) * 32 * TRI_MAXB));
  double* tn = (double*)ws_alloc(c, ws_round(sizeof(double) * nb));
  int64_t* nr = (int64_t*)ws_alloc(c, ws_round(sizeof(int64_t) * nb));
  double* work = (double*)ws_alloc(c, ws_round(sizeof(double) * 6 * nk));
  double* Y = (double*)ws_alloc(c, ws_round(sizeof(double) * nk));
  z* U0 = (z*)ws_alloc(c, ws_round(sizeof(z) * nk));
  z* U1 = (z*)ws_alloc(c, ws_round(sizeof(z) * nk));
  z* S = (z*)ws_alloc(c, ws_round(sizeof(z) * k2));
  // panels of the large blocks: V^H V, T, a product's left half, V T and V^H U
  z* PS = (z*)ws_alloc(c, ws_round(sizeof(z) * pp * (size_t)npan));
  z* PT = (z*)ws_alloc(c, ws_round(sizeof(z) * pp * (size_t)npan));
  z* PX = (z*)ws_alloc(c, ws_round(sizeof(z) * pp * (size_t)npan));
  z* VT = (z*)ws_alloc(c, ws_round(sizeof(z) * (size_t)nn));
  z* W = (z*)ws_alloc(c, ws_round(sizeof(z) * (size_t)kw));
  // one upload: problem table, eigenvalue and back-transformation indices, S offsets, T blocks
  std::vector<WySub> subs;
  for (int i = 0; i < nl; ++i)
    for (int64_t j0 = 0, s = 0; j0 < blocks[(size_t)i].n - 1; j0 += WY_PANEL, ++s)
      for (int64_t q = 0; q < WY_PANEL && j0 + q < blocks[(size_t)i].n - 1; q += WY_SUB) {
        const size_t o = pp * (size_t)(po[(size_t)i] + s) + (size_t)q * (WY_PANEL + 1);
        subs.push_back(WySub{PS + o, tau + he[(size_t)i].off + j0 + q, PT + o,
                             (int)std::min<int64_t>(WY_SUB, blocks[(size_t)i].n - 1 - j0 - q), WY_PANEL});
      }
  const size_t b_blk = ws_round(sizeof(EBlk) * nb), b_eig = ws_round(sizeof(int2) * heig.size()),
               b_bt = ws_round(sizeof(int2) * hbt.size()), b_so = ws_round(sizeof(int64_t) * nb),
               b_sub = ws_round(sizeof(WySub) * subs.size());
  char* tab = (char*)ws_alloc(c, b_blk + b_eig + b_bt + b_so + b_sub + 256);
  if (!d || !e || !tau || !p || !part || !bar || !tn || !nr || !work || !Y || !U0 || !U1 || !S || !tab ||
      (nl > 0 && (!PS || !PT || !PX || !VT || !W))) {
    c->ws.top = top;
    return set_err(c, TNT_E_ALLOC, "scratch exhausted (eigensolves)");
  }
  std::vector<char> host(b_blk + b_eig + b_bt + b_so + b_sub, 0);
  memcpy(host.data(), he.data(), sizeof(EBlk) * nb);
  memcpy(host.data() + b_blk, heig.data(), sizeof(int2) * heig.size());
  if (!hbt.empty()) memcpy(host.data() + b_blk + b_eig, hbt.data(), sizeof(int2) * hbt.size());
  memcpy(host.data() + b_blk + b_eig + b_bt, so.data(), sizeof(int64_t) * nb);
  if (!subs.empty()) memcpy(host.data() + b_blk + b_eig + b_bt + b_so, subs.data(), sizeof(WySub) * subs.size());
  TNT_TRY(to_device(c, tab, host.data(), host.size()));
  const EBlk* dblk = (const EBlk*)tab;
  const int2* deig = (const int2*)(tab + b_blk);
  const int2* dbt = (const int2*)(tab + b_blk + b_eig);
  const int64_t* dso = (const int64_t*)(tab + b_blk + b_eig + b_bt);
  const WySub* dsub = (const WySub*)(tab + b_blk + b_eig + b_bt + b_so);
  {
    double fl = 0;
    for (const SmallEig& b : blocks) fl += 16.0 / 3.0 * (double)b.n * b.n * b.n;
    ProfScope ps(c, "heig_tridiag", fl);
    for (int i0 = 0; i0 < nb;) {
      std::vector<int64_t> ns;
      for (int i = i0; i < nb; ++i) ns.push_back(blocks[(size_t)i].n);
      std::vector<int> q;
      const int cnt = tri_deal(ns, nsm, smem_max, &q);
      if (cnt < 1) {
        c->ws.top = top;
        return set_err(c, TNT_E_UNSUPPORTED, "tridiagonal kernel cannot hold a block of %lld rows", (long long)ns[0]);
      }
      TriGroup T;
      T.nblk = cnt;
      T.bar = bar;
      T.status = c->d_status;
      int ctas = 0;
      size_t smem = 0;
      for (int i = 0; i < cnt; ++i) {
        const SmallEig& b = blocks[(size_t)(i0 + i)];
        const EBlk& E = he[(size_t)(i0 + i)];
        const int64_t rows = (b.n + q[(size_t)i] - 1) / q[(size_t)i];
        T.b[i] = TriBlk{G + b.goff, tau + E.off, d + E.off, e + E.off, p + 2 * E.off, part + 3 * ctas,
                        (int)b.n, ctas, q[(size_t)i]};
        ctas += q[(size_t)i];
        smem = std::max(smem, (size_t)(rows + 3 + (q[(size_t)i] == 1)) * b.n * sizeof(z));
      }
      TNT_CUDA_TRY(c, cudaMemsetAsync(bar, 0, sizeof(unsigned) * 32 * TRI_MAXB, st));
      void* args[] = {&T};
      TNT_CUDA_TRY(c, cudaLaunchCooperativeKernel((void*)k_tridiag_group, dim3((unsigned)ctas), dim3(TRI_GTHREADS),
                                                  args, smem, st));
      c->launches++;
      i0 += cnt;
    }
  }
  {
    ProfScope ps(c, "heig_tridiag_eig");
    k_split<<<(unsigned)nb, 32, 0, st>>>(d, e, dblk, tn, nr);
    TNT_TRY(launch_bisect(c, blocks[0].n, kt, d, e, dblk, deig, nr, ev));
    k_inviter<<<(unsigned)kt, IV_THREADS, 0, st>>>(d, e, dblk, deig, nr, ev, tn, work, Y);
    c->launches += 3;
    TNT_CHECK_LAUNCH(c);
  }
  int r = TNT_OK;
  {
    double fl = 0;
    for (const SmallEig& b : blocks) fl += 8.0 * (double)b.n * b.n * b.k;
    ProfScope ps(c, "heig_backtransform", fl);
    if (!hbt.empty()) {
      const size_t smem = sizeof(z) * (size_t)blocks[(size_t)nl].n * cols;
      TNT_TRY(func_smem(c, (const void*)k_backtransform, BT_SMEM));
      k_backtransform<<<(unsigned)hbt.size(), 256, smem, st>>>(Y, G, tau, dblk, dbt, cols, U0);
      c->launches++;
    }
    if (nl > 0) r = wy_backtransform(c, G, blocks, nl, he, po, vo, wo2, npan, tau, dblk, dsub, (int)subs.size(), Y, U0,
                                     PS, PT, PX, VT, W);
  }
  // two Newton-Schulz steps over all blocks: S = X^H X; S <- 1.5 I - 0.5 S; X <- X S
  for (int step = 0; step < 2 && r == TNT_OK; ++step) {
    std::vector<GemmTask> ts, tx;
    for (int i = 0; i < nb; ++i) {
      const SmallEig& b = blocks[(size_t)i];
      z* X = (step == 0 ? U0 : U1) + he[(size_t)i].yo;  // n x k, ld k
      GemmTask t{};
      t.g.batch = 1;
      t.g.alpha = zmk(1, 0);
      t.g.M = b.k; t.g.N = b.k; t.g.K = b.n;
      t.g.A = X; t.g.a_rs = 1; t.g.a_cs = b.k; t.g.conj_a = 1;
      t.g.B = X; t.g.b_rs = b.k; t.g.b_cs = 1;
      t.g.C = S + so[(size_t)i]; t.g.c_rs = b.k;
      t.herm = 1;
      ts.push_back(t);
      GemmTask u{};
      u.g.batch = 1;
      u.g.alpha = zmk(1, 0);
      u.g.M = b.n; u.g.N = b.k; u.g.K = b.k;
      u.g.A = X; u.g.a_rs = b.k; u.g.a_cs = 1;
      u.g.B = S + so[(size_t)i]; u.g.b_rs = b.k; u.g.b_cs = 1;
      u.g.C = (step == 0) ? U1 + he[(size_t)i].yo : U + b.goff;
      u.g.c_rs = (step == 0) ? b.k : b.n;
      tx.push_back(u);
    }
    r = zgemm_tasks(c, ts);
    if (r != TNT_OK) break;
    const int64_t kmax = blocks[0].n;
    k_ns_coef_all<<<dim3((unsigned)std::min<int64_t>((kmax * kmax + 255) / 256, 64), (unsigned)nb), 256, 0, st>>>(
        S, dblk, dso);
    c->launches++;
    r = zgemm_tasks(c, tx);
  }
  TNT_CHECK_LAUNCH(c);
  c->ws.top = top;
  return r;
}

}  // namespace tnt
