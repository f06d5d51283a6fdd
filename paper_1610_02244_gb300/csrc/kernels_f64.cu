// FP64 building blocks of the two-site update: strided complex GEMM (the contraction
// primitive of App. B.1.1: reorder indices, one matrix product -- here the reorder is
// folded into the strides), a sparse small-operator kernel for the MPO and gate legs,
// the Lanczos vector operations and the tridiagonal eigensolve.
#include <algorithm>
#include <cstdarg>
#include <cmath>

#include "gs_split.cuh"
#include "tnt_internal.cuh"
#include "f32conv.cuh"

namespace tnt {

// ============================================================ complex FP64 GEMM
// 64x64 output tile, BK = 16, 256 threads as 16x16; thread (tx, ty) owns rows ty + 16 r
// and columns tx + 16 c (r, c < 4) so stores are coalesced along the row.
namespace {
constexpr int GM = 64, GN = 64, GK = 16;

__global__ void __launch_bounds__(256) k_zgemm(ZGemm g) {
  __shared__ z As[GK][GM + 1];
  __shared__ z Bs[GK][GN + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t m0 = (int64_t)blockIdx.y * GM, n0 = (int64_t)blockIdx.x * GN;
  if (g.lower_only && m0 + GM <= n0) return;  // strictly upper tile of a Hermitian result
  const int64_t bt = blockIdx.z;
  const z* A = g.A + bt * g.a_bs;
  const z* B = g.B + bt * g.b_bs;
  z* C = g.C + bt * g.c_bs;
  z acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = zmk(0, 0);
  const bool a_kfast = (g.a_cs == 1);
  const bool b_nfast = (g.b_cs == 1);
  for (int64_t k0 = 0; k0 < g.K; k0 += GK) {
#pragma unroll
    for (int t = 0; t < (GM * GK) / 256; ++t) {
      int e = threadIdx.x + 256 * t;
      int i, k;
      if (a_kfast) { k = e % GK; i = e / GK; } else { i = e % GM; k = e / GM; }
      int64_t gi = m0 + i, gk = k0 + k;
      z v = zmk(0, 0);
      if (gi < g.M && gk < g.K) {
        v = A[gi * g.a_rs + gk * g.a_cs];
        if (g.conj_a) v.y = -v.y;
      }
      As[k][i] = v;
    }
#pragma unroll
    for (int t = 0; t < (GN * GK) / 256; ++t) {
      int e = threadIdx.x + 256 * t;
      int j, k;
      if (b_nfast) { j = e % GN; k = e / GN; } else { k = e % GK; j = e / GK; }
      int64_t gj = n0 + j, gk = k0 + k;
      z v = zmk(0, 0);
      if (gj < g.N && gk < g.K) {
        v = B[gk * g.b_rs + gj * g.b_cs];
        if (g.conj_b) v.y = -v.y;
      }
      Bs[k][j] = v;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < GK; ++kk) {
      z a[4], b[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) a[r] = As[kk][ty + 16 * r];
#pragma unroll
      for (int c = 0; c < 4; ++c) b[c] = Bs[kk][tx + 16 * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) zfma(acc[r][c], a[r], b[c]);
    }
    __syncthreads();
  }
  const bool use_beta = (g.beta.x != 0.0 || g.beta.y != 0.0);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    int64_t gi = m0 + ty + 16 * r;
    if (gi >= g.M) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      int64_t gj = n0 + tx + 16 * c;
      if (gj >= g.N) continue;
      z v = zmul(g.alpha, acc[r][c]);
      z* p = C + gi * g.c_rs + gj;
      if (use_beta) v = zadd(v, zmul(g.beta, *p));
      *p = v;
    }
  }
}
}  // namespace

namespace {
// R x 16 output tiles of 256 threads (R = 16, 8, 4), 16 / R threads per output, each taking
// every (16 / R)-th term: for products too small to give every SM a 64 x 64 tile (GB300's
// FP64 units are ~2 FMA per clock per SM, so the FP64 work of a small product must be spread
// thin: a 16 x 16 tile of K = 128 takes 32 us on its SM)
template <int R>
__global__ void __launch_bounds__(256) k_zgemm16(ZGemm g) {
  __shared__ z As[R][17];
  __shared__ z Bs[16][17];
  __shared__ z part[R < 16 ? 256 : 1];
  const int64_t m0 = (int64_t)blockIdx.y * R, n0 = (int64_t)blockIdx.x * 16;
  if (g.lower_only && m0 + R <= n0) return;
  const int64_t bt = blockIdx.z;
  const z* A = g.A + bt * g.a_bs;
  const z* B = g.B + bt * g.b_bs;
  z* C = g.C + bt * g.c_bs;
  const z acc = tile_product<R>(A, g.a_rs, g.a_cs, g.conj_a, B, g.b_rs, g.b_cs, g.conj_b, m0, n0, g.M, g.N, g.K, As,
                                Bs, part);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int64_t gi = m0 + ty, gj = n0 + tx;
  if (ty < R && gi < g.M && gj < g.N) {
    z v = zmul(g.alpha, acc);
    z* p = C + gi * g.c_rs + gj;
    if (g.beta.x != 0.0 || g.beta.y != 0.0) v = zadd(v, zmul(g.beta, *p));
    *p = v;
  }
}
}  // namespace

// the tile height for `tiles` 16 x 16 tiles: the one whose rounds over the SMs take least;
// beyond two rounds the last one is no longer worth re-reading B more often
int tile_rows(int64_t tiles, int nsm) {
  if (tiles > 2 * nsm) return 16;
  const int64_t r16 = 4 * ((tiles + nsm - 1) / nsm), r8 = 2 * ((2 * tiles + nsm - 1) / nsm),
                r4 = (4 * tiles + nsm - 1) / nsm;
  return r16 <= r8 && r16 <= r4 ? 16 : r8 <= r4 ? 8 : 4;
}

int zgemm(Ctx* c, const ZGemm& g) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return TNT_OK;
  if (g.K <= 0) {
    // C = beta C (or zero): not needed by the library; reject to keep the kernel simple
    return set_err(c, TNT_E_INVALID, "zgemm with K = 0");
  }
  if (ozgemm_eligible(c, g)) {
    const int r = ozgemm(c, g);
    if (r != OZ_NOROOM) return r;
  }
  {
    const int nsm = c->nsm;
    const int64_t tiles64 = ((g.M + GM - 1) / GM) * ((g.N + GN - 1) / GN) * g.batch;
    if (tiles64 < nsm && (g.M + 15) / 16 <= 65535 && g.batch <= 65535) {
      const int64_t tiles16 = ((g.M + 15) / 16) * ((g.N + 15) / 16) * g.batch;
      const int R = (g.M + 3) / 4 <= 65535 ? tile_rows(tiles16, nsm) : 16;
      dim3 grid((unsigned)((g.N + 15) / 16), (unsigned)((g.M + R - 1) / R), (unsigned)g.batch);
      ProfScope ps(c, "zgemm_f64", (g.lower_only ? 4.0 : 8.0) * (double)g.M * (double)g.N *
                                       (double)g.K * (double)g.batch);
      if (R == 16) k_zgemm16<16><<<grid, 256, 0, c->stream>>>(g);
      else if (R == 8) k_zgemm16<8><<<grid, 256, 0, c->stream>>>(g);
      else k_zgemm16<4><<<grid, 256, 0, c->stream>>>(g);
      c->launches++;
      TNT_CHECK_LAUNCH(c);
      return TNT_OK;
    }
  }
  if ((g.N + GN - 1) / GN > 0x7fffffff || (g.M + GM - 1) / GM > 65535 || g.batch > 65535)
    return set_err(c, TNT_E_UNSUPPORTED, "zgemm grid too large (M=%lld N=%lld batch=%lld)",
                   (long long)g.M, (long long)g.N, (long long)g.batch);
  dim3 grid((unsigned)((g.N + GN - 1) / GN), (unsigned)((g.M + GM - 1) / GM),
            (unsigned)g.batch);
  ProfScope ps(c, "zgemm_f64", (g.lower_only ? 4.0 : 8.0) * (double)g.M * (double)g.N *
                                   (double)g.K * (double)g.batch);
  k_zgemm<<<grid, 256, 0, c->stream>>>(g);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

namespace {
// The same 16 x 16 tiles for a set of products in one launch; the products travel as a kernel
// argument (no table upload)
constexpr int FT_MAX = 48;
struct FmaTask {
  const z *A, *B;
  z* C;
  int64_t a_rs, a_cs, b_rs, b_cs, c_rs;
  int M, N, K, conj_a, conj_b, herm, sub, tile0;
};
struct FmaTasks {
  int n, tiles;
  FmaTask t[FT_MAX];
};
template <int R>
__global__ void __launch_bounds__(256) k_zgemm16_tasks(const __grid_constant__ FmaTasks T) {
  __shared__ z As[R][17];
  __shared__ z Bs[16][17];
  __shared__ z part[R < 16 ? 256 : 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  for (int w = blockIdx.x; w < T.tiles; w += gridDim.x) {
    int lo = 0, hi = T.n;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (T.t[mid].tile0 <= w) lo = mid;
      else hi = mid;
    }
    const FmaTask& g = T.t[lo];
    const int ntn = (g.N + 15) / 16, tile = w - g.tile0;
    const int64_t m0 = (int64_t)(tile / ntn) * R, n0 = (int64_t)(tile % ntn) * 16;
    if (g.herm && n0 >= m0 + R) continue;
    z acc = tile_product<R>(g.A, g.a_rs, g.a_cs, g.conj_a, g.B, g.b_rs, g.b_cs, g.conj_b, m0, n0, g.M, g.N, g.K, As, Bs,
                            part);
    const int64_t gi = m0 + ty, gj = n0 + tx;
    if (ty < R && gi < g.M && gj < g.N && !(g.herm && gj > gi)) {
      z* p = g.C + gi * g.c_rs + gj;
      if (g.sub) acc = zsub(*p, acc);
      *p = acc;
      if (g.herm && gj < gi) g.C[gj * g.c_rs + gi] = zconj(acc);
    }
  }
}
}  // namespace

int zgemm_fma_tasks(Ctx* c, const GemmTask* const* tasks, int n) {
  int64_t t16 = 0;
  for (int i = 0; i < n; ++i)
    t16 += ((tasks[i]->g.M + 15) / 16) * ((tasks[i]->g.N + 15) / 16) / (tasks[i]->herm ? 2 : 1);
  const int R = tile_rows(t16, c->nsm);
  for (int i0 = 0; i0 < n; i0 += FT_MAX) {
    FmaTasks T;
    T.n = std::min(FT_MAX, n - i0);
    int64_t tiles = 0;
    double flop = 0;
    for (int i = 0; i < T.n; ++i) {
      const ZGemm& g = tasks[i0 + i]->g;
      FmaTask& o = T.t[i];
      o.A = g.A; o.B = g.B; o.C = g.C;
      o.a_rs = g.a_rs; o.a_cs = g.a_cs; o.b_rs = g.b_rs; o.b_cs = g.b_cs; o.c_rs = g.c_rs;
      o.M = (int)g.M; o.N = (int)g.N; o.K = (int)g.K;
      o.conj_a = g.conj_a; o.conj_b = g.conj_b;
      o.herm = tasks[i0 + i]->herm; o.sub = tasks[i0 + i]->sub;
      o.tile0 = (int)tiles;
      tiles += ((g.M + R - 1) / R) * ((g.N + 15) / 16);
      flop += (o.herm ? 4.0 : 8.0) * (double)g.M * (double)g.N * (double)g.K;
    }
    if (tiles > INT32_MAX) return set_err(c, TNT_E_UNSUPPORTED, "grouped FP64 products: too many tiles");
    T.tiles = (int)tiles;
    ProfScope ps(c, "zgemm_f64", flop);
    const unsigned grid = (unsigned)std::min<int64_t>(tiles, 152 * 8);
    if (R == 16) k_zgemm16_tasks<16><<<grid, 256, 0, c->stream>>>(T);
    else if (R == 8) k_zgemm16_tasks<8><<<grid, 256, 0, c->stream>>>(T);
    else k_zgemm16_tasks<4><<<grid, 256, 0, c->stream>>>(T);
    c->launches++;
  }
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

namespace {
__global__ void k_herm_mirror(z* G, int64_t n) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n * n;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / n, j = e % n;
    if (i < j) G[e] = zconj(G[j * n + i]);
  }
}
}  // namespace

int herm_mirror(Ctx* c, z* G, int64_t n) {
  if (n <= 1) return TNT_OK;
  int64_t b = (n * n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  k_herm_mirror<<<(unsigned)b, 256, 0, c->stream>>>(G, n);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

// ============================================================ sparse operator apply
namespace {
constexpr int OP_MAX_NNZ = 2048;
constexpr int OP_MAX_LEG = 256;

// One thread per batch element and group of `rows` output indices (blockIdx.y): with all
// output indices in one thread a small batch (chi = 64: 4096 elements) kept 16 SMs busy, 48
// us for an operator of 64 outputs.  Operators with real entries (every MPO and bond term of
// the models here) take two FMAs per entry instead of four on the FP64 pipe.
template <bool REAL>
__device__ __forceinline__ void op_rows(const OpApply& a, int i0, int i1, const int* s_row, const int* s_col,
                                        const z* s_val, const int64_t* s_in, const int64_t* s_out) {
  const int64_t total = a.B0 * a.B1 * a.B2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    int64_t b2 = e % a.B2;
    int64_t r = e / a.B2;
    int64_t b1 = r % a.B1;
    int64_t b0 = r / a.B1;
    const z* in = a.in + b0 * a.is0 + b1 * a.is1 + b2 * a.is2;
    z* out = a.out + b0 * a.os0 + b1 * a.os1 + b2 * a.os2;
    for (int i = i0; i < i1; ++i) {
      z acc = zmk(0, 0);
      for (int t = s_row[i]; t < s_row[i + 1]; ++t) {
        const z x = in[s_in[s_col[t]]];
        if (REAL) {
          acc.x = fma(s_val[t].x, x.x, acc.x);
          acc.y = fma(s_val[t].x, x.y, acc.y);
        } else {
          zfma(acc, s_val[t], x);
        }
      }
      z* p = out + s_out[i];
      if (a.accumulate) acc = zadd(acc, *p);
      *p = acc;
    }
  }
}

__global__ void __launch_bounds__(256) k_op_apply(OpApply a, int rows) {
  __shared__ int s_row[OP_MAX_LEG + 1];
  __shared__ int s_col[OP_MAX_NNZ];
  __shared__ z s_val[OP_MAX_NNZ];
  __shared__ int64_t s_in[OP_MAX_LEG];
  __shared__ int64_t s_out[OP_MAX_LEG];
  const int i0 = blockIdx.y * rows, i1 = min(a.nI, i0 + rows);
  for (int t = threadIdx.x; t <= a.nI; t += blockDim.x) s_row[t] = a.row_ptr[t];
  for (int t = threadIdx.x; t < a.nJ; t += blockDim.x) s_in[t] = a.in_off[t];
  for (int t = threadIdx.x; t < a.nI; t += blockDim.x) s_out[t] = a.out_off[t];
  __syncthreads();
  int cplx = 0;
  for (int t = s_row[i0] + threadIdx.x; t < s_row[i1]; t += blockDim.x) {
    s_col[t] = a.col[t];
    const z v = a.val[t];
    s_val[t] = v;
    cplx |= v.y != 0.0;
  }
  cplx = __syncthreads_or(cplx);
  if (cplx) op_rows<false>(a, i0, i1, s_row, s_col, s_val, s_in, s_out);
  else op_rows<true>(a, i0, i1, s_row, s_col, s_val, s_in, s_out);
}
}  // namespace

int op_upload(Ctx* c, const std::vector<z>& dense, int nI, int nJ,
              const std::vector<int64_t>& in_off, const std::vector<int64_t>& out_off,
              OpApply* a) {
  if (nI > OP_MAX_LEG || nJ > OP_MAX_LEG)
    return set_err(c, TNT_E_UNSUPPORTED, "operator legs %d x %d exceed %d", nI, nJ,
                   OP_MAX_LEG);
  std::vector<int> row(nI + 1, 0), col;
  std::vector<z> val;
  for (int i = 0; i < nI; ++i) {
    for (int j = 0; j < nJ; ++j) {
      z v = dense[(size_t)i * nJ + j];
      if (v.x != 0.0 || v.y != 0.0) {
        col.push_back(j);
        val.push_back(v);
      }
    }
    row[i + 1] = (int)col.size();
  }
  if (col.size() > (size_t)OP_MAX_NNZ)
    return set_err(c, TNT_E_UNSUPPORTED, "operator has %zu nonzeros > %d", col.size(),
                   OP_MAX_NNZ);
  if (col.empty()) {  // keep valid pointers for the kernel
    col.push_back(0);
    val.push_back(zmk(0, 0));
  }
  // one contiguous scratch block for the five tables
  size_t b_row = ws_round(sizeof(int) * row.size());
  size_t b_col = ws_round(sizeof(int) * col.size());
  size_t b_val = ws_round(sizeof(z) * val.size());
  size_t b_in = ws_round(sizeof(int64_t) * nJ);
  size_t b_out = ws_round(sizeof(int64_t) * nI);
  size_t total = b_row + b_col + b_val + b_in + b_out;
  char* dev = (char*)ws_alloc(c, total);
  if (!dev) return set_err(c, TNT_E_ALLOC, "scratch exhausted for operator tables");
  std::vector<char> host(total, 0);
  memcpy(host.data(), row.data(), sizeof(int) * row.size());
  memcpy(host.data() + b_row, col.data(), sizeof(int) * col.size());
  memcpy(host.data() + b_row + b_col, val.data(), sizeof(z) * val.size());
  memcpy(host.data() + b_row + b_col + b_val, in_off.data(), sizeof(int64_t) * nJ);
  memcpy(host.data() + b_row + b_col + b_val + b_in, out_off.data(), sizeof(int64_t) * nI);
  TNT_TRY(to_device(c, dev, host.data(), total));
  a->nI = nI;
  a->nJ = nJ;
  a->nnz = row[nI];
  a->row_ptr = (const int*)dev;
  a->col = (const int*)(dev + b_row);
  a->val = (const z*)(dev + b_row + b_col);
  a->in_off = (const int64_t*)(dev + b_row + b_col + b_val);
  a->out_off = (const int64_t*)(dev + b_row + b_col + b_val + b_in);
  return TNT_OK;
}

int op_apply(Ctx* c, const OpApply& a) {
  int64_t total = a.B0 * a.B1 * a.B2;
  if (total <= 0) return TNT_OK;
  int64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  ProfScope ps(c, "op_apply", 8.0 * (double)a.nnz * (double)total);
  // at least four blocks per SM where the output indices allow it
  const int64_t want = std::min<int64_t>(a.nI, (152 * 4 + blocks - 1) / blocks);
  const int rows = (int)((a.nI + want - 1) / want);
  k_op_apply<<<dim3((unsigned)blocks, (unsigned)((a.nI + rows - 1) / rows)), 256, 0, c->stream>>>(a, rows);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

// ============================================================ vector kernels
// Deterministic reductions: a fixed grid of RB blocks; block b always covers the same
// elements in the same order; a single-block second pass sums the partials in order.
namespace {
constexpr int RB = 608;       // 4 blocks per SM (152 SMs): enough loads in flight for HBM
constexpr int RT = 256;
constexpr int KB = 8;         // vectors per multidot pass
// multidot's grid: 2 blocks per SM.  Each thread ends with 2 KV sums to reduce (five
// shuffle-adds each, on the FP64 pipe); at 4 blocks per SM a 2^20-element vector gave a
// thread only ~7 elements and the reduction rivalled the dot products themselves
constexpr int RB_DOT = 304;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// block-wide sum of one double (result valid in thread 0)
__device__ __forceinline__ double block_sum(double v, double* sh) {
  v = warp_sum(v);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) sh[w] = v;
  __syncthreads();
  double r = 0;
  if (w == 0) {
    r = (l < (int)(blockDim.x >> 5)) ? sh[l] : 0.0;
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}

// partial[v][blk] = sum over the block's range of conj(V_v[e]) w[e], v < KV; the KV
// loads of one element are independent and issued together.  The last CTA to finish (an
// arrival counter, reset by that CTA) sums the partials in block order into out[v]: the
// reduction stays deterministic and needs no second launch.
template <int KV>
__global__ void __launch_bounds__(RT) k_multidot(const z* __restrict__ V, int64_t ld,
                                                 const z* __restrict__ w, int64_t n,
                                                 z* __restrict__ partial,
                                                 const int* __restrict__ skip,
                                                 unsigned* __restrict__ counter,
                                                 z* __restrict__ out) {
  if (skip && *skip) return;  // a pass the caller decided on the device not to need
  __shared__ double sh[32];
  double ar[KV], ai[KV];
#pragma unroll
  for (int v = 0; v < KV; ++v) ar[v] = ai[v] = 0.0;
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    const z x = w[e];
    z u[KV];
#pragma unroll
    for (int v = 0; v < KV; ++v) u[v] = V[(int64_t)v * ld + e];
#pragma unroll
    for (int v = 0; v < KV; ++v) {
      ar[v] = fma(u[v].x, x.x, fma(u[v].y, x.y, ar[v]));
      ai[v] = fma(u[v].x, x.y, fma(-u[v].y, x.x, ai[v]));
    }
  }
  // all 2 KV sums in one pass: shuffles within each warp, then one barrier and a fixed-order
  // sum over the warps (the per-value block reductions cost two barriers each, and with a
  // few elements per thread they outweighed the loop)
  __shared__ double shp[RT / 32][2 * KV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int v = 0; v < KV; ++v) {
    ar[v] = warp_sum(ar[v]);
    ai[v] = warp_sum(ai[v]);
  }
  if (lane == 0) {
#pragma unroll
    for (int v = 0; v < KV; ++v) {
      shp[wid][2 * v] = ar[v];
      shp[wid][2 * v + 1] = ai[v];
    }
  }
  __syncthreads();
  if (threadIdx.x < 2 * KV) {
    double t = 0;
#pragma unroll
    for (int q = 0; q < RT / 32; ++q) t += shp[q][threadIdx.x];
    double* po = (double*)(partial + (int64_t)(threadIdx.x >> 1) * gridDim.x + blockIdx.x);
    po[threadIdx.x & 1] = t;
    __threadfence();
  }
  // the last CTA to arrive sums every CTA's partials, in block order
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const double* pp = (const double*)partial;
  double acc[2 * KV];
#pragma unroll
  for (int v = 0; v < 2 * KV; ++v) acc[v] = 0.0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += RT) {
#pragma unroll
    for (int v = 0; v < KV; ++v) {
      const z pv = __ldcg(partial + (int64_t)v * gridDim.x + b);
      acc[2 * v] += pv.x;
      acc[2 * v + 1] += pv.y;
    }
  }
  (void)pp;
#pragma unroll
  for (int v = 0; v < 2 * KV; ++v) acc[v] = warp_sum(acc[v]);
  __syncthreads();
  if (lane == 0) {
#pragma unroll
    for (int v = 0; v < 2 * KV; ++v) shp[wid][v] = acc[v];
  }
  __syncthreads();
  if (threadIdx.x < 2 * KV) {
    double t = 0;
#pragma unroll
    for (int q = 0; q < RT / 32; ++q) t += shp[q][threadIdx.x];
    ((double*)(out + (threadIdx.x >> 1)))[threadIdx.x & 1] = t;
  }
  if (threadIdx.x == 0) *counter = 0u;
  (void)sh;
}

void launch_multidot(int kv, dim3 g, dim3 b, cudaStream_t st, const z* V, int64_t ld,
                     const z* w, int64_t n, z* partial, const int* skip, unsigned* cnt,
                     z* out) {
  switch (kv) {
    case 1: k_multidot<1><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    case 2: k_multidot<2><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    case 3: k_multidot<3><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    case 4: k_multidot<4><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    case 5: k_multidot<5><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    case 6: k_multidot<6><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    case 7: k_multidot<7><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
    default: k_multidot<8><<<g, b, 0, st>>>(V, ld, w, n, partial, skip, cnt, out); break;
  }
}

// w[e] -= sum_v coef[v] V_v[e]; partial[blk] = sum |w[e]|^2, and the last CTA to finish
// writes the total |w|^2
__global__ void __launch_bounds__(RT) k_multiaxpy_norm(const z* __restrict__ V, int64_t ld,
                                                       int k, const z* __restrict__ coef,
                                                       z* __restrict__ w, int64_t n,
                                                       double* __restrict__ partial,
                                                       const int* __restrict__ skip,
                                                       unsigned* __restrict__ counter,
                                                       double* __restrict__ norm2_out) {
  if (skip && *skip) return;
  __shared__ z sc[64];
  __shared__ double sh[32];
  for (int t = threadIdx.x; t < k; t += blockDim.x) sc[t] = coef[t];
  __syncthreads();
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  double acc = 0;
  for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    z x = w[e];
    int v = 0;
    for (; v + 8 <= k; v += 8) {  // eight independent loads in flight per thread
      z u[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) u[q] = V[(int64_t)(v + q) * ld + e];
#pragma unroll
      for (int q = 0; q < 8; ++q) {  // x -= cv u as four FMAs
        const z cv = sc[v + q];
        x.x = fma(-cv.x, u[q].x, fma(cv.y, u[q].y, x.x));
        x.y = fma(-cv.x, u[q].y, fma(-cv.y, u[q].x, x.y));
      }
    }
    for (; v < k; ++v) {
      const z u = V[(int64_t)v * ld + e];
      const z cv = sc[v];
      x.x = fma(-cv.x, u.x, fma(cv.y, u.y, x.x));
      x.y = fma(-cv.x, u.y, fma(-cv.y, u.x, x.y));
    }
    w[e] = x;
    acc = fma(x.x, x.x, fma(x.y, x.y, acc));
  }
  double s = block_sum(acc, sh);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = s;
    __threadfence();
  }
  // the last CTA to arrive sums every CTA's partial, in block order
  __shared__ bool s_last;
  if (threadIdx.x == 0) s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double r = 0;
  for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) r += __ldcg(partial + b);
  r = block_sum(r, sh);
  if (threadIdx.x == 0) {
    *norm2_out = r;
    *counter = 0u;
  }
}

// ---------------------------------------------------------------- FP32-arithmetic passes
// The Gram-Schmidt passes of a Lanczos phase whose matvec is split TF32 (relative error
// about 2^-22): the FP64 vectors are read as they are and multiplied in FP32 with FP32
// sums per thread, warp and block; the sums over blocks, the subtraction from w and w
// itself stay FP64, so cancellation in w - V c does not amplify the FP32 rounding (the
// update's error is u_32 |V c|, like a matvec error of that size).  An SM retires 64 FP32
// FMAs per clock against 2 FP64 FMAs on GB300: these passes are bound by HBM, where the
// FP64 forms are bound by the FP64 pipe.  Conversions between the widths are integer bit
// operations on the IEEE-754 layouts (f32conv.cuh), so that no FP64-pipe instruction
// enters the element loop.
// The last CTA's sums of nv values over nb blocks (partials[v * nb + b], FP64) into
// out[v]: thread t < per nv (per the largest power of two <= RT / nv) adds blocks
// t / nv, t / nv + per, ... of value t % nv, then a fixed tree over the per copies.
// Deterministic, and a handful of FP64 adds per thread (a serial FP64 chain costs the
// FP64 pipe's full issue time per step).
__device__ void last_cta_sum(const double* __restrict__ partials, int nv, int nb,
                             double* __restrict__ out) {
  __shared__ double sp[RT];
  const int t = threadIdx.x;
  int per = 1;
  while (2 * per * nv <= RT) per *= 2;
  double r = 0;
  if (t < per * nv)
    for (int b = t / nv; b < nb; b += per) r += __ldcg(partials + (int64_t)(t % nv) * nb + b);
  sp[t] = r;
  __syncthreads();
  for (int h = per / 2; h >= 1; h >>= 1) {
    if (t < h * nv) sp[t] += sp[t + h * nv];
    __syncthreads();
  }
  if (t < nv) out[t] = sp[t];
}

template <int KV>
__global__ void __launch_bounds__(RT) k_multidot32(const z* __restrict__ V, int64_t ld,
                                                   const z* __restrict__ w, int64_t n,
                                                   double* __restrict__ partial,
                                                   unsigned* __restrict__ counter,
                                                   z* __restrict__ out) {
  float ar[KV], ai[KV];
#pragma unroll
  for (int v = 0; v < KV; ++v) ar[v] = ai[v] = 0.f;
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    const z xd = w[e];
    z u[KV];
#pragma unroll
    for (int v = 0; v < KV; ++v) u[v] = V[(int64_t)v * ld + e];
    const float xr = f32_of(xd.x), xi = f32_of(xd.y);
#pragma unroll
    for (int v = 0; v < KV; ++v) {  // conj(u) x
      const float ur = f32_of(u[v].x), ui = f32_of(u[v].y);
      ar[v] = fmaf(ur, xr, fmaf(ui, xi, ar[v]));
      ai[v] = fmaf(ur, xi, fmaf(-ui, xr, ai[v]));
    }
  }
  __shared__ float shp[RT / 32][2 * KV];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int v = 0; v < KV; ++v) {
    ar[v] = warp_sum_f(ar[v]);
    ai[v] = warp_sum_f(ai[v]);
  }
  if (lane == 0) {
#pragma unroll
    for (int v = 0; v < KV; ++v) {
      shp[wid][2 * v] = ar[v];
      shp[wid][2 * v + 1] = ai[v];
    }
  }
  __syncthreads();
  if (threadIdx.x < 2 * KV) {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < RT / 32; ++q) t += shp[q][threadIdx.x];
    partial[(int64_t)threadIdx.x * gridDim.x + blockIdx.x] = f64_of(t);
    __threadfence();
  }
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  last_cta_sum(partial, 2 * KV, (int)gridDim.x, (double*)out);
  if (threadIdx.x == 0) *counter = 0u;
}

void launch_multidot32(int kv, dim3 g, dim3 b, cudaStream_t st, const z* V, int64_t ld,
                       const z* w, int64_t n, double* partial, unsigned* cnt, z* out) {
  switch (kv) {
    case 1: k_multidot32<1><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    case 2: k_multidot32<2><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    case 3: k_multidot32<3><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    case 4: k_multidot32<4><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    case 5: k_multidot32<5><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    case 6: k_multidot32<6><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    case 7: k_multidot32<7><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
    default: k_multidot32<8><<<g, b, 0, st>>>(V, ld, w, n, partial, cnt, out); break;
  }
}

// w[e] -= sum_v coef[v] V_v[e] (the sum in FP32, the subtraction in FP64); the last CTA
// writes |w|^2 (FP32 per block, FP64 over blocks)
__global__ void __launch_bounds__(RT) k_multiaxpy_norm32(const z* __restrict__ V, int64_t ld,
                                                         int k, const z* __restrict__ coef,
                                                         z* __restrict__ w, int64_t n,
                                                         double* __restrict__ partial,
                                                         unsigned* __restrict__ counter,
                                                         double* __restrict__ norm2_out) {
  __shared__ float2 sc[64];
  __shared__ float shw[RT / 32];
  for (int t = threadIdx.x; t < k; t += blockDim.x)
    sc[t] = make_float2(f32_of(coef[t].x), f32_of(coef[t].y));
  __syncthreads();
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  float acc = 0.f;
  for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    float sr = 0.f, si = 0.f;
    int v = 0;
    for (; v + 8 <= k; v += 8) {
      z u[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) u[q] = V[(int64_t)(v + q) * ld + e];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float2 cv = sc[v + q];
        const float ur = f32_of(u[q].x), ui = f32_of(u[q].y);
        sr = fmaf(cv.x, ur, fmaf(-cv.y, ui, sr));
        si = fmaf(cv.x, ui, fmaf(cv.y, ur, si));
      }
    }
    for (; v < k; ++v) {
      const z u = V[(int64_t)v * ld + e];
      const float2 cv = sc[v];
      const float ur = f32_of(u.x), ui = f32_of(u.y);
      sr = fmaf(cv.x, ur, fmaf(-cv.y, ui, sr));
      si = fmaf(cv.x, ui, fmaf(cv.y, ur, si));
    }
    z x = w[e];
    x.x -= f64_of(sr);
    x.y -= f64_of(si);
    w[e] = x;
    const float xr = f32_of(x.x), xi = f32_of(x.y);
    acc = fmaf(xr, xr, fmaf(xi, xi, acc));
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  acc = warp_sum_f(acc);
  if (lane == 0) shw[wid] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int q = 0; q < RT / 32; ++q) t += shw[q];
    partial[blockIdx.x] = f64_of(t);
    __threadfence();
  }
  __shared__ bool s_last;
  if (threadIdx.x == 0) s_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  last_cta_sum(partial, 1, (int)gridDim.x, norm2_out);
  if (threadIdx.x == 0) *counter = 0u;
}

__global__ void k_reduce_real(const double* __restrict__ partial, int nb,
                              double* __restrict__ out, const int* __restrict__ skip) {
  if (skip && *skip) return;  // out keeps its previous value
  __shared__ double sh[32];
  double r = 0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) r += partial[b];
  r = block_sum(r, sh);
  if (threadIdx.x == 0) out[0] = r;
}

__global__ void k_norm2_partial(const z* __restrict__ x, int64_t n, double* __restrict__ partial) {
  __shared__ double sh[32];
  const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = min(n, lo + chunk);
  double acc = 0;
  for (int64_t e = lo + threadIdx.x; e < hi; e += blockDim.x) {
    z v = x[e];
    acc = fma(v.x, v.x, fma(v.y, v.y, acc));
  }
  double s = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

__global__ void k_normalize(const z* __restrict__ x, z* __restrict__ y, int64_t n,
                            const double* __restrict__ norm2) {
  // the scale by one thread of the block: an FP64 square root and division in every thread
  // cost several times the FP64-pipe issue slots of the scaling itself
  __shared__ double s_s;
  if (threadIdx.x == 0) s_s = 1.0 / sqrt(norm2[0]);
  __syncthreads();
  const double s = s_s;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    y[e] = zscale(x[e], s);
}
}  // namespace

int vec_multidot(Ctx* c, const z* V, int64_t ld, int k, const z* w, int64_t n, z* d_dots,
                 const int* d_skip) {
  if (k <= 0) return TNT_OK;
  // partial sums live in scratch only until the next launch on the same stream, so the
  // region is handed back immediately (stream order serialises its reuse)
  const size_t top = c->ws.top;
  z* partial = (z*)ws_alloc(c, ws_round(sizeof(z) * (size_t)KB * RB_DOT));
  c->ws.top = top;
  if (!partial) return set_err(c, TNT_E_ALLOC, "scratch exhausted (multidot)");
  for (int v0 = 0; v0 < k; v0 += KB) {
    int kv = (k - v0 < KB) ? (k - v0) : KB;
    // FP64 FLOPs (complex MAC = 8); a pass the device may skip is profiled apart, with no
    // work claimed (the host cannot know whether it ran)
    ProfScope ps(c, d_skip ? "multidot_cond" : "multidot", d_skip ? 0.0 : 8.0 * (double)kv * (double)n);
    launch_multidot(kv, RB_DOT, RT, c->stream, V + (int64_t)v0 * ld, ld, w, n, partial, d_skip,
                    c->d_count, d_dots + v0);
    c->launches += 1;
  }
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int vec_multiaxpy_norm(Ctx* c, const z* V, int64_t ld, int k, const z* d_coef, z* w,
                       int64_t n, double* d_norm2, const int* d_skip) {
  if (k > 64) return set_err(c, TNT_E_UNSUPPORTED, "multiaxpy with k=%d > 64", k);
  const size_t top = c->ws.top;
  double* partial = (double*)ws_alloc(c, ws_round(sizeof(double) * RB));
  c->ws.top = top;
  if (!partial) return set_err(c, TNT_E_ALLOC, "scratch exhausted (multiaxpy)");
  {
    ProfScope ps(c, d_skip ? "multiaxpy_cond" : "multiaxpy",
                 d_skip ? 0.0 : (8.0 * (double)k + 4.0) * (double)n);  // FP64 FLOPs
    k_multiaxpy_norm<<<RB, RT, 0, c->stream>>>(V, ld, k, d_coef, w, n, partial, d_skip,
                                               c->d_count + 1, d_norm2);
  }
  c->launches += 1;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int vec_multidot_f32(Ctx* c, const z* V, int64_t ld, int k, const z* w, int64_t n, z* d_dots) {
  if (k <= 0) return TNT_OK;
  const size_t top = c->ws.top;
  // four CTAs per SM: bound by HBM, these need the loads of more threads in flight than
  // the FP64 form (whose two CTAs per SM already saturate the FP64 pipe)
  double* partial = (double*)ws_alloc(c, ws_round(sizeof(double) * 2 * (size_t)KB * RB));
  c->ws.top = top;
  if (!partial) return set_err(c, TNT_E_ALLOC, "scratch exhausted (multidot32)");
  for (int v0 = 0; v0 < k; v0 += KB) {
    const int kv = (k - v0 < KB) ? (k - v0) : KB;
    ProfScope ps(c, "multidot32", 16.0 * (double)(kv + 1) * (double)n);  // bytes read
    launch_multidot32(kv, RB, RT, c->stream, V + (int64_t)v0 * ld, ld, w, n, partial,
                      c->d_count, d_dots + v0);
    c->launches += 1;
  }
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int vec_multiaxpy_norm_f32(Ctx* c, const z* V, int64_t ld, int k, const z* d_coef, z* w,
                           int64_t n, double* d_norm2) {
  if (k > 64) return set_err(c, TNT_E_UNSUPPORTED, "multiaxpy with k=%d > 64", k);
  const size_t top = c->ws.top;
  double* partial = (double*)ws_alloc(c, ws_round(sizeof(double) * RB));
  c->ws.top = top;
  if (!partial) return set_err(c, TNT_E_ALLOC, "scratch exhausted (multiaxpy32)");
  {
    ProfScope ps(c, "multiaxpy32", 16.0 * ((double)k + 2.0) * (double)n);  // bytes moved
    k_multiaxpy_norm32<<<RB, RT, 0, c->stream>>>(V, ld, k, d_coef, w, n, partial,
                                                 c->d_count + 1, d_norm2);
  }
  c->launches += 1;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int vec_norm2(Ctx* c, const z* x, int64_t n, double* d_norm2) {
  const size_t top = c->ws.top;
  double* partial = (double*)ws_alloc(c, ws_round(sizeof(double) * RB));
  c->ws.top = top;
  if (!partial) return set_err(c, TNT_E_ALLOC, "scratch exhausted (norm2)");
  k_norm2_partial<<<RB, RT, 0, c->stream>>>(x, n, partial);
  k_reduce_real<<<1, 256, 0, c->stream>>>(partial, RB, d_norm2, nullptr);
  c->launches += 2;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int vec_dot(Ctx* c, const z* x, const z* y, int64_t n, z* d_dot) {
  return vec_multidot(c, x, 0, 1, y, n, d_dot);
}

int vec_normalize(Ctx* c, const z* x, z* y, int64_t n, const double* d_norm2) {
  int64_t blocks = (n + 255) / 256;
  if (blocks > RB) blocks = RB;  // grid-stride: one scale per CTA, four CTAs per SM
  if (blocks < 1) blocks = 1;
  k_normalize<<<(unsigned)blocks, 256, 0, c->stream>>>(x, y, n, d_norm2);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

// ============================================================ one Gram-Schmidt step
// The vector work of one FP64 Krylov step in one cooperative launch: w orthogonalised against
// V[0..k), the norm, and the next basis vector.  A is Hermitian, so that w = A v_{k-1} has
// components above the rounding level along v_{k-1} and v_{k-2} only: those two are taken out
// first, then one classical Gram-Schmidt pass over all of V.
//   phase 1: c = (v_{k-2}, v_{k-1})^H w    | grid barrier
//   phase 2: w -= (v_{k-2}, v_{k-1}) c, c' = V^H w | grid barrier
//   phase 3: w -= V c', v_k = w / |w|
// |w|^2 after phase 3 is |w|^2 before it (summed with c') minus |c'|^2, V being orthonormal.
// Where c' takes more than a quarter of it (w nearly in the span of V), one pass is not
// enough: a second one over all of V follows, and the sum is taken directly (two more
// barriers).
// CTA b keeps elements [b S, (b + 1) S) of w in shared memory, and of the basis too where
// they fit (k S 16 bytes), copied there while phase 1 runs.  Each warp takes whole vectors
// (v = warp, warp + 8, ...) of its CTA's slice: the lanes' sums are combined by a transposed
// butterfly over four vectors' eight sums (nine FP64 adds instead of 40).  The partial sums
// of all CTAs are added in CTA order by every CTA, so all hold the same c, and the result is
// deterministic.
// What bounds it: the FP64 pipe, 8 (k + 2) n FMAs at two per SM and clock (15 us at n = 65536,
// k = 16), and two grid barriers.  Measured over a solve at n = 65536, k up to 32: 35 us a
// step on average, 55 us with both passes over all of V; at n of about 2000 16 and 24 us.
// The separate launches it replaces took 160 us there (four dot-product launches of eight
// vectors at 27 to 30 us, whatever n: with one element per thread each spent its time
// reducing 16 sums per thread), 115 us at n = 5000.
namespace {
constexpr int GS_THREADS = 256, GS_WARPS = GS_THREADS / 32;

struct GsArgs {  // part: 64 vectors' sums, npart: the norm's
  const z* V;
  int64_t n;
  int k;
  const z* w;
  z* vnext;  // v_k; nullptr: not wanted
  double* alpha;  // alpha[k - 1] and beta[k - 1] of the step
  double* beta;
  z* part;       // 2 x 64 x gridDim.x
  double* npart; // 2 x gridDim.x
  unsigned* bar; // arrivals since the solve began
  unsigned base; // its value before this launch
  int* status;
  int S;
  int keep;      // V slices in shared memory
};

// Every CTA adds one to the counter (release) and waits (acquire) until it has moved by
// `want` since the solve began; the count wraps.  false: the wait expired, the CTA must stop
// (and so will the others).
__device__ bool gs_barrier(const GsArgs& a, unsigned want) {
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned seen;
    int ok = 1;
    asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(a.bar), "r"(1u) : "memory");
    uint64_t t0 = 0;
    for (unsigned polls = 0;; ++polls) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.bar) : "memory");
      if ((int)(seen - want) >= 0) break;
      if ((polls & 1023u) == 1023u) {
        uint64_t now;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
        if (!t0) t0 = now;
        if (now - t0 > 2000000000ull) {
          atomicOr(a.status, 2);
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

// eight sums over the warp: lane l returns the total of s[l & 7]
__device__ __forceinline__ double sum8(double* s) {
  const int l = threadIdx.x & 31;
#pragma unroll
  for (int o = 4; o >= 1; o >>= 1) {  // lanes whose bit o is set keep the upper half
    const bool up = (l & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const double give = up ? s[i] : s[i + o], keep = up ? s[i + o] : s[i];
      s[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double r = s[0];
  r += __shfl_xor_sync(0xffffffffu, r, 8);
  r += __shfl_xor_sync(0xffffffffu, r, 16);
  return r;
}

// four sums over the warp: lane l returns the total of s[l & 3]
__device__ __forceinline__ double sum4(double* s) {
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

// the CTA's share of V^H w to part[v][blockIdx.x]
__device__ void gs_dots(const GsArgs& a, const z* sw, const z* V0, int64_t ld, int cnt, z* part) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int v0 = warp; v0 < a.k; v0 += 4 * GS_WARPS) {
    double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int nv = min(4, (a.k - v0 + GS_WARPS - 1) / GS_WARPS);
    const z* p0 = V0 + (int64_t)v0 * ld;
    const int64_t st = (int64_t)GS_WARPS * ld;
    if (nv == 4) {
#pragma unroll 2
      for (int e = lane; e < cnt; e += 32) {
        const z x = sw[e];
        z u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) u[q] = p0[q * st + e];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          s[2 * q] = fma(u[q].x, x.x, fma(u[q].y, x.y, s[2 * q]));
          s[2 * q + 1] = fma(u[q].x, x.y, fma(-u[q].y, x.x, s[2 * q + 1]));
        }
      }
    } else {
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (q >= nv) break;
#pragma unroll 4
        for (int e = lane; e < cnt; e += 32) {
          const z x = sw[e], u = p0[q * st + e];
          s[2 * q] = fma(u.x, x.x, fma(u.y, x.y, s[2 * q]));
          s[2 * q + 1] = fma(u.x, x.y, fma(-u.y, x.x, s[2 * q + 1]));
        }
      }
    }
    const double r = sum8(s);
    if (lane < 2 * nv)
      ((double*)(part + (int64_t)(v0 + (lane >> 1) * GS_WARPS) * gridDim.x + blockIdx.x))[lane & 1] = r;
  }
}

// c[v] = the sum over the CTAs, in shared memory
__device__ void gs_total(const GsArgs& a, const z* part, z* sc) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int v0 = warp; v0 < a.k; v0 += 4 * GS_WARPS) {
    double s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int nv = min(4, (a.k - v0 + GS_WARPS - 1) / GS_WARPS);
    for (int b = lane; b < (int)gridDim.x; b += 32)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (q < nv) {
          const z p = __ldcg(part + (int64_t)(v0 + q * GS_WARPS) * gridDim.x + b);
          s[2 * q] += p.x;
          s[2 * q + 1] += p.y;
        }
    const double r = sum8(s);
    if (lane < 2 * nv) ((double*)(sc + v0 + (lane >> 1) * GS_WARPS))[lane & 1] = r;
  }
  __syncthreads();
}

// w -= V c over the CTA's slice; returns the thread's share of |w|^2.  A slice of at most 64
// elements would leave most threads idle behind chains of 2 k dependent FMAs: there four
// threads share an element, each a quarter of the vectors, and their sums meet in sacc.
__device__ double gs_update(const GsArgs& a, z* sw, const z* V0, int64_t ld, int cnt, const z* sc, z* sacc) {
  double acc = 0;
  if (cnt <= 64) {
    const int e = threadIdx.x & 63, q = threadIdx.x >> 6;
    z s0 = zmk(0, 0), s1 = s0;
    if (e < cnt) {
      int v = q;
      for (; v + 4 < a.k; v += 8) {
        const z u0 = V0[(int64_t)v * ld + e], u1 = V0[(int64_t)(v + 4) * ld + e];
        zfma(s0, sc[v], u0);
        zfma(s1, sc[v + 4], u1);
      }
      if (v < a.k) zfma(s0, sc[v], V0[(int64_t)v * ld + e]);
      sacc[threadIdx.x] = zadd(s0, s1);
    }
    __syncthreads();
    if (threadIdx.x < cnt) {
      const z p = zadd(zadd(sacc[e], sacc[64 + e]), zadd(sacc[128 + e], sacc[192 + e]));
      const z x = zsub(sw[e], p);
      sw[e] = x;
      acc = fma(x.x, x.x, x.y * x.y);
    }
    return acc;
  }
  for (int e = threadIdx.x; e < cnt; e += GS_THREADS) {
    z x = sw[e];
    int v = 0;
    for (; v + 8 <= a.k; v += 8) {
      z u[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) u[q] = V0[(int64_t)(v + q) * ld + e];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const z c = sc[v + q];
        x.x = fma(-c.x, u[q].x, fma(c.y, u[q].y, x.x));
        x.y = fma(-c.x, u[q].y, fma(-c.y, u[q].x, x.y));
      }
    }
    for (; v < a.k; ++v) {
      const z u = V0[(int64_t)v * ld + e], c = sc[v];
      x.x = fma(-c.x, u.x, fma(c.y, u.y, x.x));
      x.y = fma(-c.x, u.y, fma(-c.y, u.x, x.y));
    }
    sw[e] = x;
    acc = fma(x.x, x.x, fma(x.y, x.y, acc));
  }
  return acc;
}

__global__ void __launch_bounds__(GS_THREADS, 1) k_gs_step(GsArgs a) {
  extern __shared__ z sm_gs[];
  __shared__ z sc[64];
  __shared__ z sacc[GS_THREADS];
  __shared__ double sh[32];
  __shared__ double s_rn;
  __shared__ int s_direct;
  __shared__ double s4[GS_WARPS][4];
  z* sw = sm_gs;
  z* sv = sm_gs + a.S;
  const int64_t lo = (int64_t)blockIdx.x * a.S;
  const int cnt = (int)max((int64_t)0, min((int64_t)a.S, a.n - lo));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  z* p1 = a.part;
  z* p2 = a.part + (int64_t)64 * gridDim.x;
  const z* Vg = a.V + lo;
  const z* Va = Vg + (int64_t)(a.k - 1) * a.n;                 // v_{k-1}
  const z* Vb = Vg + (int64_t)(a.k > 1 ? a.k - 2 : 0) * a.n;   // v_{k-2}; k = 1: taken with c = 0
  double d4[4] = {0, 0, 0, 0};
  for (int e = tid; e < cnt; e += GS_THREADS) {
    const z x = a.w[lo + e], u = Va[e], u1 = Vb[e];
    sw[e] = x;
    d4[0] = fma(u.x, x.x, fma(u.y, x.y, d4[0]));
    d4[1] = fma(u.x, x.y, fma(-u.y, x.x, d4[1]));
    d4[2] = fma(u1.x, x.x, fma(u1.y, x.y, d4[2]));
    d4[3] = fma(u1.x, x.y, fma(-u1.y, x.x, d4[3]));
  }
  if (a.keep) {
    for (int v = warp; v < a.k; v += GS_WARPS)
      for (int e = lane; e < cnt; e += 32)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(sv + (int64_t)v * a.S + e)),
                     "l"(Vg + (int64_t)v * a.n + e)
                     : "memory");
  }
  const int nw = min(GS_WARPS, (cnt + 31) >> 5);  // warps that have elements
  if (warp < nw) {
    const double r = sum4(d4);
    if (lane < 4) s4[warp][lane] = r;
  }
  __syncthreads();
  if (warp == 0) {
    double r = (lane >> 2) < nw ? s4[lane >> 2][lane & 3] : 0.0;
    for (int o = 4; o < 4 * nw; o <<= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (lane < 4) ((double*)(p1 + (int64_t)(lane >> 1) * gridDim.x + blockIdx.x))[lane & 1] = r;
  }
  const z* V = a.keep ? sv : Vg;
  const int64_t ld = a.keep ? a.S : a.n;
  bool ok = gs_barrier(a, a.base + 1u * gridDim.x);
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (ok) {
    if (warp < 2) {
      double re = 0, im = 0;
      for (int b = lane; b < (int)gridDim.x; b += 32) {
        const z p = __ldcg(p1 + (int64_t)warp * gridDim.x + b);
        re += p.x;
        im += p.y;
      }
      re = warp_sum(re);
      im = warp_sum(im);
      if (lane == 0) sc[warp] = warp == 1 && a.k == 1 ? zmk(0, 0) : zmk(re, im);
    }
    __syncthreads();
    const z c0 = sc[0], c1 = sc[1];
    if (blockIdx.x == 0 && tid == 0) a.alpha[a.k - 1] = c0.x;
    double acc = 0;
    for (int e = tid; e < cnt; e += GS_THREADS) {
      const z u = V[(int64_t)(a.k - 1) * ld + e], u1 = V[(int64_t)(a.k > 1 ? a.k - 2 : 0) * ld + e];
      z x = sw[e];
      x.x = fma(-c0.x, u.x, fma(c0.y, u.y, x.x));
      x.y = fma(-c0.x, u.y, fma(-c0.y, u.x, x.y));
      x.x = fma(-c1.x, u1.x, fma(c1.y, u1.y, x.x));
      x.y = fma(-c1.x, u1.y, fma(-c1.y, u1.x, x.y));
      sw[e] = x;
      acc = fma(x.x, x.x, fma(x.y, x.y, acc));
    }
    __syncthreads();
    gs_dots(a, sw, V, ld, cnt, p2);
    acc = block_sum(acc, sh);
    if (tid == 0) a.npart[blockIdx.x] = acc;
    ok = gs_barrier(a, a.base + 2u * gridDim.x);
  }
  if (ok) {
    gs_total(a, p2, sc);
    if (tid < 32) {  // |w|^2 before the second update, and what c' takes of it
      double r = 0, q = 0;
      for (int b = tid; b < (int)gridDim.x; b += 32) r += __ldcg(a.npart + b);
      for (int v = tid; v < a.k; v += 32) q = fma(sc[v].x, sc[v].x, fma(sc[v].y, sc[v].y, q));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        r += __shfl_xor_sync(0xffffffffu, r, o);
        q += __shfl_xor_sync(0xffffffffu, q, o);
      }
      if (tid == 0) {
        sh[0] = r - q;
        s_direct = !(q <= 0.25 * r);
      }
    }
    gs_update(a, sw, V, ld, cnt, sc, sacc);
    __syncthreads();
    if (s_direct) {  // the same decision in every CTA
      __shared__ double sh2[32];
      gs_dots(a, sw, V, ld, cnt, p1);
      ok = gs_barrier(a, a.base + 3u * gridDim.x);
      if (ok) {
        gs_total(a, p1, sc);
        const double acc = block_sum(gs_update(a, sw, V, ld, cnt, sc, sacc), sh2);
        if (tid == 0) a.npart[gridDim.x + blockIdx.x] = acc;
        ok = gs_barrier(a, a.base + 4u * gridDim.x);
      }
      if (ok && tid < 32) {
        double r = 0;
        for (int b = tid; b < (int)gridDim.x; b += 32) r += __ldcg(a.npart + gridDim.x + b);
        r = warp_sum(r);
        if (tid == 0) sh[0] = r;
      }
    } else if (blockIdx.x == 0 && tid == 0) {
      // the launch counts four arrivals per CTA
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], %1;" ::"l"(a.bar), "r"(2u * gridDim.x) : "memory");
    }
  }
  if (!ok) {  // the host reads the status word with the step's numbers
    if (blockIdx.x == 0 && tid == 0) a.beta[a.k - 1] = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  if (tid == 0) {
    const double r = sh[0];
    const int ex = (__double2hiint(r) >> 20) & 0x7ff;
    double nr, rn;
    if (r > 0 && ex > 0 && ex < 2047) {
      rn = rsqrt_newton(r);
      nr = r * rn;
    } else {
      nr = sqrt(r);
      rn = 1.0 / nr;
    }
    s_rn = rn;
    if (blockIdx.x == 0) a.beta[a.k - 1] = nr;
  }
  __syncthreads();
  const double rn = s_rn;
  if (a.vnext)
    for (int e = tid; e < cnt; e += GS_THREADS) a.vnext[lo + e] = zscale(sw[e], rn);
}
}  // namespace

bool vec_gs_eligible(const Ctx* c, int64_t n) { return gs_fits(n, c->nsm); }

int vec_gs_reset(Ctx* c) {
  TNT_CUDA_TRY(c, cudaMemsetAsync(c->d_count + 16, 0, sizeof(unsigned), c->stream));
  c->gs_arrivals = 0;
  return TNT_OK;
}

int vec_gs_step(Ctx* c, const z* V, int k, const z* w, int64_t n, z* vnext, double* d_alpha, double* d_beta) {
  if (k < 1 || k > 64) return set_err(c, TNT_E_UNSUPPORTED, "Gram-Schmidt step with k = %d", k);
  const int nsm = c->nsm;
  TNT_TRY(func_smem(c, (const void*)k_gs_step, GS_SMEM));
  const size_t top = c->ws.top;
  z* part = (z*)ws_alloc(c, ws_round(sizeof(z) * 2 * 64 * (size_t)nsm));
  double* npart = (double*)ws_alloc(c, ws_round(sizeof(double) * 2 * (size_t)nsm));
  c->ws.top = top;  // used by this launch only (stream order serialises its reuse)
  if (!part || !npart) return set_err(c, TNT_E_ALLOC, "scratch exhausted (Gram-Schmidt step)");
  GsArgs a;
  a.V = V; a.n = n; a.k = k; a.w = w; a.vnext = vnext;
  a.alpha = d_alpha; a.beta = d_beta;
  a.part = part; a.npart = npart;
  a.bar = c->d_count + 16;
  a.base = c->gs_arrivals;
  a.status = c->d_status;
  a.S = (int)gs_slice(n, nsm);
  const int grid = (int)((n + a.S - 1) / a.S);
  c->gs_arrivals += 4u * (unsigned)grid;
  const size_t sw = sizeof(z) * (size_t)a.S, all = sw * (size_t)(k + 1);
  a.keep = all <= (size_t)GS_SMEM;
  const size_t smem = a.keep ? all : sw;
  if (smem > (size_t)GS_SMEM) return set_err(c, TNT_E_UNSUPPORTED, "Gram-Schmidt step with n = %lld", (long long)n);
  void* args[] = {&a};
  {
    ProfScope ps(c, "gs_step", (16.0 * (double)k + 38.0) * (double)n);  // FP64 FLOPs
    TNT_CUDA_TRY(c, cudaLaunchCooperativeKernel((void*)k_gs_step, dim3((unsigned)grid), dim3(GS_THREADS), args,
                                                smem, c->stream));
  }
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

// ============================================================ tridiagonal eigensolve
// Lowest eigenpair of the Lanczos matrix T (k <= 64), one warp per problem.  out[0] = E,
// out[1] = |y_{k-1}|.  On GB300 an FP64 instruction holds a sub-partition's FP64 pipe for 64
// clocks however few lanes are active, so what counts is the number of FP64 instructions in
// sequence:
//   * the lowest eigenvalue to ~1e-7 |T| by multisection on Sturm counts in FP32;
//   * Rayleigh quotient iteration from there (two or three rounds, cubic): the vector of the
//     shift by the three-term recurrences from both ends (lane 0 from the top, lane 1 from
//     the bottom, two FP64 instructions a row), joined at the row r whose residual
//     gamma_r = ((T - lam) y)_r is smallest, all rows' residuals and the norm in parallel;
//     the next shift is lam + gamma_r / |y|^2;
//   * the quotients of neighbouring entries are the pivots of the twisted factorisation of
//     T - lam: all of them (but gamma_r) positive says that no eigenvalue lies below, so the
//     pair found is the lowest.
// If that check or the convergence fails (a zero beta, eigenvalues closer than rounding), the
// pair comes from FP64 multisection and inverse iteration.  That form alone took 95 to 105
// us at k = 20..32, more than the rest of a small problem's Krylov step.
namespace {
// number of eigenvalues < x: sign changes of the leading principal minors
// p_i = (a_i - x) p_{i-1} - b_{i-1}^2 p_{i-2} (division-free Sturm sequence; a zero minor
// takes 2^-60 |p_{i-1}| with the sign opposite to its predecessor; the pair is rescaled
// by an exact power of two when its exponent leaves [-400, 400])
__device__ int sturm_count(const double* a, const double* b, int k, double x) {
  double pm2 = 1.0, pm1 = a[0] - x;
  if (pm1 == 0.0) pm1 = -0x1p-60;
  int neg_prev = __double2hiint(pm1) < 0;
  int cnt = neg_prev;
  for (int i = 1; i < k; ++i) {
    double p = fma(a[i] - x, pm1, -(b[i - 1] * b[i - 1]) * pm2);
    if (p == 0.0) p = neg_prev ? 0x1p-60 * fabs(pm1) : -0x1p-60 * fabs(pm1);
    const int neg = __double2hiint(p) < 0;
    cnt += neg != neg_prev;
    neg_prev = neg;
    pm2 = pm1;
    pm1 = p;
    const int ex = (__double2hiint(p) >> 20) & 0x7ff;
    if (ex > 1023 + 400 || ex < 1023 - 400) {
      const double f = ldexp(1.0, 1023 - ex);
      pm1 *= f;
      pm2 *= f;
    }
  }
  return cnt;
}

// FP64 multisection (33 sub-intervals per step) from the Gershgorin interval [lo, hi], then
// inverse iteration with a pivoted tridiagonal LU (lane 0)
__device__ __noinline__ void tridiag_bisect(const double* a, const double* b, int k, double lo, double hi,
                                            double* __restrict__ out, double* __restrict__ y) {
  const int l = threadIdx.x & 31;
  const double pad = 1e-12 * fmax(fabs(lo), fabs(hi)) + 1e-300;
  lo -= pad;
  hi += pad;
  for (int it = 0; it < 64; ++it) {
    double width = hi - lo;
    if (width <= 4.0 * 2.220446049250313e-16 * fmax(fabs(lo), fabs(hi)) || width <= 1e-300)
      break;
    double x = lo + width * (double)(l + 1) / 33.0;
    int cnt = sturm_count(a, b, k, x);
    unsigned m = __ballot_sync(0xffffffffu, cnt >= 1);
    // smallest lane whose point lies above the lowest eigenvalue
    int first = m ? (__ffs(m) - 1) : 32;
    double nlo = lo + width * (double)first / 33.0;
    double nhi = lo + width * (double)(first + 1) / 33.0;
    if (first == 32) nhi = hi;
    lo = nlo;
    hi = nhi;
  }
  if (l == 0) {
    const double lam = 0.5 * (lo + hi);
    // inverse iteration on (T - lam I) y = y_prev with partial pivoting
    double dl[64], dm[64], du[64], du2[64], v[64];
    int piv[64];
    for (int i = 0; i < k; ++i) v[i] = 1.0 / sqrt((double)k) * (1.0 + 0.01 * i);
    const double eps = 2.220446049250313e-16;
    double scale = 0;
    for (int i = 0; i < k; ++i) scale = fmax(scale, fabs(a[i]) + (i < k - 1 ? fabs(b[i]) : 0));
    scale = fmax(scale, 1e-300);
    // T - lam I = P L U once (the shift is the same for every sweep); pivots inverted once,
    // so the three solves multiply instead of divide (a full-warp FP64 division costs
    // several FP64-pipe issue slots per lane on GB300)
    for (int i = 0; i < k; ++i) {
      dm[i] = a[i] - lam;
      du[i] = (i < k - 1) ? b[i] : 0.0;
      dl[i] = (i < k - 1) ? b[i] : 0.0;
      du2[i] = 0.0;
      piv[i] = i;
    }
    for (int i = 0; i < k - 1; ++i) {  // LU with partial pivoting (tridiagonal, textbook gtsv)
      if (fabs(dm[i]) >= fabs(dl[i])) {
        if (fabs(dm[i]) < eps * scale) dm[i] = eps * scale;
        double f = dl[i] / dm[i];
        dl[i] = f;
        dm[i + 1] -= f * du[i];
        du2[i] = 0.0;
        piv[i] = i;
      } else {
        double f = dm[i] / dl[i];
        dm[i] = dl[i];
        dl[i] = f;
        double t = du[i];
        du[i] = dm[i + 1];
        dm[i + 1] = t - f * du[i];
        if (i < k - 2) {
          du2[i] = du[i + 1];
          du[i + 1] = -f * du[i + 1];
        }
        piv[i] = i + 1;
      }
    }
    if (fabs(dm[k - 1]) < eps * scale) dm[k - 1] = eps * scale;
    for (int i = 0; i < k; ++i) dm[i] = 1.0 / dm[i];  // inverse pivots
    for (int iter = 0; iter < 3; ++iter) {
      // forward: apply row swaps and L
      for (int i = 0; i < k - 1; ++i) {
        if (piv[i] == i) {
          v[i + 1] -= dl[i] * v[i];
        } else {
          double t = v[i];
          v[i] = v[i + 1];
          v[i + 1] = t - dl[i] * v[i];
        }
      }
      // backward: U has diagonals 1/dm, du, du2; the vector is scaled down whenever an
      // entry passes 2^500 (compounding pivots of near-degenerate Ritz values)
      for (int i = k - 1; i >= 0; --i) {
        double t = v[i];
        if (i + 1 < k) t -= du[i] * v[i + 1];
        if (i + 2 < k) t -= du2[i] * v[i + 2];
        t *= dm[i];
        v[i] = t;
        if (fabs(t) > 0x1p500)
          for (int q = 0; q < k; ++q) v[q] *= 0x1p-500;
      }
      double nrm = 0;
      for (int i = 0; i < k; ++i) nrm = fma(v[i], v[i], nrm);
      const double rn = 1.0 / sqrt(nrm);
      for (int i = 0; i < k; ++i) v[i] *= rn;
    }
    // fix the sign so that the first nonzero component is positive (deterministic)
    double sgn = 1.0;
    for (int i = 0; i < k; ++i)
      if (v[i] != 0.0) {
        sgn = v[i] > 0 ? 1.0 : -1.0;
        break;
      }
    for (int i = 0; i < k; ++i) y[i] = sgn * v[i];
    out[0] = lam;
    out[1] = fabs(v[k - 1]);
  }
}

// the vector of one shift: entries of the recurrences from the top (f) and from the bottom
// (h) with their powers of two, as (value, exponent); s_P, s_Q hold per row the factors of
// the two recurrences (top first)
struct TwistShared {
  double a[64], b[64];
  double P[2][64], Q[2][64];  // y_{i+1} = P y_i - Q y_{i-1} (top), y_{i-1} = P y_i - Q y_{i+1} (bottom)
  double v[2][64];
  int ex[2][64];
};

__device__ bool tridiag_twisted(TwistShared& S, int k, double lo, double hi, double* __restrict__ out,
                                double* __restrict__ y) {
  const int l = threadIdx.x & 31;
  const unsigned full = 0xffffffffu;
  const double width = hi - lo;
  if (!(width > 1e-290) || !(width < 1e290)) return false;
  // FP32 multisection on (T - lo) / width, eigenvalues in [0, 1]
  __shared__ float s_a[64], s_b2[64];
  {
    const double inv = 1.0 / width;
    bool bad = false;
    for (int i = l; i < k; i += 32) {
      s_a[i] = (float)((S.a[i] - lo) * inv);
      if (i < k - 1) {
        const float bf = (float)(S.b[i] * inv);
        s_b2[i] = bf * bf;
        bad |= !(fabs(S.b[i]) >= 1e-140 * width);
      }
    }
    if (__any_sync(full, bad)) return false;
  }
  __syncwarp();
  float xl = 0.f, xw = 1.f;
  for (int it = 0; it < 6 && xw > 6e-8f; ++it) {
    const float x = xl + xw * (float)(l + 1) * (1.f / 33.f);
    bool neg = false;
    float q = s_a[0] - x;
    for (int i = 1;; ++i) {
      if (fabsf(q) < 1e-20f) q = -1e-20f;
      neg |= q < 0.f;
      if (i >= k) break;
      q = s_a[i] - x - __fdividef(s_b2[i - 1], q);
    }
    const unsigned m = __ballot_sync(full, neg);
    const int first = m ? __ffs((int)m) - 1 : 32;
    xl += xw * (float)first * (1.f / 33.f);
    xw *= 1.f / 33.f;
  }
  double lam = lo + width * (double)(xl + 0.5f * xw);
  const double tiny = 4.0 * 2.220446049250313e-16 * fmax(fabs(lo), fabs(hi));
  // per row: 1 / b of the row's own and the previous off-diagonal
  double rb[2], rbm[2];
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int i = l + 32 * t;
    rb[t] = i < k - 1 ? 1.0 / S.b[i] : 0.0;
    rbm[t] = __shfl_up_sync(full, rb[t], 1);
    if (l == 0) rbm[t] = 0.0;
  }
  {  // row 32's previous off-diagonal is lane 31's first
    const double r31 = __shfl_sync(full, rb[0], 31);
    if (l == 0) rbm[1] = r31;
  }
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int i = l + 32 * t;
    if (i < k) {
      S.Q[0][i] = i > 0 ? S.b[i - 1] * rb[t] : 0.0;
      S.Q[1][i] = i < k - 1 ? S.b[i] * rbm[t] : 0.0;
    }
  }
  double gam = 0, nrm = 1;
  double yv[2] = {0, 0};
  bool done = false;
  for (int it = 0; it < 6; ++it) {
    __syncwarp();
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int i = l + 32 * t;
      if (i < k) {
        const double g = lam - S.a[i];
        S.P[0][i] = g * rb[t];
        S.P[1][i] = g * rbm[t];
      }
    }
    __syncwarp();
    if (l < 2) {  // lane 0 from the top, lane 1 from the bottom
      double y1 = 1.0, y0 = 0.0;  // the last two entries
      int ex = 0;
      int i = l ? k - 1 : 0;
      const int d = l ? -1 : 1;
      S.v[l][i] = 1.0;
      S.ex[l][i] = 0;
      for (int st = 1; st < k; ++st) {
        const double yn = fma(S.P[l][i], y1, -S.Q[l][i] * y0);
        i += d;
        y0 = y1;
        y1 = yn;
        const int e = (__double2hiint(yn) >> 20) & 0x7ff;
        if (e > 1023 + 300 || (e < 1023 - 300 && e > 0)) {  // exact scaling of the pair
          const double f = __hiloint2double((2046 - e) << 20, 0);
          y0 *= f;
          y1 *= f;
          ex += e - 1023;
        }
        S.v[l][i] = y1;
        S.ex[l][i] = ex;
      }
    }
    __syncwarp();
    // residual of the vector joined at row i, and the signs of the neighbours' quotients
    double gi[2];
    unsigned nf[2], nh[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int i = l + 32 * t;
      double g = 0;
      bool pf = false, ph = false;  // quotient f_{i+1} / f_i, h_{i-1} / h_i not of the right sign
      if (i < k) {
        g = S.a[i] - lam;
        const double f = S.v[0][i], h = S.v[1][i];
        if (i > 0) {
          const int e = S.ex[0][i - 1] - S.ex[0][i];
          const double q = S.v[0][i - 1] / f;
          g = fma(S.b[i - 1], e ? ldexp(q, e) : q, g);
          ph = !((S.v[1][i - 1] < 0) != ((h < 0) != (S.b[i - 1] < 0))) || S.v[1][i - 1] == 0.0;
        }
        if (i < k - 1) {
          const int e = S.ex[1][i + 1] - S.ex[1][i];
          const double q = S.v[1][i + 1] / h;
          g = fma(S.b[i], e ? ldexp(q, e) : q, g);
          pf = !((S.v[0][i + 1] < 0) != ((f < 0) != (S.b[i] < 0))) || S.v[0][i + 1] == 0.0;
        }
        if (!isfinite(g)) g = INFINITY;
      } else {
        g = INFINITY;
      }
      gi[t] = g;
      nf[t] = __ballot_sync(full, pf);
      nh[t] = __ballot_sync(full, ph);
    }
    // the row of the smallest residual: on the bits of |g| rounded to its upper half
    unsigned key = min(((unsigned)__double2hiint(fabs(gi[0])) & ~63u) | (unsigned)l,
                       ((unsigned)__double2hiint(fabs(gi[1])) & ~63u) | (unsigned)(l + 32));
    key = __reduce_min_sync(full, key);
    const int r = (int)(key & 63u);
    gam = __shfl_sync(full, r < 32 ? gi[0] : gi[1], r & 31);
    if (!isfinite(gam)) return false;
    const uint64_t F = ((uint64_t)nf[1] << 32) | nf[0], H = ((uint64_t)nh[1] << 32) | nh[0];
    const uint64_t below = r ? (~0ull >> (64 - r)) : 0ull;  // rows above the join
    const uint64_t above = r < 63 ? ~0ull << (r + 1) : 0ull;
    const bool lowest = (F & below) == 0 && (H & above) == 0;
    const double rf = 1.0 / S.v[0][r], rh = 1.0 / S.v[1][r];
    double s2 = 0;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int i = l + 32 * t;
      double v = 0;
      if (i < k) {
        const int o = i <= r ? 0 : 1;
        v = S.v[o][i] * (o ? rh : rf);
        const int e = S.ex[o][i] - S.ex[o][r];
        if (e) v = ldexp(v, e);
        if (i == r) v = 1.0;
      }
      yv[t] = v;
      s2 = fma(v, v, s2);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s2 += __shfl_xor_sync(full, s2, o);
    nrm = s2;
    if (!isfinite(nrm)) return false;
    const double step = gam / nrm;
    lam += step;
    if (fabs(step) <= tiny) {
      if (!lowest) return false;
      done = true;
      break;
    }
  }
  if (!done) return false;
  // |y| = 1, first non-zero entry positive
  const double rn = 1.0 / sqrt(nrm);
  const unsigned z0 = __ballot_sync(full, yv[0] != 0.0), z1 = __ballot_sync(full, yv[1] != 0.0);
  const double first = z0 ? __shfl_sync(full, yv[0], __ffs((int)z0) - 1) : __shfl_sync(full, yv[1], z1 ? __ffs((int)z1) - 1 : 0);
  const double sc = first < 0 ? -rn : rn;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    const int i = l + 32 * t;
    if (i < k) {
      y[i] = yv[t] * sc;
      if (i == k - 1) out[1] = fabs(yv[t] * sc);
    }
  }
  if (l == 0) out[0] = lam;
  return true;
}

// one block per problem: problem p's alpha, beta, y at p * 64, out at p * 2 (skipped
// where skip[p] is set); a single problem's E, |y_{k-1}|, beta_{k-1} and the status word also to
// pinned host memory (no copy on the stream behind the kernel)
__global__ void __launch_bounds__(32) k_tridiag_lowest(const double* __restrict__ alpha,
                                                       const double* __restrict__ beta, int k,
                                                       double* out, double* __restrict__ y,
                                                       const int* __restrict__ skip, const int* status,
                                                       KrylovSlot* host) {
  const int pb = blockIdx.x;
  if (skip && skip[pb]) return;
  alpha += 64 * pb;
  beta += 64 * pb;
  out += 2 * pb;
  y += 64 * pb;
  __shared__ TwistShared S;
  const int l = threadIdx.x;
  for (int i = l; i < k; i += 32) S.a[i] = alpha[i];
  for (int i = l; i < k - 1; i += 32) S.b[i] = beta[i];
  __syncwarp();
  // Gershgorin interval
  double lo = INFINITY, hi = -INFINITY;
  for (int i = l; i < k; i += 32) {
    const double r = (i > 0 ? fabs(S.b[i - 1]) : 0.0) + (i < k - 1 ? fabs(S.b[i]) : 0.0);
    lo = fmin(lo, S.a[i] - r);
    hi = fmax(hi, S.a[i] + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (!tridiag_twisted(S, k, lo, hi, out, y)) tridiag_bisect(S.a, S.b, k, lo, hi, out, y);
  if (host) {
    __syncwarp();
    if (l == 0) host->E = out[0];
    if (l == 1) host->ylast = out[1];
    if (l == 2) host->beta = beta[k - 1];
    if (l == 3) host->status = (double)*status;
  }
}
}  // namespace

int tridiag_lowest_on(Ctx* c, cudaStream_t st, const double* d_alpha, const double* d_beta, int k,
                      double* d_out, double* d_y, KrylovSlot* h_out) {
  if (k < 1 || k > 64) return set_err(c, TNT_E_UNSUPPORTED, "tridiagonal size %d", k);
  k_tridiag_lowest<<<1, 32, 0, st>>>(d_alpha, d_beta, k, d_out, d_y, nullptr, c->d_status, h_out);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int side_stream(Ctx* c) {
  if (c->side) return TNT_OK;
  TNT_CUDA_TRY(c, cudaStreamCreateWithFlags(&c->side, cudaStreamNonBlocking));
  for (int i = 0; i < 2; ++i) {
    TNT_CUDA_TRY(c, cudaEventCreateWithFlags(&c->ev_main[i], cudaEventDisableTiming));
    TNT_CUDA_TRY(c, cudaEventCreateWithFlags(&c->ev_side[i], cudaEventDisableTiming));
  }
  return TNT_OK;
}

int tridiag_lowest_batched(Ctx* c, const double* d_alpha, const double* d_beta, int k,
                           double* d_out, double* d_y, int nprob, const int* d_skip) {
  if (k < 1 || k > 64) return set_err(c, TNT_E_UNSUPPORTED, "tridiagonal size %d", k);
  k_tridiag_lowest<<<nprob, 32, 0, c->stream>>>(d_alpha, d_beta, k, d_out, d_y, d_skip, nullptr, nullptr);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

// ============================================================ fill / scale
namespace {
__global__ void k_zfill(z* p, int64_t n, z v) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    p[e] = v;
}

// mode 0: p *= s[0]; mode 1: p *= 1/sqrt(s[0])
__global__ void k_zscale(z* p, int64_t n, const double* s, int mode) {
  __shared__ double s_f;  // by one thread, as in k_normalize
  if (threadIdx.x == 0) s_f = (mode == 0) ? s[0] : 1.0 / sqrt(s[0]);
  __syncthreads();
  const double f = s_f;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x)
    p[e] = zscale(p[e], f);
}

unsigned grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b > 152 * 8) b = 152 * 8;
  if (b < 1) b = 1;
  return (unsigned)b;
}
}  // namespace

int zfill(Ctx* c, z* p, int64_t n, z v) {
  if (n <= 0) return TNT_OK;
  k_zfill<<<grid_for(n), 256, 0, c->stream>>>(p, n, v);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

int zscale_inplace(Ctx* c, z* p, int64_t n, const double* d_scale, int mode) {
  if (n <= 0) return TNT_OK;
  k_zscale<<<grid_for(n), 256, 0, c->stream>>>(p, n, d_scale, mode);
  c->launches++;
  TNT_CHECK_LAUNCH(c);
  return TNT_OK;
}

}  // namespace tnt
