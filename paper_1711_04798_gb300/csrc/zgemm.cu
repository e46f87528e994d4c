// Complex FP64 GEMM on the CUDA cores (the plain-FP64 path of the CTM
// contractions) and the generic index permutation that feeds it.
#include <cooperative_groups.h>

#include "ctm_internal.h"

#include <atomic>

static std::atomic<uint64_t> g_launches{0};
void count_launch(int n) { g_launches += (uint64_t)n; }
uint64_t launch_counter() { return g_launches.load(); }

namespace cg = cooperative_groups;

namespace {

constexpr int BK = 16;
constexpr cplx ONE_C = {1.0, 0.0};
constexpr cplx ZERO_C = {0.0, 0.0};

__device__ __forceinline__ cplx ld_op(const cplx* p, bool cj) {
  cplx v = *p;
  if (cj) v.y = neg_bits(v.y);
  return v;
}

// T x T output tile per CTA of 256 threads, each thread MI x MI outputs (T =
// 16 MI) strided by 16 so that shared-memory reads are broadcast /
// conflict-free.  The FP64 units bound every tile (about 1.75 multiply-adds
// per cycle and SM; even MI = 1 needs only 2 shared loads for the 4 that hold
// the SM's units for some 70 cycles), so the tile only sets how evenly the
// product covers the SMs and how much of it is padding: a 32 x 32 tile with K =
// 64 is 70 us of one SM's FP64 time.
// FUSED (MI = 1): the K splits of a tile are the CTAs of a cluster, whose sums meet
// in shared memory, in split order, without a second kernel.
template <int MI, bool FUSED = false>
__global__ void __launch_bounds__(256) zgemm_kernel(int M, int N, int K, cplx alpha, const cplx* __restrict__ A,
                                                    long long lda, int opA, const cplx* __restrict__ B,
                                                    long long ldb, int opB, cplx beta, cplx* __restrict__ C,
                                                    long long ldc, long long sA, long long sB, long long sC,
                                                    int ksplit, int flags) {
  constexpr int T = 16 * MI, NT = 256;
  __shared__ cplx As[BK][T + 1];
  __shared__ cplx Bs[BK][T + 1];
  const long long bz = blockIdx.z;
  const int m0 = blockIdx.y * T, n0 = blockIdx.x * T;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  if ((flags & ZG_UPPER_TILES) && blockIdx.y > blockIdx.x) {  // tile below the diagonal: not needed
    if (FUSED && blockIdx.z == 0 && m0 + ty < M && n0 + tx < N) C[(long long)(m0 + ty) * ldc + n0 + tx] = ZERO_C;
    return;
  }
  const bool tA = opA & OP_T, cA = opA & OP_CONJ;
  const bool tB = opB & OP_T, cB = opB & OP_CONJ;
  if (ksplit > 0) {
    // split-K: entry z sums k in [z*ksplit, min(K, (z+1)*ksplit)) into its own C slice
    const long long kb = bz * (long long)ksplit;
    A += tA ? kb * lda : kb;
    B += tB ? kb : kb * ldb;
    K = (int)min((long long)ksplit, (long long)K - kb);
    if (flags & ZG_A_LOWER) K = (int)max(0LL, min((long long)K, (long long)(m0 + T) - kb));
    if (!FUSED) C += bz * sC;
  } else {
    if (flags & ZG_A_LOWER) K = min(K, m0 + T);  // A[m, k] = 0 for k > m: later k-tiles add nothing
    A += bz * sA;
    B += bz * sB;
    C += bz * sC;
  }
  double cr[MI][MI], ci[MI][MI];
#pragma unroll
  for (int i = 0; i < MI; ++i)
#pragma unroll
    for (int j = 0; j < MI; ++j) cr[i][j] = ci[i][j] = 0.0;

  auto step = [&](int kk) {
    cplx a[MI], b[MI];
#pragma unroll
    for (int i = 0; i < MI; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
    for (int j = 0; j < MI; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
      for (int j = 0; j < MI; ++j) {
        cr[i][j] = fma(a[i].x, b[j].x, cr[i][j]);
        cr[i][j] = fma(-a[i].y, b[j].y, cr[i][j]);
        ci[i][j] = fma(a[i].x, b[j].y, ci[i][j]);
        ci[i][j] = fma(a[i].y, b[j].x, ci[i][j]);
      }
  };
  for (int k0 = 0; k0 < K; k0 += BK) {
    for (int e = threadIdx.x; e < T * BK; e += NT) {
      int mm, kk;
      if (tA) { mm = e % T; kk = e / T; } else { kk = e % BK; mm = e / BK; }
      const int m = m0 + mm, k = k0 + kk;
      cplx v = make_double2(0.0, 0.0);
      if (m < M && k < K) v = ld_op(tA ? A + (long long)k * lda + m : A + (long long)m * lda + k, cA);
      As[kk][mm] = v;
    }
    for (int e = threadIdx.x; e < T * BK; e += NT) {
      int nn, kk;
      if (tB) { kk = e % BK; nn = e / BK; } else { nn = e % T; kk = e / T; }
      const int n = n0 + nn, k = k0 + kk;
      cplx v = make_double2(0.0, 0.0);
      if (n < N && k < K) v = ld_op(tB ? B + (long long)n * ldb + k : B + (long long)k * ldb + n, cB);
      Bs[kk][nn] = v;
    }
    __syncthreads();
    if (K - k0 >= BK) {
#pragma unroll 4
      for (int kk = 0; kk < BK; ++kk) step(kk);
    } else {  // no FP64 work for the padding of a short last k-tile
      for (int kk = 0; kk < K - k0; ++kk) step(kk);
    }
    __syncthreads();
  }
  const bool use_beta = (beta.x != 0.0 || beta.y != 0.0);
  if constexpr (FUSED) {
    cg::cluster_group cl = cg::this_cluster();
    const int S = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    cplx* tile = &As[0][0];  // 256 sums; the last k-tile's reads ended at a block barrier
    tile[threadIdx.x] = make_double2(cr[0][0], ci[0][0]);
    cl.sync();
    const int per = (256 + S - 1) / S, e = rank * per + threadIdx.x;
    const int m = m0 + e / 16, n = n0 + e % 16;
    if (threadIdx.x < per && e < 256 && m < M && n < N) {
      double r = 0.0, i = 0.0;
      for (int z = 0; z < S; ++z) {
        const cplx v = cl.map_shared_rank(tile, z)[e];
        r += v.x;
        i += v.y;
      }
      cplx* cp = C + (long long)m * ldc + n;
      double orr = alpha.x * r - alpha.y * i, oi = alpha.x * i + alpha.y * r;
      if (use_beta) {
        const cplx o = *cp;
        orr += beta.x * o.x - beta.y * o.y;
        oi += beta.x * o.y + beta.y * o.x;
      }
      *cp = make_double2(orr, oi);
    }
    cl.sync();  // no CTA leaves while another reads its sums
    return;
  }
#pragma unroll
  for (int i = 0; i < MI; ++i) {
    const int m = m0 + ty + 16 * i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < MI; ++j) {
      const int n = n0 + tx + 16 * j;
      if (n >= N) continue;
      cplx* cp = C + (long long)m * ldc + n;
      double r = alpha.x * cr[i][j] - alpha.y * ci[i][j];
      double im = alpha.x * ci[i][j] + alpha.y * cr[i][j];
      if (use_beta) {
        const cplx o = *cp;
        r += beta.x * o.x - beta.y * o.y;
        im += beta.x * o.y + beta.y * o.x;
      }
      *cp = make_double2(r, im);
    }
  }
}

// C = alpha * sum_z W[z] (+ beta C), fixed summation order
__global__ void splitk_sum_kernel(const cplx* __restrict__ W, int S, int M, int N, cplx alpha, cplx beta,
                                  cplx* __restrict__ C, long long ldc, int flags, int tm, int tn) {
  const long long total = (long long)M * N;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    if ((flags & ZG_UPPER_TILES) && ((int)(e / N)) / tm > ((int)(e % N)) / tn) {
      C[(long long)(e / N) * ldc + (e % N)] = make_double2(0.0, 0.0);  // tile not computed
      continue;
    }
    double r = 0.0, im = 0.0;
    for (int z = 0; z < S; ++z) {
      r += W[z * total + e].x;
      im += W[z * total + e].y;
    }
    const int m = (int)(e / N), n = (int)(e % N);
    cplx* cp = C + (long long)m * ldc + n;
    double orr = alpha.x * r - alpha.y * im, oi = alpha.x * im + alpha.y * r;
    if (beta.x != 0.0 || beta.y != 0.0) {
      const cplx o = *cp;
      orr += beta.x * o.x - beta.y * o.y;
      oi += beta.x * o.y + beta.y * o.x;
    }
    *cp = make_double2(orr, oi);
  }
}

struct PermParams {
  int nd;
  long long odims[8];
  long long istr[8];
};

template <typename Idx>
__global__ void permute_kernel(const cplx* __restrict__ in, cplx* __restrict__ out,
                               long long total, PermParams p, int conj, cplx alpha, int unit) {
  for (Idx i = (Idx)blockIdx.x * (Idx)blockDim.x + threadIdx.x; i < (Idx)total; i += (Idx)gridDim.x * blockDim.x) {
    Idx r = i, off = 0;
    for (int a = p.nd - 1; a >= 0; --a) {
      const Idx d = (Idx)p.odims[a];
      const Idx q = r / d;
      off += (r - q * d) * (Idx)p.istr[a];
      r = q;
    }
    cplx v = in[off];
    if (conj) v.y = neg_bits(v.y);
    if (unit) {
      out[i] = v;  // no FP64 arithmetic for the usual alpha = 1
    } else {
      out[i] = make_double2(alpha.x * v.x - alpha.y * v.y, alpha.x * v.y + alpha.y * v.x);
    }
  }
}

}  // namespace

// Tile size and K split from a cost model, in microseconds: the busiest SM's
// share of the multiply-adds at the FP64 units' rate (a k step of a 64 x 64 tile
// takes them 4.5 us; 0.61 of the rate with one CTA on the SM, measured on GB300,
// its loads not hidden), a load latency (1 us) for each of its k-tiles as far as
// other CTAs do not cover it, and for a split the second kernel with the
// partials' round trip.  ksplit: k per split, 0 = unsplit (no minimum there: with
// the splits' minimum of 8 on it too, every product of K < 8 fell to 64-wide tiles,
// 1024 x 32 x 4 to 16 CTAs and 23 us).  For sums that short a narrow tile has to
// be the better one by its waves: where all widths fill the chip, each CTA's
// start and stores count for more than the model's latency term.
void zgemm_plan(int M, int N, int K, int count, long long work_elems, int flags, int* tile, int* ksplit) {
  *tile = 64;
  *ksplit = 0;
  double best_cost = -1.0;
  const bool can_split = count == 1 && K >= 16;
  for (int T : {64, 32, 16}) {
    if (T != 64 && (count != 1 || M > 65535LL * T)) continue;
    const long long tm = (M + T - 1) / T, tn = (N + T - 1) / T;
    const double per_k = 4.5 * (T / 64.0) * (T / 64.0);
    int last = -1;
    for (int S = 1; S <= (can_split ? 160 : 1); ++S) {
      const int kps = S == 1 ? K : ((K + S - 1) / S + 7) / 8 * 8;
      if ((S > 1 && kps < 8) || kps == last) continue;
      last = kps;
      const long long Se = (K + kps - 1) / kps;
      if (Se > 1 && Se * M * N > work_elems && !(T == 16 && Se <= 8)) continue;
      // an unsplit product computes the tiles below the diagonal too
      const long long tiles = Se > 1 && (flags & ZG_UPPER_TILES) ? tm * (tm + 1) / 2 : tm * tn;
      const long long busy = (tiles * Se * count + 151) / 152;
      const double rate = busy == 1 ? 0.61 : 1.0;
      double cost = (double)kps * (double)busy * per_k / rate + (double)((kps + BK - 1) / BK) / (double)busy;
      // up to eight splits of 16-wide tiles meet in a cluster's shared memory
      // (1.5 us), others in a second kernel with the partials' round trip
      const bool fused = T == 16 && Se > 1 && Se <= 8;
      if (fused)
        cost += 1.5;
      else if (Se > 1)
        cost += 4.0 + (double)Se * (double)M * (double)N * 32.0 / 5e6;
      if (best_cost < 0.0 || cost < best_cost * (K < 8 ? 0.95 : 1.0)) {
        best_cost = cost;
        *ksplit = Se > 1 ? kps : 0;
        *tile = T;
      }
    }
  }
}

cudaError_t zgemm(cudaStream_t s, int M, int N, int K, cplx alpha, const cplx* A, long long lda,
                  int opA, const cplx* B, long long ldb, int opB, cplx beta, cplx* C,
                  long long ldc, GemmBatch batch, cplx* work, long long work_elems, int flags) {
  if (M <= 0 || N <= 0 || batch.count <= 0) return cudaSuccess;
  if ((flags & ZG_UPPER_TILES) && M != N) return cudaErrorInvalidValue;
  int T, best_k;
  zgemm_plan(M, N, K, batch.count, work_elems, flags, &T, &best_k);
  const long long tm = (M + T - 1) / T, tn = (N + T - 1) / T;
  auto launch = [&](dim3 grid, cplx al, cplx be, cplx* out, long long ldo, long long sC, int ksplit, int fl) {
    auto go = [&](auto kern) {
      kern<<<grid, 256, 0, s>>>(M, N, K, al, A, lda, opA, B, ldb, opB, be, out, ldo, batch.sA, batch.sB, sC, ksplit,
                                fl);
    };
    if (T == 64)
      go(zgemm_kernel<4>);
    else if (T == 32)
      go(zgemm_kernel<2>);
    else
      go(zgemm_kernel<1>);
  };
  if (tm > 65535) return cudaErrorInvalidConfiguration;
  if (best_k > 0) {
    const long long S = (K + best_k - 1) / best_k;
    if (T == 16 && S <= 8) {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr;
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = 1;
      attr.val.clusterDim.y = 1;
      attr.val.clusterDim.z = (unsigned)S;
      cfg.gridDim = dim3((unsigned)tn, (unsigned)tm, (unsigned)S);
      cfg.blockDim = dim3(256);
      cfg.stream = s;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      const cudaError_t e = cudaLaunchKernelEx(&cfg, zgemm_kernel<1, true>, M, N, K, alpha, A, lda, opA, B, ldb, opB,
                                               beta, C, ldc, 0LL, 0LL, 0LL, best_k, flags);
      count_launch();
      return e;
    }
    launch(dim3((unsigned)tn, (unsigned)tm, (unsigned)S), ONE_C, ZERO_C, work, N, (long long)M * N, best_k, flags);
    long long blocks = ((long long)M * N + 255) / 256;
    if (blocks > 152 * 16) blocks = 152 * 16;
    splitk_sum_kernel<<<(unsigned)blocks, 256, 0, s>>>(work, (int)S, M, N, alpha, beta, C, ldc, flags, T, T);
    count_launch(2);
    return cudaGetLastError();
  }
  if (flags & ZG_UPPER_TILES) flags &= ~ZG_UPPER_TILES;  // unsplit: full tiles (lower ones are cheap here)
  dim3 grid((unsigned)tn, (unsigned)tm, batch.count);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidConfiguration;
  launch(grid, alpha, beta, C, ldc, batch.sC, 0, flags);
  count_launch();
  return cudaGetLastError();
}

cudaError_t permute(cudaStream_t s, const cplx* in, cplx* out, int nd, const int* in_dims,
                    const int* perm, bool conj, cplx alpha) {
  if (nd < 1 || nd > 8) return cudaErrorInvalidValue;
  PermParams p;
  p.nd = nd;
  long long istride[8];
  long long acc = 1;
  for (int a = nd - 1; a >= 0; --a) {
    istride[a] = acc;
    acc *= in_dims[a];
  }
  // output axes that stay adjacent and in order in the input merge into one
  // (fewer divisions per element)
  p.nd = 0;
  for (int i = 0; i < nd; ++i) {
    if (p.nd > 0 && perm[i] == perm[i - 1] + 1) {
      p.odims[p.nd - 1] *= in_dims[perm[i]];
      p.istr[p.nd - 1] = istride[perm[i]];
    } else {
      p.odims[p.nd] = in_dims[perm[i]];
      p.istr[p.nd] = istride[perm[i]];
      ++p.nd;
    }
  }
  const long long total = acc;
  if (total == 0) return cudaSuccess;
  long long blocks = (total + 255) / 256;
  if (blocks > 152 * 32) blocks = 152 * 32;
  const int unit = alpha.x == 1.0 && alpha.y == 0.0;
  if (total < (1LL << 31))  // 32-bit index arithmetic (offsets are below total)
    permute_kernel<unsigned><<<(unsigned)blocks, 256, 0, s>>>(in, out, total, p, conj ? 1 : 0, alpha, unit);
  else
    permute_kernel<unsigned long long><<<(unsigned)blocks, 256, 0, s>>>(in, out, total, p, conj ? 1 : 0, alpha,
                                                                         unit);
  count_launch();
  return cudaGetLastError();
}
