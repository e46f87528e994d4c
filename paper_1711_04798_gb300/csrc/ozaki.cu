// FP64-accurate complex GEMM on the tcgen05 tensor cores.
//
// GB300 runs FP64 at a small fraction of its tensor-core rate, so the FP64
// products of the projector step (CholeskyQR Grams and applies of k x K
// matrices), and in the FP64-accurate form every contraction product, are
// computed here by exact splitting into integer digit planes,
// after the error-free splitting of Ozaki, Ogita, Oishi and Rump (2012),
// arranged for BF16 tensor cores with FP32 accumulation:
//
//  * the complex product is the real product of the embedding of tc_gemm.cu:
//    Ar (M x 2K) and Br^T (2N x 2K), both K-major;
//  * every row r of Ar and of Br^T gets a power-of-two bound 2^e_r above its
//    largest magnitude, and each element is rounded to 55 fraction bits below
//    it, x = 2^e_r sum_{s<7} d_s 2^(-7-8s), with balanced base-256 digits d_s
//    in [-128, 128] (exact in BF16), taken from the FP64 bit pattern with
//    integer operations;
//  * the digit-plane products P_st = sum_k dA_s dB_t are sums of integers below
//    2^14 in magnitude; those of equal weight g = s + t accumulate in one FP32
//    accumulator, and over a chunk of 128 reals of K a group (at most 7 pairs)
//    stays below 2^24, so the tensor cores' FP32 sums are exact.  The 28
//    pairs with s + t <= 6 are computed; the others weigh below 2^-53 of the
//    terms' scale;
//  * after each chunk the seven group sums leave tensor memory: groups 0..3
//    combine exactly in 64-bit integers, I += 2^24 P_0 + 2^16 P_1 + 2^8 P_2 +
//    P_3 (below 2^49 per chunk), groups 4..6 (weight 2^-32 and below) in FP32,
//    u += P_4 + 2^-8 (P_5 + 2^-8 P_6), whose rounding weighs below 2^-56;
//  * Cr = 2^(ea + eb - 38) (I + 2^-8 u): the only rounding to FP64 is the last.
//
// The error is that of the 55-bit rounding of each element relative to its
// row's bound (and the dropped digit pairs), i.e. relative to max|a| max|b|
// of the rows involved rather than to sum |a||b|: FP64-level for rows
// without a wide spread of magnitudes, as the projector step's are.
//
// One CTA computes a 128 x 32 or 128 x 64 tile of Cr over a range of K
// chunks: warp 0 issues the TMA loads (per stage a k-block of all planes of
// both operands), warp 1 the tcgen05.mma, the other warps (four or
// eight) drain the seven group accumulators after each chunk.  Ranges of K
// are split over the grid; the exact partials (I, u) are summed by a second
// kernel.
#include <cuda_bf16.h>

#include "tc_gemm.h"
#include "tc_ptx.h"

namespace {

constexpr int OZ_DIGITS = 7;                          // base-256 digits per element
constexpr int OZ_GROUPS = 7;                          // weights g = s + t = 0..6
constexpr int OZ_BM = 128;                            // output tile rows
constexpr int OZ_BK = 32;                             // bf16 elements per k-block
constexpr int OZ_KB_BYTES = 2 * OZ_BK;                // 64-byte rows, 64-byte swizzle
constexpr int OZ_CHUNK = 128;                         // reals of K per exact FP32 chunk
constexpr int OZ_KB_PER_CHUNK = OZ_CHUNK / OZ_BK;     // 4
constexpr int OZ_A_BYTES = OZ_BM * OZ_KB_BYTES;       // one A plane k-block: 8 KB
constexpr int OZ_TMEM_COLS = 512;
static_assert(OZ_GROUPS == OZ_DIGITS, "weights 0..6 of the digit pairs s + t <= 6");

// Output tiles of 128 x BN real columns.  A pipeline stage holds a k-block of
// all seven planes of both operands, so that each plane is loaded once per
// tile and k-block (a stage per A plane with the B planes it meets loaded the
// B planes four times over: 672 KB per 128-wide chunk and SM through L2, which
// bound the 64-wide tile at 15 us a chunk).  BN = 32: two sets of the seven
// group accumulators (224 of 256 columns each), so that a chunk's products run
// while the epilogue drains the previous chunk; three 70 KB stages; four
// epilogue warps.  BN = 64: one set (448 columns), the products of a chunk
// wait for the previous chunk's drain, but each MMA does twice the work; two
// 84 KB stages; eight epilogue warps (two per lane quarter, 32 columns each).
template <int BN>
struct OzTile {
  static constexpr int B_BYTES = BN * OZ_KB_BYTES;                   // one B plane k-block
  static constexpr int STAGE = OZ_DIGITS * (OZ_A_BYTES + B_BYTES);  // 70 KB / 84 KB
  static constexpr int STAGES = BN == 32 ? 3 : 2;
  static constexpr int SETS = BN == 32 ? 2 : 1;
  static constexpr int ACC_COLS = BN == 32 ? 256 : 512;          // columns per accumulator set
  static constexpr int EPI_WARPS = BN / 8;
  static constexpr int THREADS = 64 + 32 * EPI_WARPS;            // producer, MMA issuer, epilogue
  static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                    ((uint32_t)(OZ_BM >> 4) << 24);  // FP32 += BF16 x BF16, K-major
  static_assert(OZ_GROUPS * BN <= ACC_COLS && SETS * ACC_COLS <= OZ_TMEM_COLS, "accumulators fit");
  static_assert(SMEM <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void umma_bf16(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc,
                                          uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accum)
      : "memory");
}

// The same MMA with the A operand kept in the tensor core's collector buffer
// across consecutive MMAs that share it: FILL reads A from shared memory and
// keeps it, USE takes the kept A, LAST takes it and releases the buffer.
enum { COLL_FILL = 1, COLL_USE = 2, COLL_LAST = 3 };
template <int COLL>
__device__ __forceinline__ void umma_bf16_coll(uint32_t dtmem, uint64_t a, uint64_t b, uint32_t idesc,
                                               uint32_t accum) {
  if constexpr (COLL == COLL_FILL)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
  else if constexpr (COLL == COLL_USE)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n}\n" ::"r"(dtmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum)
        : "memory");
}

// 2^k for k in the normal range, built from its bit pattern
__device__ __forceinline__ double pow2(int k) {
  k = k < -1022 ? -1022 : (k > 1023 ? 1023 : k);
  return __longlong_as_double((long long)(k + 1023) << 52);
}

// biased binary64 exponent of x (0 for zero and subnormals)
__device__ __forceinline__ int bexp(double x) { return (int)((__double_as_longlong(x) >> 52) & 0x7FF); }

// balanced base-256 digits of x / 2^e (|x| < 2^e), rounded to 55 fraction bits:
// x = 2^e sum_s d[s] 2^(-7-8s), d[s] in [-128, 128]
__device__ __forceinline__ void digits7(double x, int e, int (&d)[OZ_DIGITS]) {
  const long long b = __double_as_longlong(x);
  const int E = (int)((b >> 52) & 0x7FF);
  long long v = 0;
  if (E != 0) {
    const long long m = (b & 0xFFFFFFFFFFFFFLL) | (1LL << 52);
    const int shift = (E - 1023) - e + 3;  // v = x 2^(55 - e) = m 2^shift, shift <= 2
    if (shift >= 0)
      v = m << shift;
    else if (shift > -60)
      v = (m + (1LL << (-shift - 1))) >> (-shift);
    if (b < 0) v = -v;
  }
#pragma unroll
  for (int s = OZ_DIGITS - 1; s >= 1; --s) {
    const int dd = (int)(((v + 128) & 255) - 128);
    d[s] = dd;
    v = (v - dd) >> 8;  // exact: v - dd is a multiple of 256
  }
  d[0] = (int)v;
}

__device__ __forceinline__ cplx oz_load(const cplx* X, long long ld, int op, int r, int c) {
  // element (r, c) of op(X)
  cplx v = (op & OP_T) ? X[(long long)c * ld + r] : X[(long long)r * ld + c];
  if (op & OP_CONJ) v.y = -v.y;
  return v;
}

// The power-of-two bound of a row (or column) whose largest biased exponent is E:
// 0 for zeros; OZ_NONFINITE with an infinity or a NaN among them, which leaves the
// digits zero and makes every output of the row NaN (oz_value).
constexpr int OZ_NONFINITE = 1 << 20;
__device__ __forceinline__ int row_bound(int E) { return E == 0x7FF ? OZ_NONFINITE : (E ? E - 1022 : 0); }

// Both operands' exponents and digit planes in one launch.  Block b < Mp takes
// row b of op(A) (M x K complex): e = (largest biased exponent of the row) -
// 1022, the power-of-two bound of that row of Ar (0 for rows at or beyond M
// and for zero rows), and digit plane s of Ar is [Mp x Krp] bf16 at
// pa + s * Mp * Krp.  Block Mp + n takes column n of op(B) (K x N) the same
// way: its bound goes to rows 2n and 2n+1 of Br^T, and complex (k, n) gives
// row 2n (Re, -Im) and row 2n+1 (Im, Re) at columns 2k, 2k+1 of each plane of
// Br^T [Nrp x Krp].  The block first reduces the row's largest exponent, then
// writes its digits; the row is read twice, the second time from cache.
// WARP: a warp per row, four rows to a block, for many short rows (a block's
// start and its two barriers took longer than the at most four elements per
// lane: 19456 rows of 27 took 38 us, 18 us so).
constexpr int OZ_PREP_THREADS = 128;
template <bool WARP>
__global__ void __launch_bounds__(OZ_PREP_THREADS)
    oz_prep_kernel(const cplx* __restrict__ A, long long lda, int opA, const cplx* __restrict__ B, long long ldb,
                   int opB, int M, int N, int K, int Mp, int Nrp, int Krp, int* __restrict__ ea, int* __restrict__ eb,
                   __nv_bfloat16* __restrict__ pa, __nv_bfloat16* __restrict__ pb) {
  __shared__ int s_e[OZ_PREP_THREADS / 32];
  constexpr int NT = WARP ? 32 : OZ_PREP_THREADS;
  const int row = WARP ? (int)blockIdx.x * (OZ_PREP_THREADS / 32) + (int)(threadIdx.x >> 5) : (int)blockIdx.x;
  const int tid = WARP ? threadIdx.x & 31 : threadIdx.x;
  if (WARP && row >= Mp + Nrp / 2) return;
  const bool is_a = row < Mp;
  const int r = is_a ? row : row - Mp;  // row of op(A), or column of op(B)
  const bool live = is_a ? r < M : r < N;
  auto load = [&](int c) {
    return is_a ? oz_load(A, lda, opA, r, c) : oz_load(B, ldb, opB, c, r);
  };
  int E = 0;
  if (live)
    for (int c = tid; c < K; c += NT) {
      const cplx v = load(c);
      E = max(E, max(bexp(v.x), bexp(v.y)));
    }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if constexpr (!WARP) {
    if ((threadIdx.x & 31) == 0) s_e[threadIdx.x >> 5] = E;
    __syncthreads();
    E = s_e[0];
#pragma unroll
    for (int w = 1; w < OZ_PREP_THREADS / 32; ++w) E = max(E, s_e[w]);
  }
  const int e = row_bound(E);
  if (tid == 0) {
    if (is_a)
      ea[r] = e;
    else
      eb[2 * r] = eb[2 * r + 1] = e;
  }
  const long long kc = Krp / 2;
  const long long plane = is_a ? (long long)Mp * Krp : (long long)Nrp * Krp;
  for (int c = tid; c < kc; c += NT) {
    cplx v = make_double2(0.0, 0.0);
    if (live && c < K) v = load(c);
    int dr[OZ_DIGITS], di[OZ_DIGITS];
    digits7(v.x, e, dr);
    digits7(v.y, e, di);
    if (is_a) {
      __nv_bfloat162* out = (__nv_bfloat162*)(pa + (long long)r * Krp + 2LL * c);
#pragma unroll
      for (int s = 0; s < OZ_DIGITS; ++s)
        out[s * plane / 2] = __halves2bfloat162(__float2bfloat16_rn((float)dr[s]), __float2bfloat16_rn((float)di[s]));
    } else {
      __nv_bfloat162* r0 = (__nv_bfloat162*)(pb + (long long)(2 * r) * Krp + 2LL * c);
      __nv_bfloat162* r1 = (__nv_bfloat162*)(pb + (long long)(2 * r + 1) * Krp + 2LL * c);
#pragma unroll
      for (int s = 0; s < OZ_DIGITS; ++s) {
        const __nv_bfloat16 re = __float2bfloat16_rn((float)dr[s]), im = __float2bfloat16_rn((float)di[s]);
        r0[s * plane / 2] = __halves2bfloat162(re, __float2bfloat16_rn((float)-di[s]));
        r1[s * plane / 2] = __halves2bfloat162(im, re);
      }
    }
  }
}

// Cr element from its exact sums: 2^(ea + eb - 38) (I + 2^-8 u), NaN where a
// bound is OZ_NONFINITE
__device__ __forceinline__ double oz_value(long long I, float u, int ea, int eb) {
  if (ea + eb > OZ_NONFINITE / 2) return __longlong_as_double(0x7FF8000000000000LL);
  return ((double)I + (double)u * (1.0 / 256.0)) * pow2(ea + eb - 38);
}

template <int BN>
__global__ void __launch_bounds__(OzTile<BN>::THREADS, 1)
    oz_gemm_kernel(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, int Mp, int Nrp,
                   int chunks_total, int chunks_per_split, int M, int N, const int* __restrict__ ea,
                   const int* __restrict__ eb, cplx* __restrict__ C, long long ldc, int trans, int conj_out,
                   long long* __restrict__ pI, float* __restrict__ pU, int* __restrict__ timeouts) {
  using T = OzTile<BN>;
  constexpr int OZ_STAGES = T::STAGES, OZ_STAGE = T::STAGE, OZ_B_BYTES = T::B_BYTES, SETS = T::SETS;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + OZ_STAGES * OZ_STAGE);
  uint64_t* empty = full + OZ_STAGES;
  uint64_t* acc_full = empty + OZ_STAGES;  // [2], per accumulator set
  uint64_t* acc_empty = acc_full + 2;      // [2]
  uint64_t* mma_done = acc_empty + 2;
  uint32_t* tmem_slot = (uint32_t*)(mma_done + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tile = blockIdx.x, m_tile = blockIdx.y, split = blockIdx.z;
  const int c0 = split * chunks_per_split;
  const int nch = min(chunks_total, c0 + chunks_per_split) - c0;  // >= 1 by construction
  const int nstage = nch * OZ_KB_PER_CHUNK;  // (chunk, k-block)

  if (threadIdx.x == 0) {
    for (int s = 0; s < OZ_STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], T::EPI_WARPS);  // one arrival per epilogue warp
    }
    mbar_init(mma_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(OZ_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // producer: stage q = (chunk, k-block) holds the seven planes of A, then of B
    int issued = 0;
    for (int q = 0; q < nstage; ++q) {
      const int slot = q % OZ_STAGES, round = q / OZ_STAGES;
      const int kx = (c0 * OZ_KB_PER_CHUNK + q) * OZ_BK;
      if (!mbar_wait(&empty[slot], (round & 1) ^ 1)) {
        atomicAdd(timeouts, 1);
        break;
      }
      unsigned char* st = smem + slot * OZ_STAGE;
      mbar_expect_tx(&full[slot], OZ_STAGE);
      for (int s = 0; s < OZ_DIGITS; ++s) {
        tma_load_2d(st + s * OZ_A_BYTES, &mA, &full[slot], kx, s * Mp + m_tile * OZ_BM);
        tma_load_2d(st + OZ_DIGITS * OZ_A_BYTES + s * OZ_B_BYTES, &mB, &full[slot], kx, s * Nrp + n_tile * BN);
      }
      issued = q + 1;
    }
    // the last loads of every slot have landed before the CTA can leave
    for (int q = max(0, issued - OZ_STAGES); q < issued; ++q)
      if (!mbar_wait(&full[q % OZ_STAGES], (q / OZ_STAGES) & 1)) atomicAdd(timeouts, 1);
  } else if (warp == 1 && lane == 0) {
    // MMA issuer: group g = s + t of chunk c accumulates in tensor-memory
    // columns ACC_COLS (c % SETS) + BN g .. (with two sets chunk c's products
    // run while the epilogue drains chunk c - 1)
    bool ok = true;
    for (int q = 0; q < nstage && ok; ++q) {
      const int slot = q % OZ_STAGES, round = q / OZ_STAGES;
      const int kbc = q % OZ_KB_PER_CHUNK, c = q / OZ_KB_PER_CHUNK;
      // the set was drained: chunk c - SETS was that set's drain number c/SETS - 1
      if (kbc == 0 && c >= SETS && !mbar_wait(&acc_empty[c % SETS], ((c / SETS) - 1) & 1)) {
        atomicAdd(timeouts, 1);
        ok = false;
        break;
      }
      if (!mbar_wait(&full[slot], round & 1)) {
        atomicAdd(timeouts, 1);
        ok = false;
        break;
      }
      fence_after();
      const uint32_t st = smem_u32(smem + slot * OZ_STAGE);
      const uint32_t d = tmem + (uint32_t)((c % SETS) * T::ACC_COLS);
      // per k-step, A plane s meets the B planes t = 0 .. 6 - s in turn (group
      // s + t each): A is read from shared memory once per k-step and kept in
      // the collector buffer for the other B planes.  The plane s = 0 of a
      // chunk's first k-step starts every group.
#pragma unroll
      for (int ks = 0; ks < OZ_BK / 16; ++ks) {
        const uint32_t bb = st + OZ_DIGITS * OZ_A_BYTES + ks * 32;
#pragma unroll
        for (int s = 0; s < OZ_DIGITS; ++s) {
          const uint64_t ad = sdesc_kb<OZ_KB_BYTES>(st + s * OZ_A_BYTES + ks * 32);
          const uint32_t acc = (kbc == 0 && ks == 0 && s == 0) ? 0u : 1u;
          constexpr int ND = OZ_DIGITS;
          auto bd = [&](int t) { return sdesc_kb<OZ_KB_BYTES>(bb + t * OZ_B_BYTES); };
          if (s == ND - 1) {
            umma_bf16(d + s * BN, ad, bd(0), T::IDESC, acc);
            continue;
          }
          umma_bf16_coll<COLL_FILL>(d + s * BN, ad, bd(0), T::IDESC, acc);
#pragma unroll
          for (int t = 1; t < ND - 1 - s; ++t)
            umma_bf16_coll<COLL_USE>(d + (s + t) * BN, ad, bd(t), T::IDESC, acc);
          umma_bf16_coll<COLL_LAST>(d + (ND - 1) * BN, ad, bd(ND - 1 - s), T::IDESC, acc);
        }
      }
      umma_commit(&empty[slot]);  // frees the slot when these MMAs are done
      if (kbc == OZ_KB_PER_CHUNK - 1) umma_commit(&acc_full[c % SETS]);
    }
    // every MMA issued has completed before the accumulators are released
    umma_commit(mma_done);
    if (!mbar_wait(mma_done, 0)) atomicAdd(timeouts, 1);
  } else if (warp >= 2) {
    // epilogue: warp w reads tensor-memory lanes 32 (w % 4) .. (the rows of its
    // quarter), columns 32 h .. 32 h + 31 of each group (h = 0, and 1 for the
    // second four epilogue warps of BN = 64)
    constexpr int EC = 32;  // columns per epilogue thread
    const int q4 = warp & 3, h = (warp - 2) >> 2;
    const int row = m_tile * OZ_BM + 32 * q4 + lane;
    const uint32_t trow = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(EC * h);
    long long I[EC];
    float u[EC];
#pragma unroll
    for (int j = 0; j < EC; ++j) {
      I[j] = 0;
      u[j] = 0.0f;
    }
    bool ok = true;
    for (int c = 0; c < nch; ++c) {
      const bool ready = mbar_wait(&acc_full[c % SETS], (c / SETS) & 1);
      if (!ready) {
        if (lane == 0) atomicAdd(timeouts, 1);
        ok = false;
        break;
      }
      fence_after();
      const uint32_t tset = trow + (uint32_t)((c % SETS) * T::ACC_COLS);
      // two halves of 16 columns (fewer live registers beside the running sums),
      // two or three groups' loads waited for together
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        uint32_t v[3][16];
        // groups 0..3: exact integers up to 2^21, 2^22, 1.5 2^22 and 2^23, so each
        // pair combines in 32 bits before the 64-bit sum
#pragma unroll
        for (int g = 0; g < 4; g += 2) {
          tmem_ld16_issue(tset + g * BN + 16 * hf, v[0]);
          tmem_ld16_issue(tset + (g + 1) * BN + 16 * hf, v[1]);
          tmem_ld_wait(v[0]);
          tmem_ld_after(v[1]);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int p = __float2int_rn(__uint_as_float(v[0][j])) * 256 + __float2int_rn(__uint_as_float(v[1][j]));
            I[16 * hf + j] += g == 0 ? (long long)p * 65536 : (long long)p;
          }
        }
        // groups 4..6 (weight 2^-32 and below relative to group 0): FP32
#pragma unroll
        for (int g = 0; g < 3; ++g) tmem_ld16_issue(tset + (4 + g) * BN + 16 * hf, v[g]);
        tmem_ld_wait(v[0]);
#pragma unroll
        for (int g = 1; g < 3; ++g) tmem_ld_after(v[g]);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float t = fmaf(__uint_as_float(v[2][j]), 1.0f / 256.0f, __uint_as_float(v[1][j]));
          u[16 * hf + j] += fmaf(t, 1.0f / 256.0f, __uint_as_float(v[0][j]));
        }
      }
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[c % SETS]);
    }
    if (ok) {
      const int col0 = n_tile * BN + EC * h;
      if (pI) {
        // exact partial sums of this K range
        const long long base = ((long long)split * Mp + row) * Nrp + col0;
#pragma unroll
        for (int j = 0; j < EC; ++j) {
          pI[base + j] = I[j];
          pU[base + j] = u[j];
        }
      } else if (row < M) {
        const int er = ea[row];
#pragma unroll
        for (int j = 0; j < EC; j += 2) {
          const int n = (col0 + j) >> 1;
          if (n < N) {
            const double im = oz_value(I[j + 1], u[j + 1], er, eb[col0 + j + 1]);
            C[trans ? (long long)n * ldc + row : (long long)row * ldc + n] =
                make_double2(oz_value(I[j], u[j], er, eb[col0 + j]), conj_out ? -im : im);
          }
        }
      }
    }
  }
  fence_before();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS) : "memory");
  }
}

// C[m, n] from the S exact partials of (I, u) (integer sums are exact; u in FP32)
__global__ void oz_reduce_kernel(const long long* __restrict__ pI, const float* __restrict__ pU, int S, int Mp,
                                 int Nrp, int M, int N, const int* __restrict__ ea, const int* __restrict__ eb,
                                 cplx* __restrict__ C, long long ldc) {
  const long long total = (long long)M * N, pstride = (long long)Mp * Nrp;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int m = (int)(e / N), n = (int)(e - (long long)m * N);
    long long I0 = 0, I1 = 0;
    float u0 = 0.0f, u1 = 0.0f;
    for (int z = 0; z < S; ++z) {
      const long long o = z * pstride + (long long)m * Nrp + 2 * n;
      I0 += pI[o];
      I1 += pI[o + 1];
      u0 += pU[o];
      u1 += pU[o + 1];
    }
    C[(long long)m * ldc + n] = make_double2(oz_value(I0, u0, ea[m], eb[2 * n]), oz_value(I1, u1, ea[m], eb[2 * n + 1]));
  }
}

// The same for a product computed transposed: C[n, m] from row m, column n of
// the partials, by 32 x 32 tiles through shared memory (reads along n, writes
// along m).
__global__ void oz_reduce_t_kernel(const long long* __restrict__ pI, const float* __restrict__ pU, int S, int Mp,
                                   int Nrp, int M, int N, const int* __restrict__ ea, const int* __restrict__ eb,
                                   cplx* __restrict__ C, long long ldc, int conj_out) {
  __shared__ cplx tile[32][33];
  const int m0 = blockIdx.x * 32, n0 = blockIdx.y * 32;
  const long long pstride = (long long)Mp * Nrp;
  const int n = n0 + threadIdx.x;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int m = m0 + i;
    long long I0 = 0, I1 = 0;
    float u0 = 0.0f, u1 = 0.0f;
    if (m < M && n < N) {
      const long long o = (long long)m * Nrp + 2 * n;
#pragma unroll 4
      for (int z = 0; z < S; ++z) {
        const longlong2 p = *(const longlong2*)(pI + z * pstride + o);
        const float2 q = *(const float2*)(pU + z * pstride + o);
        I0 += p.x;
        I1 += p.y;
        u0 += q.x;
        u1 += q.y;
      }
      tile[i][threadIdx.x] =
          make_double2(oz_value(I0, u0, ea[m], eb[2 * n]), oz_value(I1, u1, ea[m], eb[2 * n + 1]));
    }
  }
  __syncthreads();
  const int m = m0 + threadIdx.x;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    if (m < M && n0 + i < N) {
      cplx v = tile[threadIdx.x][i];
      if (conj_out) v.y = -v.y;
      C[(long long)(n0 + i) * ldc + m] = v;
    }
  }
}

// The largest biased exponents of the rows (er) and columns (ec) of a K x K
// matrix, both arrays zero on entry; a block takes 32 columns of 128 rows.
__global__ void __launch_bounds__(256) oz_square_exp_kernel(const cplx* __restrict__ Q, int K, int* __restrict__ er,
                                                            int* __restrict__ ec) {
  __shared__ int s_c[8][32];
  const int c = blockIdx.x * 32 + threadIdx.x;
  int E = 0;
  for (int r = blockIdx.y * 128 + threadIdx.y; r < min(K, (int)blockIdx.y * 128 + 128); r += 8) {
    int e = 0;
    if (c < K) {
      const cplx v = Q[(long long)r * K + c];
      e = max(bexp(v.x), bexp(v.y));
    }
    E = max(E, e);
    e = __reduce_max_sync(0xffffffffu, e);
    if (threadIdx.x == 0) atomicMax(&er[r], e);
  }
  s_c[threadIdx.y][threadIdx.x] = E;
  __syncthreads();
  if (threadIdx.y == 0 && c < K) {
    for (int y = 1; y < 8; ++y) E = max(E, s_c[y][threadIdx.x]);
    atomicMax(&ec[c], E);
  }
}

// Digit planes of a K x K matrix as the row operand of products with Q^T (rows
// r, columns k of Q[r, k]: pt, exponents er) and with Q (rows c, columns k of
// Q[k, c]: pn, exponents ec), both Mp x Krp reals (Re, Im pairs along k, zeros
// beyond), from one read in 32 x 32 tiles.  The raw exponents become the row
// bounds et, en.
__global__ void __launch_bounds__(256)
    oz_square_prep_kernel(const cplx* __restrict__ Q, int K, int Mp, int Krp, const int* __restrict__ er,
                          const int* __restrict__ ec, int* __restrict__ et, int* __restrict__ en,
                          __nv_bfloat16* __restrict__ pt, __nv_bfloat16* __restrict__ pn) {
  __shared__ cplx tile[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32, kc = Krp >> 1;
  const long long plane = (long long)Mp * Krp;
  if (blockIdx.x == 0 && threadIdx.y == 0) {
    et[r0 + threadIdx.x] = row_bound(er[r0 + threadIdx.x]);
    en[r0 + threadIdx.x] = row_bound(ec[r0 + threadIdx.x]);
  }
  auto put = [&](__nv_bfloat16* p, int row, int k, cplx v, int e) {
    int dr[OZ_DIGITS], di[OZ_DIGITS];
    digits7(v.x, e, dr);
    digits7(v.y, e, di);
    __nv_bfloat162* out = (__nv_bfloat162*)(p + (long long)row * Krp + 2LL * k);
#pragma unroll
    for (int s = 0; s < OZ_DIGITS; ++s)
      out[s * plane / 2] = __halves2bfloat162(__float2bfloat16_rn((float)dr[s]), __float2bfloat16_rn((float)di[s]));
  };
  const int c = c0 + threadIdx.x;
  for (int i = threadIdx.y; i < 32; i += 8) {
    const int r = r0 + i;
    cplx v = make_double2(0.0, 0.0);
    if (r < K && c < K) v = Q[(long long)r * K + c];
    tile[i][threadIdx.x] = v;
    if (c < kc) put(pt, r, c, v, row_bound(er[r]));
  }
  __syncthreads();
  const int k = r0 + threadIdx.x;
  if (k >= kc) return;
  for (int i = threadIdx.y; i < 32; i += 8) put(pn, c0 + i, k, tile[threadIdx.x][i], row_bound(ec[c0 + i]));
}

unsigned oz_grid(long long n) {
  long long b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > 152 * 16) b = 152 * 16;
  return (unsigned)b;
}

struct OzLayout {
  int Mp, Nrp, Krp, chunks, S, cps, bn;
  size_t off_ea, off_eb, off_a, off_b, off_pi, off_pu, total;
};

// Tile width and chunks per CTA: the fewest chunk-times over whole waves of CTAs
// (152 SMs, one CTA each), counting a CTA's start (barriers, tensor memory, the
// pipeline's fill) as one chunk-time and, for K splits, the exact partials'
// round trip through memory (24 bytes per output element and split, about 16 MB
// per chunk-time).  A chunk of a 64-wide tile takes about the time of a 32-wide
// one (its MMAs do twice the work at the same issue rate, its drain is not
// overlapped).  Ties: the wider tile, the fewer K splits.  `room`: bytes for
// the partials (12 per output element and split).
void oz_choose(int Mp, int N, int chunks, double room, int* bn_, int* Nrp_, int* cps_) {
  double best = -1.0;
  for (int bn = 64; bn >= 32; bn -= 32) {
    const int Nrp = (2 * N + bn - 1) / bn * bn;
    const long long tiles = (long long)(Mp / OZ_BM) * (Nrp / bn);
    for (int cps = chunks; cps >= 1; --cps) {
      const long long S = (chunks + cps - 1) / cps;
      if (S > 1 && 12.0 * (double)S * Mp * Nrp > room) break;
      const double partials = S > 1 ? 24.0 * (double)S * Mp * Nrp / 16.0e6 : 0.0;
      const double cost = (double)((tiles * S + 151) / 152) * (cps + 1) + partials;
      if (best < 0 || cost < best) {
        best = cost;
        *bn_ = bn;
        *Nrp_ = Nrp;
        *cps_ = cps;
      }
    }
  }
}

OzLayout oz_layout(int M, int N, int K) {
  OzLayout L;
  L.Mp = (M + OZ_BM - 1) / OZ_BM * OZ_BM;
  L.Krp = (2 * K + OZ_CHUNK - 1) / OZ_CHUNK * OZ_CHUNK;
  L.chunks = L.Krp / OZ_CHUNK;
  oz_choose(L.Mp, N, L.chunks, 1e300, &L.bn, &L.Nrp, &L.cps);
  L.S = (L.chunks + L.cps - 1) / L.cps;
  auto al = [](size_t x) { return (x + 1023) & ~(size_t)1023; };
  size_t o = 0;
  L.off_ea = o;
  o += al(sizeof(int) * L.Mp);
  L.off_eb = o;
  o += al(sizeof(int) * L.Nrp);
  L.off_a = o;
  o += al((size_t)OZ_DIGITS * L.Mp * L.Krp * 2);
  L.off_b = o;
  o += al((size_t)OZ_DIGITS * L.Nrp * L.Krp * 2);
  L.off_pi = o;
  o += L.S > 1 ? al((size_t)L.S * L.Mp * L.Nrp * 8) : 0;
  L.off_pu = o;
  o += L.S > 1 ? al((size_t)L.S * L.Mp * L.Nrp * 4) : 0;
  L.total = o + 1024;
  return L;
}

cudaError_t oz_launch(cudaStream_t s, __nv_bfloat16* pa, __nv_bfloat16* pb, int Mp, int Nrp, int Krp, int bn,
                      int chunks, int cps, int M, int N, const int* ea, const int* eb, cplx* C, long long ldc, bool trans,
                      bool conj_out, long long* pI, float* pU, int* timeouts) {
  static bool attr = false;
  cudaError_t e;
  if (!attr) {
    if ((e = cudaFuncSetAttribute(oz_gemm_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  OzTile<32>::SMEM)) != cudaSuccess)
      return e;
    if ((e = cudaFuncSetAttribute(oz_gemm_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  OzTile<64>::SMEM)) != cudaSuccess)
      return e;
    attr = true;
  }
  CUtensorMap mA, mB;
  if ((e = tc_encode_bf16_map(&mA, pa, (long long)OZ_DIGITS * Mp, Krp, OZ_BM, OZ_KB_BYTES)) != cudaSuccess) return e;
  if ((e = tc_encode_bf16_map(&mB, pb, (long long)OZ_DIGITS * Nrp, Krp, bn, OZ_KB_BYTES)) != cudaSuccess) return e;
  const dim3 grid((unsigned)(Nrp / bn), (unsigned)(Mp / OZ_BM), (unsigned)((chunks + cps - 1) / cps));
  auto go = [&](auto kern, int threads, int smem) {
    kern<<<grid, threads, smem, s>>>(mA, mB, Mp, Nrp, chunks, cps, M, N, ea, eb, C, ldc, trans ? 1 : 0,
                                     conj_out ? 1 : 0, pI, pU, timeouts);
  };
  if (bn == 64)
    go(oz_gemm_kernel<64>, OzTile<64>::THREADS, OzTile<64>::SMEM);
  else
    go(oz_gemm_kernel<32>, OzTile<32>::THREADS, OzTile<32>::SMEM);
  count_launch();
  return cudaGetLastError();
}

size_t oz_al(size_t x) { return (x + 1023) & ~(size_t)1023; }

}  // namespace

size_t oz_square_bytes(int K) {
  const size_t Mp = (size_t)(K + OZ_BM - 1) / OZ_BM * OZ_BM, Krp = (2 * (size_t)K + OZ_CHUNK - 1) / OZ_CHUNK * OZ_CHUNK;
  return 2 * oz_al(4 * Mp) + oz_al((size_t)OZ_DIGITS * Mp * Krp * 2) + 1024;
}

size_t oz_thin_bytes(int M, int K) {
  const size_t rows = (2 * (size_t)M + 63) / 64 * 64, Krp = (2 * (size_t)K + OZ_CHUNK - 1) / OZ_CHUNK * OZ_CHUNK;
  return oz_al((size_t)OZ_DIGITS * rows * Krp * 2) + oz_al(4 * rows) + 3072;
}

cudaError_t oz_pack_square(cudaStream_t s, const cplx* Q, int K, void* memN, void* memT, OzSquare* outN,
                           OzSquare* outT) {
  const int Mp = (K + OZ_BM - 1) / OZ_BM * OZ_BM, Krp = (2 * K + OZ_CHUNK - 1) / OZ_CHUNK * OZ_CHUNK;
  void* mem[2] = {memN, memT};
  OzSquare* out[2] = {outN, outT};
  int* raw[2];
  cudaError_t e;
  for (int v = 0; v < 2; ++v) {
    char* p = (char*)(((uintptr_t)mem[v] + 1023) & ~(uintptr_t)1023);
    out[v]->K = K;
    out[v]->Mp = Mp;
    out[v]->Krp = Krp;
    raw[v] = (int*)p;
    out[v]->e = (int*)(p + oz_al(4 * (size_t)Mp));
    out[v]->p = p + 2 * oz_al(4 * (size_t)Mp);
    if ((e = cudaMemsetAsync(raw[v], 0, 4 * (size_t)Mp, s)) != cudaSuccess) return e;
  }
  oz_square_exp_kernel<<<dim3((unsigned)((K + 31) / 32), (unsigned)((K + 127) / 128)), dim3(32, 8), 0, s>>>(
      Q, K, raw[1], raw[0]);
  // tiles cover Mp rows in both directions (Krp / 2 <= Mp)
  oz_square_prep_kernel<<<dim3((unsigned)(Mp / 32), (unsigned)(Mp / 32)), dim3(32, 8), 0, s>>>(
      Q, K, Mp, Krp, raw[1], raw[0], outT->e, outN->e, (__nv_bfloat16*)outT->p, (__nv_bfloat16*)outN->p);
  count_launch(2);
  return cudaGetLastError();
}

cudaError_t oz_thin(cudaStream_t s, int M, const cplx* A, long long lda, bool conj_in, const OzSquare& Q, cplx* C,
                    long long ldc, bool conj_out, void* work, size_t work_bytes, int* timeouts) {
  if (M <= 0) return cudaSuccess;
  if (!timeouts || !work) return cudaErrorInvalidValue;
  const int K = Q.K, chunks = Q.Krp / OZ_CHUNK;
  char* base = (char*)(((uintptr_t)work + 1023) & ~(uintptr_t)1023);
  const size_t fixed = oz_thin_bytes(M, K);
  if (work_bytes < fixed) return cudaErrorMemoryAllocation;
  int bn = 64, Nrp = 0, cps = chunks;
  oz_choose(Q.Mp, M, chunks, (double)(work_bytes - fixed), &bn, &Nrp, &cps);
  const int S = (chunks + cps - 1) / cps;
  int* eb = (int*)base;
  __nv_bfloat16* pb = (__nv_bfloat16*)(base + oz_al(4 * (size_t)Nrp));
  char* part = (char*)pb + oz_al((size_t)OZ_DIGITS * Nrp * Q.Krp * 2);
  long long* pI = S > 1 ? (long long*)part : nullptr;
  float* pU = S > 1 ? (float*)(part + (size_t)S * Q.Mp * Nrp * 8) : nullptr;
  cudaError_t e;
  oz_prep_kernel<false><<<(unsigned)(Nrp / 2), OZ_PREP_THREADS, 0, s>>>(
      nullptr, 0, OP_N, A, lda, OP_T | (conj_in ? OP_CONJ : 0), 0, M, K, 0, Nrp, Q.Krp, nullptr, eb, nullptr, pb);
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = oz_launch(s, (__nv_bfloat16*)Q.p, pb, Q.Mp, Nrp, Q.Krp, bn, chunks, cps, K, M, Q.e, eb, C, ldc, true,
                     conj_out, pI, pU, timeouts)) != cudaSuccess)
    return e;
  if (S > 1) {
    oz_reduce_t_kernel<<<dim3((unsigned)((K + 31) / 32), (unsigned)((M + 31) / 32)), dim3(32, 8), 0, s>>>(
        pI, pU, S, Q.Mp, Nrp, K, M, Q.e, eb, C, ldc, conj_out ? 1 : 0);
    count_launch();
    return cudaGetLastError();
  }
  return cudaSuccess;
}

size_t oz_work_bytes(int M, int N, int K) { return oz_layout(M, N, K).total; }

cudaError_t oz_zgemm(cudaStream_t s, int M, int N, int K, const cplx* A, long long lda, int opA, const cplx* B,
                     long long ldb, int opB, cplx* C, long long ldc, void* work, size_t work_bytes, int* timeouts) {
  if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
  if (!timeouts) return cudaErrorInvalidValue;
  const OzLayout L = oz_layout(M, N, K);
  if (!work || work_bytes < L.total) return cudaErrorMemoryAllocation;
  cudaError_t e;
  char* base = (char*)(((uintptr_t)work + 1023) & ~(uintptr_t)1023);
  int* ea = (int*)(base + L.off_ea);
  int* eb = (int*)(base + L.off_eb);
  __nv_bfloat16* pa = (__nv_bfloat16*)(base + L.off_a);
  __nv_bfloat16* pb = (__nv_bfloat16*)(base + L.off_b);
  long long* pI = L.S > 1 ? (long long*)(base + L.off_pi) : nullptr;
  float* pU = L.S > 1 ? (float*)(base + L.off_pu) : nullptr;
  const int rows = L.Mp + L.Nrp / 2, per = OZ_PREP_THREADS / 32;
  auto prep = [&](auto kern, int blocks) {
    kern<<<(unsigned)blocks, OZ_PREP_THREADS, 0, s>>>(A, lda, opA, B, ldb, opB, M, N, K, L.Mp, L.Nrp, L.Krp, ea, eb, pa,
                                                      pb);
  };
  // a warp per row where the rows are short and fill the chip several times so
  if (L.Krp <= 256 && rows >= 152 * 32)
    prep(oz_prep_kernel<true>, (rows + per - 1) / per);
  else
    prep(oz_prep_kernel<false>, rows);
  count_launch();
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if ((e = oz_launch(s, pa, pb, L.Mp, L.Nrp, L.Krp, L.bn, L.chunks, L.cps, M, N, ea, eb, C, ldc, false, false, pI, pU,
                     timeouts)) != cudaSuccess)
    return e;
  if (L.S > 1) {
    oz_reduce_kernel<<<oz_grid((long long)M * N), 256, 0, s>>>(pI, pU, L.S, L.Mp, L.Nrp, M, N, ea, eb, C, ldc);
    count_launch();
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}
