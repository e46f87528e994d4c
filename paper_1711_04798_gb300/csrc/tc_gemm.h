// Tensor-core (tcgen05) complex GEMM of the precision form: TF32, split-BF16x3
// (hi*hi + hi*lo + lo*hi) or split-BF16x6 (three parts, the six products of
// combined order <= 2) with FP32 accumulation in TMEM.
#pragma once
#include <cuda.h>

#include "ctm_internal.h"

// C[M,N] = alpha * opA(A) opB(B) with complex FP64 storage of A, B, C; the
// operands are packed (permuted, converted, real-embedded) into `scratch`
// above scratch_top.  Returns cudaErrorNotSupported when the precision or the
// shape has no tensor-core kernel.  `timeouts` (device int, required) counts
// the bounded waits inside the kernel that ran out; the caller owns it and
// reads it after the stream has drained (each handle passes its own slot).
struct TcTuner;
struct TcChoice;

// Optional timing probe of one product (measurement support): events recorded
// on the launching stream before the main tensor-core kernel, after it, and
// after the split-K reduction; the call fills in the padded shape and tile
// choice it ran, so the caller can credit algorithmic flops and bytes.
struct TcProbe {
  cudaEvent_t ev[3];
  long long Mp, Nrp, Krp;  // padded real-embedded shape
  int splits, bn, parts, elem_bytes;
};

// An operand read through a strided view instead of a permuted copy: element
// (r, c) is p[roff(r) + coff(c)], roff / coff sums of per-axis strides over
// up to four axes each (the last axis fastest), conjugated when conj.  For
// the A role rows are m and columns k; for the B role rows are n and columns
// k (the transpose of op(B)).
struct TcView {
  const void* p;   // complex FP64, or complex FP32 with f32
  int f32;
  int nr, nc;
  int rdim[4], cdim[4];
  long long rstr[4], cstr[4];
  int conj;
};
// force: a fixed tile choice instead of the tuner's or the default one
cudaError_t tc_zgemm(cudaStream_t s, int prec, int M, int N, int K, cplx alpha, const cplx* A,
                     long long lda, int opA, const cplx* B, long long ldb, int opB, cplx* C,
                     long long ldc, cplx* scratch, long long scratch_elems, long long scratch_top,
                     int* timeouts, TcTuner* tuner = nullptr, const TcChoice* force = nullptr,
                     TcProbe* probe = nullptr);

// Thin products: C (M x K) = A (M x K) times a square K x K matrix, with few
// rows (the range finder, the projector assembly).  They are computed
// transposed, C^T = Q^T A^T, so that the real embedding doubles the thin operand
// and not the matrix, whose packed form (Re, Im pairs, 2 reals per complex
// number and part) is what bounds them: at K = 2500 in three BF16 parts 75 MB
// per product instead of 150 MB.  The partials' sum writes the next product's
// packed operand itself, so a chain packs its first operand only.
struct TcPacked {  // one orientation of Q
  int prec, K;
  void* b[3];      // parts (TF32: one)
};
struct TcThin {    // a packed thin operand: 2M x 2K reals
  int prec, M, K;
  void* b[3];
};
size_t tc_packed_bytes(int prec, int K);
size_t tc_thin_bytes(int prec, int M, int K);
// Q packed for thin * Q (outN) and thin * Q^T (outT), one read.  D2 = 0: Q row-major
// complex FP64.  D2 > 0: Q[(x a), (y b)] complex FP32 stored as [x][y][a][b] with a,
// b < D2 and x, y < K / D2 (a corner as its last product leaves it).
cudaError_t tc_pack_square(cudaStream_t s, int prec, const void* Q, int K, int D2, void* memN, void* memT,
                           TcPacked* outN, TcPacked* outT);
// a thin operand's parts in mem (tc_thin_bytes)
cudaError_t tc_thin_layout(int prec, int M, int K, void* mem, TcThin* out);
// t = A (M x K, row-major, conjugated with conj), packed
cudaError_t tc_pack_thin(cudaStream_t s, const cplx* A, long long lda, bool conj, const TcThin& t);
// A Q as C (optional; conjugated with conj_out) and / or packed as *next (optional)
cudaError_t tc_thin(cudaStream_t s, const TcThin& A, const TcPacked& Q, cplx* C, long long ldc, bool conj_out,
                    const TcThin* next, cplx* scratch, long long scratch_elems, long long scratch_top, int* timeouts,
                    TcTuner* tuner = nullptr, TcProbe* probe = nullptr);

// Tile choice of one product: output tile 128 x bn (bn = 128 or 256 real
// columns) and the number of K splits (FP32 partials summed in a fixed order).
struct TcChoice {
  int bn;
  int splits;
};

// Autotuner table (shape -> tile choice).  Products run through a tuner use
// its choice for their shape; while measuring, a shape not yet in the table is
// timed with every candidate choice (CUDA events, synchronising) and the
// fastest is recorded.  Without a tuner, or for unknown shapes when not
// measuring, the default heuristic applies.  Not thread-safe.
TcTuner* tc_tuner_create();
void tc_tuner_destroy(TcTuner* t);
void tc_tuner_set_measuring(TcTuner* t, bool on);
int tc_tuner_size(const TcTuner* t);
// entry i: fields = {prec, M, N, K, bn, splits}; us = {best time, default-choice time}
bool tc_tuner_entry(const TcTuner* t, int i, int fields[6], double us[2]);

// one-time setup (kernel attributes, driver entry point); called before any
// stream capture so that captured products make no such calls.
cudaError_t tc_init();

// C[M,N] = alpha A B with either operand given as a view (the other, when the
// view pointer is null, as (ptr, ld, op) like tc_zgemm): the operand packing
// gathers straight from the source tensor (a fused permute-and-pack).  c_f32
// (alpha 1): C as complex FP32, which is all that the FP32 sums carry.
cudaError_t tc_zgemm_views(cudaStream_t s, int prec, int M, int N, int K, cplx alpha, const TcView* va,
                           const cplx* A, long long lda, int opA, const TcView* vb, const cplx* B, long long ldb,
                           int opB, void* C, long long ldc, bool c_f32, cplx* scratch, long long scratch_elems,
                           long long scratch_top, int* timeouts, TcTuner* tuner = nullptr,
                           TcProbe* probe = nullptr);

// 2D tensor map of a K-major BF16 operand [rows x kcols] with boxes of
// box_rows x kb_bytes (128 or 64, swizzled over that many bytes), for the
// tcgen05 kernels.
cudaError_t tc_encode_bf16_map(CUtensorMap* map, void* base, long long rows, long long kcols, int box_rows,
                               int kb_bytes);

// FP64-accurate complex GEMM on the tensor cores (ozaki.cu): C = opA(A) opB(B)
// (complex FP64 storage, alpha 1, beta 0).  `work` (device, work_bytes) holds
// the digit planes, row scales and split partials: oz_work_bytes(M, N, K).
size_t oz_work_bytes(int M, int N, int K);
cudaError_t oz_zgemm(cudaStream_t s, int M, int N, int K, const cplx* A, long long lda, int opA, const cplx* B,
                     long long ldb, int opB, cplx* C, long long ldc, void* work, size_t work_bytes, int* timeouts);

// Thin FP64-accurate products C (M x K) = A (M x K) Q, computed transposed: the
// digit planes of a square Q in both orientations are split once and serve every
// product with it (splitting them for each of a cut's 28 products took as
// long as a fifth of the products), and the real embedding doubles the thin
// operand's planes instead of Q's.
struct OzSquare {
  int K, Mp, Krp;
  int* e;   // row bounds
  void* p;  // seven planes of Mp x Krp
};
size_t oz_square_bytes(int K);
// Q (row-major K x K) for thin * Q (outN) and thin * Q^T (outT)
cudaError_t oz_pack_square(cudaStream_t s, const cplx* Q, int K, void* memN, void* memT, OzSquare* outN,
                           OzSquare* outT);
// the least work of oz_thin (without room for K splits)
size_t oz_thin_bytes(int M, int K);
// C = op(A) Q (op: conjugation with conj_in; the result conjugated with conj_out)
cudaError_t oz_thin(cudaStream_t s, int M, const cplx* A, long long lda, bool conj_in, const OzSquare& Q, cplx* C,
                    long long ldc, bool conj_out, void* work, size_t work_bytes, int* timeouts);
