// Block sparse matrix-vector product y = alpha A x + beta y, FP64, 4x4 blocks
// (the public bsr_spmv).
//
// FGMRES needs one product per iteration plus the residual at each restart
// (Sec. 6 setup); inside the solve those run in the kernel that also takes the
// Gram-Schmidt dot products (k_spmv_dots, fgmres.cu) and in the residual
// kernels, all with this kernel's row product (spmv.cuh).  Bytes dominate:
// every block is 128 bytes of FP64 values
// plus a 4-byte column index, read exactly once; x (4N doubles) is gathered
// through L1/L2.  A quad of threads handles one block row: thread q reads row q
// of every block of the row (32 contiguous bytes; the quad together reads each
// 128-byte block as one fully used line), forms the 4-term dot product with
// x_j, and writes y_i[q].  The first four blocks of a row are loaded before
// any arithmetic so each thread keeps up to 8 independent 16-byte loads in
// flight.  Half of a row's products are FP64 FMAs, half integer sums
// (spmv.cuh).  Large systems stream the rows through shared memory, one CTA
// per SM: 512x512 51.0 us, 6.1 TB/s (65.7 with FMAs alone, 62.9 in the direct
// form).
#include "common.cuh"
#include "spmv.cuh"

namespace abilu {

constexpr int SPMV_THREADS = 256;
constexpr int SPMV_ROWS = SPMV_THREADS / 4;

// PLAIN: y = A x (alpha = 1, beta = 0, decided on the host), the form FGMRES
// uses: no FP64 instruction beyond the row product's (a compare and a multiply
// per output cost 12% when the FP64 pipe bounded this kernel).
// Otherwise y = alpha A x + beta y, and beta == 0 never reads y (which may
// hold NaN).
template <bool PLAIN, int TH>
__global__ void __launch_bounds__(TH, TH == STREAM_THREADS ? 1 : 4)
k_spmv(PatternView P, const double *__restrict__ A, double alpha, const double *__restrict__ x,
       double beta, double *__restrict__ y) {
    extern __shared__ __align__(128) char smem[];
    pdl_wait();
    pdl_trigger();
    const int q = threadIdx.x & 3;
    for_rows<TH, true>(P, A, x, smem,
        [&](int i) { return PLAIN || beta == 0.0 ? 0.0 : y[(size_t)i * BS + q]; },
        [&](int i, double s, double y0) {
            const size_t o = (size_t)i * BS + q;
            if constexpr (PLAIN) y[o] = s;
            else y[o] = beta == 0.0 ? alpha * s : alpha * s + beta * y0;
        });
}

abilu_status spmv_launch(const PatternView &P, const double *A, double alpha, const double *x,
                         double beta, double *y, cudaStream_t st) {
    const int grid = (P.n + SPMV_ROWS - 1) / SPMV_ROWS;
    const bool plain = alpha == 1.0 && beta == 0.0;
    if (streamed(P)) {
        if (plain) launch_stream<k_spmv<true, STREAM_THREADS>>(st, P, A, alpha, x, beta, y);
        else launch_stream<k_spmv<false, STREAM_THREADS>>(st, P, A, alpha, x, beta, y);
    } else if (plain) {
        launch_pdl(k_spmv<true, SPMV_THREADS>, grid, SPMV_THREADS, 0, st, P, A, alpha, x, beta, y);
    } else {
        launch_pdl(k_spmv<false, SPMV_THREADS>, grid, SPMV_THREADS, 0, st, P, A, alpha, x, beta, y);
    }
    ABILU_LAUNCH_CHECK("k_spmv");
    return ABILU_OK;
}

}  // namespace abilu
