// Threshold block ILU by fixed-point sweeps.
//
// The paper's closing section names a parallel threshold ILU (ParILUT) as the
// next extension of its sweeps, without an algorithm.  This is the library's:
//   start   X = A on A's pattern S, `sweeps` synchronous sweeps of Eq. (bilu);
//   repeat `iters` times:
//     fill  S' = the block pattern of L U (L unit lower, U upper on S; it
//           contains S), new blocks start at zero, A is zero outside its own
//           pattern, `sweeps` synchronous sweeps on S';
//     drop  of the strictly lower blocks keep those whose squared Frobenius
//           norm exceeds the (budget+1)-th largest (every one if there are at
//           most budget), likewise the strictly upper blocks; diagonal blocks
//           stay.  Budgets: floor(fill * count) with the counts of A's
//           pattern.  `sweeps` synchronous sweeps on the kept pattern.
// Every sweep is the FP64 synchronous build of build.cu on an analysed
// pattern (abilu_pattern_create), so the pair lists of the fill blocks come
// from the same analysis as A's.  Pattern work on the device: a thread per row
// merges the upper parts of the rows its L blocks name (sorted, at most
// PLU_MAX_ROW blocks per row); values move between patterns by a per-row merge
// of the sorted columns; the selection threshold is found byte by byte on the
// bit patterns of the non-negative keys (integer counts, exact).
#include <string.h>

#include <utility>
#include <vector>

#include "common.cuh"

namespace abilu {

abilu_status build_dispatch(abilu_factors f, const double *A, int nsweeps, abilu_mode mode,
                            abilu_init init, cudaStream_t st);
abilu_status export_dispatch(abilu_factors f, double *X, double *Dinv, cudaStream_t st);
abilu_status factors_create_bare(abilu_pattern p, abilu_dtype dtype, abilu_factors *out);
abilu_status factors_add_status(abilu_factors f);
abilu_status scan_i32(const int32_t *in, int32_t *out, int n, long long *scratch, unsigned *err,
                      cudaStream_t st);
abilu_status form_scaled_upper(abilu_factors f, cudaStream_t st);
__global__ void k_block_norm2(const double *__restrict__ A, long long nnzb, double *__restrict__ w);

constexpr int PLU_THREADS = 128;
constexpr int PLU_MAX_ROW = 192;   // blocks per row of the pattern of L U

// Row i of the pattern of L U: the columns j >= k of row k for k = i and for
// every column k < i of row i, sorted and distinct.  FILL = false: count only
// (cnt[i]); FILL: write them at out_col + out_ptr[i].  A row longer than
// PLU_MAX_ROW sets *err and is cut (the host then fails the call).
template <bool FILL>
__global__ void __launch_bounds__(PLU_THREADS)
k_lu_pattern(int n, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind,
             const int32_t *__restrict__ diagpos, int32_t *__restrict__ cnt,
             const int32_t *__restrict__ out_ptr, int32_t *__restrict__ out_col, unsigned *err) {
    const int i = blockIdx.x * PLU_THREADS + threadIdx.x;
    if (i >= n) return;
    int buf[PLU_MAX_ROW];
    int m = 0;
    const int p0 = rowptr[i], pd = diagpos[i];
    for (int p = p0; p <= pd; p++) {   // k < i (L blocks), then k = i
        const int k = colind[p];
        for (int q = diagpos[k]; q < rowptr[k + 1]; q++) {
            const int j = colind[q];
            int a = 0, b = m;   // lower bound of j in buf[0..m)
            while (a < b) {
                const int h = (a + b) >> 1;
                if (buf[h] < j) a = h + 1; else b = h;
            }
            if (a < m && buf[a] == j) continue;
            if (m == PLU_MAX_ROW) {
                atomicOr(err, 1u);
                continue;
            }
            for (int t = m; t > a; t--) buf[t] = buf[t - 1];
            buf[a] = j;
            m++;
        }
    }
    if constexpr (FILL) {
        int32_t *o = out_col + out_ptr[i];
        for (int t = 0; t < m; t++) o[t] = buf[t];
    } else {
        cnt[i] = m;
    }
}

// Values of row i on the new pattern: a quad per row merges the sorted old
// and new columns; thread q copies row q of each matched block (zero where the
// old pattern has none).  Two sources (X on the old pattern, A on its own).
__global__ void __launch_bounds__(PLU_THREADS)
k_map_blocks(int n, const int32_t *__restrict__ rp_new, const int32_t *__restrict__ ci_new,
             const int32_t *__restrict__ rp_x, const int32_t *__restrict__ ci_x,
             const double *__restrict__ X, const int32_t *__restrict__ rp_a,
             const int32_t *__restrict__ ci_a, const double *__restrict__ A,
             double *__restrict__ X_new, double *__restrict__ A_new) {
    const int i = blockIdx.x * (PLU_THREADS / 4) + (threadIdx.x >> 2), q = threadIdx.x & 3;
    if (i >= n) return;
    int px = rp_x[i], pa = rp_a[i];
    const int px1 = rp_x[i + 1], pa1 = rp_a[i + 1];
    for (int p = rp_new[i]; p < rp_new[i + 1]; p++) {
        const int j = ci_new[p];
        while (px < px1 && ci_x[px] < j) px++;
        while (pa < pa1 && ci_a[pa] < j) pa++;
        double v[4] = {0.0, 0.0, 0.0, 0.0}, w[4] = {0.0, 0.0, 0.0, 0.0};
        if (px < px1 && ci_x[px] == j) ld_row(X + (size_t)px * BB + q * BS, v);
        if (pa < pa1 && ci_a[pa] == j) ld_row(A + (size_t)pa * BB + q * BS, w);
        st_row(X_new + (size_t)p * BB + q * BS, v);
        st_row(A_new + (size_t)p * BB + q * BS, w);
    }
}

// Factors from X in the pattern layout (L_ij at column < row, U_ij at column
// > row, U_ii on the diagonal) and Dinv: the compact arrays of iterate `cur`,
// rounded to the storage type T
template <typename T>
__global__ void __launch_bounds__(PLU_THREADS)
k_import(PatternView P, const double *__restrict__ X, const double *__restrict__ Dinv,
         T *__restrict__ L, T *__restrict__ U, T *__restrict__ D, T *__restrict__ Udiag) {
    const int i = blockIdx.x * (PLU_THREADS / 4) + (threadIdx.x >> 2), q = threadIdx.x & 3;
    if (i >= P.n) return;
    const int p0 = P.rowptr[i], p1 = P.rowptr[i + 1], dp = P.diagpos[i];
    for (int p = p0; p < p1; p++) {
        double v[4];
        ld_row(X + (size_t)p * BB + q * BS, v);
        if (p < dp) st_row(L + (size_t)(P.lrow[i] + p - p0) * BB + q * BS, v);
        else if (p > dp) st_row(U + (size_t)(P.urow[i] + p - dp - 1) * BB + q * BS, v);
        else st_row(Udiag + (size_t)i * BB + q * BS, v);
    }
    double d[4];
    ld_row(Dinv + (size_t)i * BB + q * BS, d);
    st_row(D + (size_t)i * BB + q * BS, d);
}

// Selection of the (budget+1)-th largest key of each side (0: strictly lower
// blocks, 1: strictly upper; keys are squared norms, non-negative, so their bit
// patterns order like the values): eight passes of one byte each, from the top.
// A pass counts, among the keys that agree with the bytes found so far, the 256
// values of the next byte; its last CTA walks the counts down from 255 to the
// value that holds the wanted rank, and clears them for the next pass.  Integer
// counts, so exact and independent of the order.  (A bisection on the host, 64
// counting passes with a round trip each, took 1.4 ms of a 9 ms call.)
struct Select {
    unsigned long long key[2];     // bytes found so far; after the last pass the threshold
    long long rank[2];             // wanted rank among the keys that agree (from 1)
    unsigned hist[2][256];
    unsigned done;
};

__global__ void k_select_init(Select *s, long long rl, long long ru) {
    for (int t = threadIdx.x; t < 512; t += blockDim.x) s->hist[t >> 8][t & 255] = 0u;
    if (threadIdx.x == 0) {
        s->key[0] = s->key[1] = 0ull;
        s->rank[0] = rl;
        s->rank[1] = ru;
        s->done = 0u;
    }
}

__global__ void __launch_bounds__(256)
k_select_pass(int n, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ diagpos,
              const unsigned long long *__restrict__ key, int shift, Select *s) {
    __shared__ unsigned h[2][256];
    __shared__ bool last;
    h[0][threadIdx.x] = h[1][threadIdx.x] = 0u;
    __syncthreads();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n) {
        const int dp = diagpos[i], p1 = rowptr[i + 1];
        for (int p = rowptr[i]; p < p1; p++) {
            if (p == dp) continue;
            const int side = p > dp;
            const unsigned long long k = key[p];
            // the bytes above this one (none in the first pass)
            if (shift == 56 || (k >> (shift + 8)) == (s->key[side] >> (shift + 8)))
                atomicAdd(&h[side][(unsigned)(k >> shift) & 255u], 1u);
        }
    }
    __syncthreads();
    for (int side = 0; side < 2; side++)
        if (h[side][threadIdx.x]) atomicAdd(&s->hist[side][threadIdx.x], h[side][threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&s->done, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    // thread v: does value v of the byte hold the rank?
    for (int side = 0; side < 2; side++) {
        h[side][threadIdx.x] = __ldcg(&s->hist[side][threadIdx.x]);
        s->hist[side][threadIdx.x] = 0u;
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        const int side = threadIdx.x;
        long long r = s->rank[side];
        int v = 255;
        while (v > 0 && r > (long long)h[side][v]) r -= h[side][v--];
        s->key[side] |= (unsigned long long)v << shift;
        s->rank[side] = r;
    }
    if (threadIdx.x == 0) s->done = 0u;
}

// kept blocks of row i: diagonal, lower with key bits > tl, upper with > tu
// (KEEP_ALL_L / _U in the flags: every lower / upper block)
template <bool FILL>
__global__ void __launch_bounds__(PLU_THREADS)
k_compact(int n, const int32_t *__restrict__ rowptr, const int32_t *__restrict__ colind,
          const unsigned long long *__restrict__ key, const Select *__restrict__ sel, int keep_all_l, int keep_all_u,
          int32_t *__restrict__ cnt,
          const int32_t *__restrict__ out_ptr, int32_t *__restrict__ out_col,
          const double *__restrict__ X, const double *__restrict__ A, double *__restrict__ X_out,
          double *__restrict__ A_out) {
    const int i = blockIdx.x * (PLU_THREADS / 4) + (threadIdx.x >> 2), q = threadIdx.x & 3;
    if (i >= n) return;
    const unsigned long long tl = sel->key[0], tu = sel->key[1];
    int o = FILL ? out_ptr[i] : 0;
    for (int p = rowptr[i]; p < rowptr[i + 1]; p++) {
        const int j = colind[p];
        const bool keep = j == i || (j < i ? (keep_all_l || key[p] > tl) : (keep_all_u || key[p] > tu));
        if (!keep) continue;
        if constexpr (FILL) {
            if (q == 0) out_col[o] = j;
            double v[4];
            ld_row(X + (size_t)p * BB + q * BS, v);
            st_row(X_out + (size_t)o * BB + q * BS, v);
            ld_row(A + (size_t)p * BB + q * BS, v);
            st_row(A_out + (size_t)o * BB + q * BS, v);
        }
        o++;
    }
    if (!FILL && q == 0) cnt[i] = o;
}

}  // namespace abilu

// ------------------------------------------------------------------- host

namespace abilu {

namespace {

// device allocations released at scope exit; several arrays share one (carve):
// an allocation with its release costs this call tens of microseconds
struct DevBufs {
    std::vector<void *> p;
    ~DevBufs() {
        for (void *q : p) cudaFree(q);
    }
    template <typename T> abilu_status get(T **out, size_t count) {
        void *q = nullptr;
        cudaError_t e = cudaMalloc(&q, sizeof(T) * (count > 0 ? count : 1));
        if (e != cudaSuccess) return cuda_fail(e, "abilu_parilut: cudaMalloc");
        p.push_back(q);
        *out = static_cast<T *>(q);
        return ABILU_OK;
    }
};

// arrays of one allocation, each on a 256-byte boundary
struct Carve {
    char *base = nullptr;
    size_t at = 0;
    template <typename T> T *take(size_t count) {
        T *q = base ? reinterpret_cast<T *>(base + at) : nullptr;
        at += (sizeof(T) * (count > 0 ? count : 1) + 255) & ~(size_t)255;
        return q;
    }
};

// `lay` takes its arrays from a Carve: once to size the allocation, once on it
template <typename F> abilu_status carve(DevBufs &bufs, F lay) {
    Carve c;
    lay(c);
    abilu_status s = bufs.get(&c.base, c.at);
    if (s != ABILU_OK) return s;
    c.at = 0;
    lay(c);
    return ABILU_OK;
}

struct PatternGuard {
    abilu_pattern p = nullptr;
    ~PatternGuard() {
        if (p) abilu_pattern_destroy(p);
    }
};
struct FactorsGuard {
    abilu_factors f = nullptr;
    ~FactorsGuard() {
        if (f) abilu_factors_destroy(f);
    }
};

}  // namespace

static int grid_rows(int n, int per_cta) { return (n + per_cta - 1) / per_cta; }

// factors on p from X (pattern layout) and Dinv, then `sweeps` synchronous
// sweeps with the values Ap (p's layout); *out receives the handle
static abilu_status factors_from(abilu_pattern p, const double *X, const double *Dinv,
                                 const double *Ap, int sweeps, cudaStream_t st, abilu_factors *out) {
    abilu_factors f = nullptr;
    abilu_status s = factors_create_bare(p, ABILU_F64, &f);
    if (s != ABILU_OK) return s;
    const int c = f->cur;
    k_import<double><<<counted(grid_rows(p->v.n, PLU_THREADS / 4)), PLU_THREADS, 0, st>>>(
        p->v, X, Dinv, static_cast<double *>(f->L[c]), static_cast<double *>(f->U[c]),
        static_cast<double *>(f->D[c]), static_cast<double *>(f->Udiag));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        abilu_factors_destroy(f);
        return cuda_fail(e, "k_import");
    }
    s = build_dispatch(f, Ap, sweeps, ABILU_SYNC, ABILU_INIT_FROM_PREVIOUS, st);
    if (s != ABILU_OK) {
        abilu_factors_destroy(f);
        return s;
    }
    *out = f;
    return ABILU_OK;
}

// the (budget+1)-th largest keys of both sides into *sel (a side that keeps
// every block does not use its own)
static abilu_status select_thresholds(int n, const int32_t *rowptr, const int32_t *diagpos,
                                      const unsigned long long *key, long long bl, long long bu,
                                      Select *sel, cudaStream_t st) {
    k_select_init<<<counted(1), 256, 0, st>>>(sel, bl + 1, bu + 1);
    for (int shift = 56; shift >= 0; shift -= 8)
        k_select_pass<<<counted(grid_rows(n, 256)), 256, 0, st>>>(n, rowptr, diagpos, key, shift, sel);
    ABILU_LAUNCH_CHECK("k_select_pass");
    return ABILU_OK;
}

// the final FP64 factors stored in `dtype` (FP32: with Dinv U for the upper
// sweeps): a new handle on the same pattern
template <typename T>
static abilu_status store_as(abilu_factors f64, abilu_dtype dtype, double *X, double *D,
                             cudaStream_t st, abilu_factors *out) {
    abilu_pattern p = f64->p;
    abilu_status s = export_dispatch(f64, X, D, st);
    if (s != ABILU_OK) return s;
    abilu_factors f = nullptr;
    if ((s = factors_create_bare(p, dtype, &f)) != ABILU_OK) return s;
    const int c = f->cur;
    k_import<T><<<counted(grid_rows(p->v.n, PLU_THREADS / 4)), PLU_THREADS, 0, st>>>(
        p->v, X, D, static_cast<T *>(f->L[c]), static_cast<T *>(f->U[c]), static_cast<T *>(f->D[c]),
        static_cast<T *>(f->Udiag));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        abilu_factors_destroy(f);
        return cuda_fail(e, "k_import");
    }
    if ((s = form_scaled_upper(f, st)) != ABILU_OK) {
        abilu_factors_destroy(f);
        return s;
    }
    *out = f;
    return ABILU_OK;
}

static abilu_status read_total(const int32_t *ptr_n, const unsigned *err, cudaStream_t st,
                               int32_t *total) {
    unsigned e = 0;
    ABILU_CUDA(cudaMemcpyAsync(total, ptr_n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    ABILU_CUDA(cudaMemcpyAsync(&e, err, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
    ABILU_CUDA(cudaStreamSynchronize(st));
    if (e & 1u) return fail(ABILU_EINVAL, "abilu_parilut: a row of L U exceeds %d blocks", PLU_MAX_ROW);
    if (e & (1u << 8)) return fail(ABILU_EINVAL, "abilu_parilut: more than 2^31 - 1 blocks");
    return ABILU_OK;
}

}  // namespace abilu

using namespace abilu;

extern "C" void abilu_parilut_default_opts(abilu_parilut_opts *o) {
    if (!o) return;
    o->fill = 2.0;
    o->iters = 3;
    o->sweeps = 2;
    o->factor_dtype = ABILU_F64;
}

extern "C" abilu_status abilu_parilut(abilu_pattern pA, const double *A,
                                      const abilu_parilut_opts *o, abilu_stream stream,
                                      abilu_pattern *pattern_out, abilu_factors *factors_out) {
    if (!pA || !A || !o || !pattern_out || !factors_out)
        return fail(ABILU_EINVAL, "abilu_parilut: NULL argument");
    *pattern_out = nullptr;
    *factors_out = nullptr;
    if ((reinterpret_cast<uintptr_t>(A) & 15u) != 0)
        return fail(ABILU_EINVAL, "abilu_parilut: A_vals must be 16-byte aligned");
    if (!(o->fill >= 0.0 && o->fill <= 1e9) || o->iters < 0 || o->sweeps < 0 ||
        (o->factor_dtype != ABILU_F64 && o->factor_dtype != ABILU_F32 && o->factor_dtype != ABILU_BF16))
        return fail(ABILU_EINVAL, "abilu_parilut: bad options");
    cudaStream_t st = S(stream);
    const PatternView &VA = pA->v;
    const int n = VA.n;
    const long long bl = (long long)(o->fill * (double)VA.nl), bu = (long long)(o->fill * (double)VA.nu);
    DevBufs bufs;
    unsigned *err = nullptr;
    Select *sel = nullptr;
    long long *scratch = nullptr;
    int32_t *rowcnt = nullptr, *rp2 = nullptr, *rp3 = nullptr;
    double *D = nullptr, *X = nullptr;
    abilu_status s = carve(bufs, [&](Carve &c) {
        err = c.take<unsigned>(1);
        sel = c.take<Select>(1);
        scratch = c.take<long long>((size_t)n / 4096 + 2);
        rowcnt = c.take<int32_t>(n);
        rp2 = c.take<int32_t>((size_t)n + 1);
        rp3 = c.take<int32_t>((size_t)n + 1);
        D = c.take<double>((size_t)n * BB);
        if (o->iters > 0) X = c.take<double>((size_t)VA.nnzb * BB);
    });
    if (s != ABILU_OK) return s;
    ABILU_CUDA(cudaMemsetAsync(err, 0, sizeof(unsigned), st));

    // start: X = A, `sweeps` synchronous sweeps on A's pattern
    PatternGuard pcur;   // the current pattern when owned (NULL: A's)
    {
        FactorsGuard f0;
        if ((s = factors_create_bare(pA, ABILU_F64, &f0.f)) != ABILU_OK) return s;
        if ((s = build_dispatch(f0.f, A, o->sweeps, ABILU_SYNC, ABILU_INIT_FROM_A, st)) != ABILU_OK) return s;
        if (o->iters == 0) {
            PatternGuard pc;
            if ((s = abilu_pattern_create(n, VA.nnzb, VA.rowptr, VA.colind, stream, &pc.p)) != ABILU_OK) return s;
            FactorsGuard fo;
            if ((s = factors_create_bare(pc.p, ABILU_F64, &fo.f)) != ABILU_OK) return s;
            if ((s = build_dispatch(fo.f, A, o->sweeps, ABILU_SYNC, ABILU_INIT_FROM_A, st)) != ABILU_OK) return s;
            if (o->factor_dtype != ABILU_F64) {
                double *Xs = nullptr;
                if ((s = bufs.get(&Xs, (size_t)VA.nnzb * BB)) != ABILU_OK) return s;
                FactorsGuard fn;
                s = o->factor_dtype == ABILU_F32
                        ? store_as<float>(fo.f, ABILU_F32, Xs, D, st, &fn.f)
                        : store_as<__nv_bfloat16>(fo.f, ABILU_BF16, Xs, D, st, &fn.f);
                if (s != ABILU_OK) return s;
                std::swap(fo.f, fn.f);
            }
            if ((s = factors_add_status(fo.f)) != ABILU_OK) return s;
            ABILU_CUDA(cudaStreamSynchronize(st));
            *pattern_out = pc.p;
            *factors_out = fo.f;
            pc.p = nullptr;
            fo.f = nullptr;
            return ABILU_OK;
        }
        if ((s = export_dispatch(f0.f, X, D, st)) != ABILU_OK) return s;
        ABILU_CUDA(cudaStreamSynchronize(st));
    }
    for (int it = 0; it < o->iters; it++) {
        const PatternView &VC = pcur.p ? pcur.p->v : VA;
        // fill: the pattern of L U
        k_lu_pattern<false><<<counted(grid_rows(n, PLU_THREADS)), PLU_THREADS, 0, st>>>(
            n, VC.rowptr, VC.colind, VC.diagpos, rowcnt, nullptr, nullptr, err);
        ABILU_LAUNCH_CHECK("k_lu_pattern");
        if ((s = scan_i32(rowcnt, rp2, n, scratch, err, st)) != ABILU_OK) return s;
        int32_t nnz2 = 0;
        if ((s = read_total(rp2 + n, err, st, &nnz2)) != ABILU_OK) return s;
        int32_t *ci2 = nullptr;
        double *X2 = nullptr, *A2 = nullptr;
        unsigned long long *key = nullptr;
        s = carve(bufs, [&](Carve &c) {
            ci2 = c.take<int32_t>((size_t)nnz2);
            X2 = c.take<double>((size_t)nnz2 * BB);
            A2 = c.take<double>((size_t)nnz2 * BB);
            key = c.take<unsigned long long>((size_t)nnz2);
        });
        if (s != ABILU_OK) return s;
        k_lu_pattern<true><<<counted(grid_rows(n, PLU_THREADS)), PLU_THREADS, 0, st>>>(
            n, VC.rowptr, VC.colind, VC.diagpos, nullptr, rp2, ci2, err);
        ABILU_LAUNCH_CHECK("k_lu_pattern");
        k_map_blocks<<<counted(grid_rows(n, PLU_THREADS / 4)), PLU_THREADS, 0, st>>>(
            n, rp2, ci2, VC.rowptr, VC.colind, X, VA.rowptr, VA.colind, A, X2, A2);
        ABILU_LAUNCH_CHECK("k_map_blocks");
        PatternGuard p2;
        if ((s = abilu_pattern_create(n, nnz2, rp2, ci2, stream, &p2.p)) != ABILU_OK) return s;
        {
            FactorsGuard f2;
            if ((s = factors_from(p2.p, X2, D, A2, o->sweeps, st, &f2.f)) != ABILU_OK) return s;
            if ((s = export_dispatch(f2.f, X2, D, st)) != ABILU_OK) return s;
            ABILU_CUDA(cudaStreamSynchronize(st));
        }
        // drop: the largest strictly lower and strictly upper blocks
        const PatternView &V2 = p2.p->v;
        k_block_norm2<<<counted(grid_rows(nnz2, 256)), 256, 0, st>>>(X2, nnz2, reinterpret_cast<double *>(key));
        ABILU_LAUNCH_CHECK("k_block_norm2");
        const bool all_l = (long long)V2.nl <= bl, all_u = (long long)V2.nu <= bu;
        if (!all_l || !all_u) {
            s = select_thresholds(n, V2.rowptr, V2.diagpos, key, bl, bu, sel, st);
            if (s != ABILU_OK) return s;
        }
        k_compact<false><<<counted(grid_rows(n, PLU_THREADS / 4)), PLU_THREADS, 0, st>>>(
            n, V2.rowptr, V2.colind, key, sel, all_l, all_u, rowcnt, nullptr, nullptr, nullptr,
            nullptr, nullptr, nullptr);
        ABILU_LAUNCH_CHECK("k_compact");
        if ((s = scan_i32(rowcnt, rp3, n, scratch, err, st)) != ABILU_OK) return s;
        int32_t nnz3 = 0;
        if ((s = read_total(rp3 + n, err, st, &nnz3)) != ABILU_OK) return s;
        int32_t *ci3 = nullptr;
        double *X3 = nullptr, *A3 = nullptr;
        s = carve(bufs, [&](Carve &c) {
            ci3 = c.take<int32_t>((size_t)nnz3);
            X3 = c.take<double>((size_t)nnz3 * BB);
            A3 = c.take<double>((size_t)nnz3 * BB);
        });
        if (s != ABILU_OK) return s;
        k_compact<true><<<counted(grid_rows(n, PLU_THREADS / 4)), PLU_THREADS, 0, st>>>(
            n, V2.rowptr, V2.colind, key, sel, all_l, all_u, nullptr, rp3, ci3, X2, A2, X3, A3);
        ABILU_LAUNCH_CHECK("k_compact");
        PatternGuard p3;
        if ((s = abilu_pattern_create(n, nnz3, rp3, ci3, stream, &p3.p)) != ABILU_OK) return s;
        FactorsGuard f3;
        if ((s = factors_from(p3.p, X3, D, A3, o->sweeps, st, &f3.f)) != ABILU_OK) return s;
        if (it == o->iters - 1) {
            if (o->factor_dtype != ABILU_F64) {
                FactorsGuard fn;
                s = o->factor_dtype == ABILU_F32
                        ? store_as<float>(f3.f, ABILU_F32, X3, D, st, &fn.f)
                        : store_as<__nv_bfloat16>(f3.f, ABILU_BF16, X3, D, st, &fn.f);
                if (s != ABILU_OK) return s;
                std::swap(f3.f, fn.f);   // the FP64 factors are released with fn
            }
            if ((s = factors_add_status(f3.f)) != ABILU_OK) return s;
            ABILU_CUDA(cudaStreamSynchronize(st));
            *pattern_out = p3.p;
            *factors_out = f3.f;
            p3.p = nullptr;
            f3.f = nullptr;
            return ABILU_OK;
        }
        if ((s = export_dispatch(f3.f, X3, D, st)) != ABILU_OK) return s;
        ABILU_CUDA(cudaStreamSynchronize(st));
        X = X3;
        std::swap(pcur.p, p3.p);   // the old current pattern is released with p3
    }
    return fail(ABILU_EINVAL, "abilu_parilut: unreachable");
}
