// Row q of block row i of A times x, FP64: the SpMV's inner product, shared by
// the product kernel and the residual kernels so that every FP64 product of A
// runs the same operations.  The first four blocks' loads are issued before
// any arithmetic, so each thread keeps up to 8 independent 16-byte loads in
// flight.  Blocks in order, within a block x_j[0..3]; the third and fourth
// blocks' eight products are summed with integer instructions (fx_dot8).
#pragma once
#include <atomic>

#include "common.cuh"

namespace abilu {

// sum_k a[k] x[k], k < 8, in integer arithmetic, rounded once to FP64.
//
// Why: this GPU executes two FP64 FMA per SM and clock, so a row's 16 FMAs
// take longer (53 us per product of 2.1 M blocks at 100% of that pipe) than its
// 528 bytes take to arrive (47 us), while the integer lanes idle: 64 issue
// slots pass per warp-wide FP64 FMA, and an integer product-and-add below is
// about 25 instructions.  With half of a row's products here that pipe is 52%
// busy and the integer pipe 43% (all FMA: 86% and little), and a row's chain of
// dependent FMAs is half as long.  512x512 (us): product 65.7 -> 60.8, fused
// product and dots of one to five vectors 76-95 -> 73-91, residual 78 -> 71;
// 2.6 M rows, batch: fused 358 -> 330.  One block of four in integers gained
// nothing (75 us: its chain is as long, its share of the pipe small).
//
// Precision: each product of two 53-bit significands, aligned to the largest
// product's exponent, is kept to 2^-58 of the largest product (off by at most
// three such units) and added exactly in 64 bits; the sum is rounded once: at most
// 24 2^-58 of the largest product and half an ulp of the sum away.  Eight FP64 FMAs
// round eight times, to 2^-53 of the running sum.  On random products its error was
// half of theirs (rms 6.5e-17 against 1.4e-16 of the largest product, largest 5.8e-16
// against 1.4e-15), and a whole product of the 512x512 grid is 1.1e-16 from the
// exact one where FMAs gave 1.5e-16.  The bound is relative to the largest product,
// not to the sum: where large products cancel before small ones are added, FMAs
// keep the small ones (1e20, -1e20, 1 in this order: 1) and this sum does not (0), as
// FMAs in another order would not.  Sums of integers stay exact while every partial sum
// of FMAs would be (operands up to 2^25: eight products of 2^50).
//
// Range: taken when every operand is below 2^478 in magnitude and the largest
// product is at least 2^-446: then a zero's or subnormal's product (exponent
// field 0, read as if normal) is shifted out entirely, which is its value to
// far below the rounding.  Otherwise (also Inf and NaN) FP64 FMAs.
__device__ __forceinline__ double fx_dot8(const double (&a)[8], const double (&x)[8]) {
    constexpr unsigned EXP = 0x7FF00000u;   // the exponent field of an operand's high word
    unsigned e[8], top = 0u, emax = 0u;     // e: the two exponents' sum, in place
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const unsigned ea = (unsigned)__double2hiint(a[k]) & EXP, ex = (unsigned)__double2hiint(x[k]) & EXP;
        e[k] = ea + ex;
        top = max(top, max(ea, ex));
        emax = max(emax, e[k]);
    }
    if (top > (1500u << 20) || emax < (1600u << 20)) {
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 8; k++) s = fma(a[k], x[k], s);
        return s;
    }
    long long acc = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
        const int ah = __double2hiint(a[k]), xh = __double2hiint(x[k]);
        const unsigned al = (unsigned)__double2loint(a[k]), xl = (unsigned)__double2loint(x[k]);
        // significands shifted up by 9 (62 bits)
        const unsigned ahi = __funnelshift_l(al, (unsigned)(ah & 0xFFFFF) | 0x100000u, 9), alo = al << 9;
        const unsigned xhi = __funnelshift_l(xl, (unsigned)(xh & 0xFFFFF) | 0x100000u, 9), xlo = xl << 9;
        const unsigned long long m = (unsigned long long)alo * xhi + (unsigned long long)ahi * xlo;
        unsigned long long r = (unsigned long long)ahi * xhi + (m >> 32);   // 2^58 .. 2^60
        r >>= min((emax - e[k]) >> 20, 63u);
        const int sg = (ah ^ xh) >> 31;   // 0 or -1
        acc += ((long long)r ^ (long long)sg) + (long long)(sg & 1);
    }
    // |acc| < 2^63, to FP64
    if (acc == 0) return 0.0;
    const unsigned sgn = (unsigned)((unsigned long long)acc >> 32) & 0x80000000u;
    unsigned long long u = (unsigned long long)(acc < 0 ? -acc : acc);
    const int z = __clzll((long long)u);
    u <<= z;                                   // bit 63 set
    unsigned long long f = (u >> 11) + ((u >> 10) & 1ull);   // 53 bits, rounded (may carry to 2^53)
    // the significands carry 2^1075 each and r 2^-46: value = u 2^(emax - 2104 - z)
    const int ef = (int)(emax >> 20) - 1018 - z;            // exponent field of bit 63
    f += ((unsigned long long)(unsigned)(ef - 1)) << 52;     // adds the hidden bit's one
    return __hiloint2double((int)((unsigned)(f >> 32) | sgn), (int)(unsigned)f);
}

__device__ __forceinline__ double row_dot_blocks(const PatternView &P, const double *__restrict__ A,
                                                 const double *__restrict__ x, int i, int q) {
    const int p0 = P.rowptr[i], p1 = P.rowptr[i + 1];
    double2 a0[4], a1[4];
    int jj[4];
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const int p = p0 + k;
        if (p < p1) {
            jj[k] = __ldg(P.colind + p);
            const double2 *ap = reinterpret_cast<const double2 *>(A + (size_t)p * BB + q * BS);
            a0[k] = __ldg(ap);
            a1[k] = __ldg(ap + 1);
        } else {
            jj[k] = -1;
        }
    }
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        if (jj[k] >= 0) {
            const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)jj[k] * BS);
            double2 x0 = __ldg(xp), x1 = __ldg(xp + 1);
            s = fma(a0[k].x, x0.x, s);
            s = fma(a0[k].y, x0.y, s);
            s = fma(a1[k].x, x1.x, s);
            s = fma(a1[k].y, x1.y, s);
        }
    }
    if (jj[2] >= 0) {
        double av[8], xv[8];
#pragma unroll
        for (int k = 2; k < 4; k++) {
            double2 x0 = make_double2(0.0, 0.0), x1 = x0;
            if (jj[k] >= 0) {
                const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)jj[k] * BS);
                x0 = __ldg(xp);
                x1 = __ldg(xp + 1);
            } else {
                a0[k] = a1[k] = x0;
            }
            double *ak = av + 4 * (k - 2), *xk = xv + 4 * (k - 2);
            ak[0] = a0[k].x; ak[1] = a0[k].y; ak[2] = a1[k].x; ak[3] = a1[k].y;
            xk[0] = x0.x; xk[1] = x0.y; xk[2] = x1.x; xk[3] = x1.y;
        }
        s += fx_dot8(av, xv);
    }
    for (int p = p0 + 4; p < p1; p++) {  // rows longer than four blocks
        const int j = __ldg(P.colind + p);
        const double2 *ap = reinterpret_cast<const double2 *>(A + (size_t)p * BB + q * BS);
        const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)j * BS);
        double2 b0 = __ldg(ap), b1 = __ldg(ap + 1), x0 = __ldg(xp), x1 = __ldg(xp + 1);
        s = fma(b0.x, x0.x, s);
        s = fma(b0.y, x0.y, s);
        s = fma(b1.x, x1.x, s);
        s = fma(b1.y, x1.y, s);
    }
    return s;
}

// ---- large systems: the rows' blocks and their x through shared memory
//
// One CTA per SM takes 160 rows at a time and has the next 160 rows' first four
// blocks and the x they meet in flight into a second shared-memory stage while
// it works on the current ones: 16-byte cp.async copies, waited for by the
// copying warp alone (a wait instruction, no polling), so no block-wide barrier,
// no registers for blocks in flight (32 in row_dot_blocks, which spilled in the
// fused kernels) and no gather on a row's critical path: pointers are read three
// rows ahead, columns two.  512x512 (us, direct -> streamed; 47 are the bytes at
// the copy rate): product 60.8 -> 51.0, residual 71 -> 61, fused product and 1 .. 5
// dots 72, 79, 82, 91, 91 -> 64, 67, 71, 75, 80.  Gathers of x left to the row's own
// loads: product 58.
// One CTA per SM and not three: behind the staged sweeps, whose CTAs leave an SM
// one by one, three CTAs of 64 KB did not always fit side by side, and the grid
// took two waves (fused kernels of 73 .. 91 us took 96 .. 150).
//
// A quad's copies of blocks are 64 contiguous bytes per instruction; odd rows
// swap the 16-byte halves of each 32 bytes, so the lanes of a shared-memory phase
// (two rows) use distinct banks.
constexpr int STREAM_THREADS = 640;
constexpr int STREAM_ROWS = STREAM_THREADS / 4;
constexpr int STREAM_SLOT = 4 * BB * (int)sizeof(double) + 4 * BS * (int)sizeof(double);   // 640 bytes a row
constexpr int STREAM_STAGE = STREAM_ROWS * STREAM_SLOT;
constexpr int STREAM_SMEM = 2 * STREAM_STAGE;                                              // 200 KB

__device__ __forceinline__ void cp_async16_cg(unsigned dst, const void *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async16_ca(unsigned dst, const void *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// the positions of a row's blocks; thread q of the quad: the column of block p0 + q
struct StreamRow {
    int p0, p1, jq;
    __device__ __forceinline__ void ptrs(const PatternView &P, int i, int end) {
        p0 = p1 = 0;
        if (i < end) {
            p0 = __ldg(P.rowptr + i);
            p1 = __ldg(P.rowptr + i + 1);
        }
    }
    __device__ __forceinline__ void col(const PatternView &P) {
        const int p = p0 + (int)(threadIdx.x & 3);
        jq = p < p1 ? __ldg(P.colind + p) : -1;
    }
};

// copies of the row's first four blocks and their x into the quad's slot (zeros
// where the row has fewer)
__device__ __forceinline__ void stream_issue(const double *__restrict__ A, const double *__restrict__ x,
                                             unsigned slot, const StreamRow &r) {
    const int q = threadIdx.x & 3, sw = (threadIdx.x >> 2) & 1;
    const unsigned dst = slot + (unsigned)((q ^ sw) * 16);
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const bool in = r.p0 + k < r.p1;
        const double *src = A + (in ? (size_t)(r.p0 + k) * BB + q * 2 : 0);
        cp_async16_cg(dst + k * 128, src, in ? 16 : 0);
        cp_async16_cg(dst + k * 128 + 64, in ? src + 8 : src, in ? 16 : 0);
    }
    const bool in = r.jq >= 0;
    const double *src = x + (in ? (size_t)r.jq * BS : 0);
    const unsigned xd = slot + 512u + (unsigned)(q * 32);
    cp_async16_ca(xd + (unsigned)(sw * 16), src, in ? 16 : 0);
    cp_async16_ca(xd + (unsigned)((sw ^ 1) * 16), in ? src + 2 : src, in ? 16 : 0);
}

// entry q of the row in the quad's slot: row_dot_blocks's operations
__device__ __forceinline__ double stream_dot(const PatternView &P, const double *__restrict__ A,
                                             const double *__restrict__ x, const char *slot, int p0, int p1) {
    const int q = threadIdx.x & 3, sw = (threadIdx.x >> 2) & 1;
    const char *alo = slot + ((2 * q) ^ sw) * 16, *ahi = slot + ((2 * q + 1) ^ sw) * 16;
    const char *xlo = slot + 512 + sw * 16, *xhi = slot + 512 + (sw ^ 1) * 16;
    auto ld = [](const char *p) { return *reinterpret_cast<const double2 *>(p); };
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < 2; k++) {
        const double2 a0 = ld(alo + k * 128), a1 = ld(ahi + k * 128), x0 = ld(xlo + k * 32), x1 = ld(xhi + k * 32);
        s = fma(a0.x, x0.x, s);
        s = fma(a0.y, x0.y, s);
        s = fma(a1.x, x1.x, s);
        s = fma(a1.y, x1.y, s);
    }
    if (p1 - p0 > 2) {
        double av[8], xv[8];
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const double2 a0 = ld(alo + 256 + k * 128), a1 = ld(ahi + 256 + k * 128);
            const double2 x0 = ld(xlo + 64 + k * 32), x1 = ld(xhi + 64 + k * 32);
            av[4 * k] = a0.x; av[4 * k + 1] = a0.y; av[4 * k + 2] = a1.x; av[4 * k + 3] = a1.y;
            xv[4 * k] = x0.x; xv[4 * k + 1] = x0.y; xv[4 * k + 2] = x1.x; xv[4 * k + 3] = x1.y;
        }
        s += fx_dot8(av, xv);
    }
    for (int p = p0 + 4; p < p1; p++) {  // rows longer than four blocks
        const int j = __ldg(P.colind + p);
        const double2 *ap = reinterpret_cast<const double2 *>(A + (size_t)p * BB + q * BS);
        const double2 *xp = reinterpret_cast<const double2 *>(x + (size_t)j * BS);
        double2 b0 = __ldg(ap), b1 = __ldg(ap + 1), x0 = __ldg(xp), x1 = __ldg(xp + 1);
        s = fma(b0.x, x0.x, s);
        s = fma(b0.y, x0.y, s);
        s = fma(b1.x, x1.x, s);
        s = fma(b1.y, x1.y, s);
    }
    return s;
}

// The CTA's rows blockIdx.x * TH / 4 .., a grid stride of TH / 4 rows per CTA,
// below n: post(i, (A x)_i[q], pre(i)) in the quad of row i, pre's loads issued
// before the row's product.  TH = STREAM_THREADS: through `smem`, the CTA's
// STREAM_SMEM bytes, free again after a block-wide barrier; else directly.  ONE:
// the grid covers the rows, no loop (the direct form then fits 64 registers and
// four CTAs per SM; product of 262k rows of 9 blocks 75.4 -> 65.1 us, 524k of 4
// 68.4 -> 62.9).  Every thread of the CTA calls it.
template <int TH, bool ONE = false, typename Pre, typename Post>
__device__ __forceinline__ void for_rows(const PatternView &P, const double *__restrict__ A,
                                         const double *__restrict__ x, char *smem, Pre pre, Post post) {
    const int q = threadIdx.x & 3, n = P.n, step = gridDim.x * (TH / 4);
    int i = blockIdx.x * (TH / 4) + (threadIdx.x >> 2);
    if constexpr (TH != STREAM_THREADS) {
        for (; i < n; i += step) {
            auto v = pre(i);
            post(i, row_dot_blocks(P, A, x, i, q), v);
            if constexpr (ONE) return;
        }
    } else {
        int wi = i - (int)((threadIdx.x & 31) >> 2);   // the warp's first row: its loop is uniform
        if (wi >= n) return;
        char *slot = smem + (threadIdx.x >> 2) * STREAM_SLOT;
        const unsigned uslot = (unsigned)__cvta_generic_to_shared(slot);
        StreamRow r, r1, r2;
        r.ptrs(P, i, n);
        r1.ptrs(P, i + step, n);
        r2.ptrs(P, i + 2 * step, n);
        r.col(P);
        r1.col(P);
        stream_issue(A, x, uslot, r);
        asm volatile("cp.async.commit_group;" ::: "memory");
        for (int off = 0;; off = STREAM_STAGE - off) {
            const bool more = wi + step < n;
            if (more) stream_issue(A, x, uslot + (unsigned)(STREAM_STAGE - off), r1);
            asm volatile("cp.async.commit_group;" ::: "memory");
            r2.col(P);
            StreamRow r3;
            r3.ptrs(P, i + 3 * step, n);
            auto v = pre(i < n ? i : n - 1);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
            __syncwarp();   // the quad's other copies
            if (i < n) post(i, stream_dot(P, A, x, slot + off, r.p0, r.p1), v);
            if (!more) break;
            __syncwarp();   // every lane has read this stage
            r = r1;
            r1 = r2;
            r2 = r3;
            i += step;
            wi += step;
        }
    }
}

// Whether the streamed form takes a system, by rows and blocks per row (blocks
// five and on of a row are loaded from global memory as they are used, by 20 warps
// per SM; the direct form has 24 to 32).  Both forms measured (us, product / FGMRES
// solve of six steps, direct -> streamed): four blocks a row: 80k rows 10.6 / 314 ->
// 12.8 / 330, 120k 14.4 / 385 -> 13.9 / 385, 140k 17.1 / 417 -> 16.2 / 410, 262k 35.3 /
// 596 -> 29.6 / 588, 524k 63.2 / 960 -> 52.8 / 917 (120k: about five passes of 160 rows
// per SM pay for the pipeline's ramp).  Five: 200k 32.1 / 539 -> 30.9 / 548, 262k
// 39.7 / 646 -> 37.0 / 643, 700k 93.6 / 1,309 -> 85.5 / 1,267.  Six: 262k 47.1 / 723 ->
// 50.3 / 738, 700k 112.8 / 1,509 -> 118.8 / 1,505.  Nine, 262k: 65.1 -> 76.4; 26, 125k:
// 95.2 -> 127.5.
inline bool streamed(const PatternView &P) {
    const long long blocks = P.nnzb, n = P.n;
    return blocks <= 5 * n && n >= (2 * blocks <= 9 * n ? 120000 : 250000);
}
int sm_count();

// launch_pdl of a kernel of STREAM_THREADS threads with the stages (its dynamic
// shared memory allowed once per kernel and device)
template <auto K, typename... Args>
inline cudaError_t launch_stream(cudaStream_t st, Args &&...args) {
    static std::atomic<unsigned long long> allowed{0ull};
    int dev = 0;
    cudaGetDevice(&dev);
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(allowed.load(std::memory_order_relaxed) & bit)) {
        const cudaError_t e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, STREAM_SMEM);
        if (e != cudaSuccess) return e;
        allowed.fetch_or(bit, std::memory_order_relaxed);
    }
    return launch_pdl(K, sm_count(), STREAM_THREADS, STREAM_SMEM, st, std::forward<Args>(args)...);
}

}  // namespace abilu
