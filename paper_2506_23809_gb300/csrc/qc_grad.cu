// qc_grad.cu -- Eq. 4 (Sec. II-A): the energy gradient
//   d<E>/d theta_p = 2 Re < d_theta_p ln Psi*(n) (E_loc(n) - <E>) >_n
// as a count-weighted average over the unique samples of one evaluation.  Three device steps:
//   K5 grad_weights_kernel   w_i = c_i (E_loc,i - Ebar) / W   (0 where E_loc is not finite)
//   K6 grad_contract_kernel  partial_rp = sum over rows of chunk r of Re(w_i D_ip)
//   K7 grad_finish_kernel    g_p = 2 sum_r partial_rp   (fixed order: deterministic)
// Ebar and W come from the evaluation's device summary (written by the Eq. 1 reduction on
// the same stream), so the call is asynchronous.  The contraction streams the n_u x P
// complex rows D = d ln Psi* once from HBM (16 B per element, 16-byte streaming loads,
// coalesced along a row): 0.97 ms for 1e5 x 4,096 at the 6.78 TB/s of a copy.  Two FP64
// fused multiply-adds per element would take 1.38 ms (the FP64 pipe retires two per clock and
// SM), so the real parts go through that pipe and the imaginary parts through integer
// multiplications (FixedSum), which run beside it: 1.44 -> 0.98 ms a call, 6.7 TB/s.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "qc_eloc.h"
#include "qc_handle.h"
#include "qc_internal.h"

namespace {

constexpr int kGradThreads = 256;
constexpr int kGradRowsMax = 256;  // rows of a chunk staged in shared memory at a time
constexpr int kGradLoads = 4;      // row elements in flight per thread

__device__ __forceinline__ double2 weight(const double2 e, const long long c, const qc_eloc_summary* sum) {
    const double W = sum->w;
    if (!(W > 0.0) || c < 0 || !isfinite(e.x) || !isfinite(e.y)) return make_double2(0.0, 0.0);
    const double s = static_cast<double>(c) / W;
    return make_double2(s * (e.x - sum->e_re), s * (e.y - sum->e_im));
}

__global__ void __launch_bounds__(256) grad_weights_kernel(const double2* __restrict__ eloc,
                                                           const long long* __restrict__ counts, long long n,
                                                           const qc_eloc_summary* __restrict__ sum,
                                                           double2* __restrict__ w) {
    for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
         i += static_cast<long long>(gridDim.x) * blockDim.x)
        w[i] = weight(eloc[i], counts[i], sum);
}

// One staged row: its weight, and the imaginary weight's mantissa (the leading bit at bit 63),
// biased exponent and the sign of -w.y as a mask.  A weight that is zero, subnormal or not
// finite has an exponent of its own that puts each of its products out of FixedSum's window.
struct __align__(16) GradRow {
    double2 w;
    unsigned mhi, mlo;
    int ex;
    unsigned neg;
};
constexpr int kNotFinite = 1 << 20, kSubnormal = -kNotFinite, kZero = -2 * kNotFinite;

__device__ __forceinline__ GradRow grad_row(double2 w) {
    const unsigned hi = static_cast<unsigned>(__double2hiint(w.y)), lo = static_cast<unsigned>(__double2loint(w.y));
    const int ex = static_cast<int>((hi >> 20) & 0x7ffu);
    GradRow r;
    r.w = w;
    r.mhi = 0x80000000u | __funnelshift_l(lo, hi, 11);
    r.mlo = lo << 11;
    r.ex = ex == 0 ? (w.y == 0.0 ? kZero : kSubnormal) : ex == 0x7ff ? kNotFinite : ex;
    r.neg = static_cast<unsigned>(~static_cast<int>(hi) >> 31);
    return r;
}

// A sum of FP64 products in 128-bit fixed point, on the integer pipes.  A product is the top 64
// bits of the mantissas' product (short of it by less than 3 units of its last place: 2^-61
// relative, and exact where it fits 53 bits), added whole at the place its exponent gives: the unit
// of the sum is 2^(lim - kUnit), a product of exponents ex + ed sits s = lim - (ex + ed) places below
// the top word, and at s >= kMinShift 2^8 of them cannot overflow.  So in the window [kMinShift, 64)
// of 55 binades no product loses anything to larger ones, which may have cancelled by the end (with
// 96 bits a product 2^42 below the window's top kept 33 bits: 200 rows of which two cancel, 2^30
// above the rest, were off by 2e-8).  A larger product moves the sum so far into the FP64
// accumulator and lays it out anew, kMargin places above that product; one below the window, a
// subnormal, an infinity or NaN goes to the FP64 accumulator by a fused multiply-add.
constexpr int kMinShift = 9, kMargin = 12, kUnit = 2 * 1023 + 62 + 64;
struct FixedSum {
    unsigned a0 = 0, a1 = 0, a2 = 0, a3 = 0;
    int lim = 0;

    // adds -w.y * d; returns false when the product does not fit (nothing is added then).  A zero
    // fits, unless its other factor is not finite: it is no exception but a user's ordinary input --
    // a real wave function has w.y = 0 in every row, a real derivative d = 0 in a whole column, a
    // dead unit some of one.  (As exceptions 1e5 x 4,096 of them took 1.47 ms, a tenth of them
    // scattered 1.64; now 1.00 and 1.04, dense rows 1.03.)
    __device__ __forceinline__ bool add(const GradRow& r, double d) {
        const unsigned hi = static_cast<unsigned>(__double2hiint(d)), lo = static_cast<unsigned>(__double2loint(d));
        const int ed = static_cast<int>((hi >> 20) & 0x7ffu);
        const int s = lim - r.ex - ed;
        const bool ok = static_cast<unsigned>(ed - 1) < 0x7feu && static_cast<unsigned>(s - kMinShift) < 64u - kMinShift;
        const bool zero = ((hi & 0x7fffffffu) | lo) == 0u ? r.ex != kNotFinite : s >= -kZero - 0x7ff && ed != 0x7ff;
        const unsigned keep = ok ? 0xffffffffu : 0u;
        const unsigned mhi = 0x80000000u | __funnelshift_l(lo, hi, 11), mlo = lo << 11;
        const unsigned neg = static_cast<unsigned>(static_cast<int>(hi) >> 31) ^ r.neg;
        unsigned long long p = static_cast<unsigned long long>(mhi) * r.mhi + __umulhi(mhi, r.mlo);
        p += __umulhi(mlo, r.mhi);
        // the one's complement of a negative product, to the last bit of the sum, and a carry into it
        const unsigned m = neg & keep;
        const unsigned pl = (static_cast<unsigned>(p) ^ neg) & keep, ph = (static_cast<unsigned>(p >> 32) ^ neg) & keep;
        const unsigned f0 = __funnelshift_r(m, pl, s), f1 = __funnelshift_r(pl, ph, s), f2 = __funnelshift_r(ph, m, s);
        const bool far = s >= 32;
        const unsigned w0 = far ? f0 : m, w1 = far ? f1 : f0, w2 = far ? f2 : f1, w3 = far ? m : f2;
        asm("{\n\t.reg .u32 c;\n\tadd.cc.u32 c, %8, 1;\n\t"
            "addc.cc.u32 %0, %0, %4;\n\taddc.cc.u32 %1, %1, %5;\n\taddc.cc.u32 %2, %2, %6;\n\taddc.u32 %3, %3, %7;\n\t}"
            : "+r"(a0), "+r"(a1), "+r"(a2), "+r"(a3)
            : "r"(w0), "r"(w1), "r"(w2), "r"(w3), "r"(m));
        return ok || zero;
    }
    // the sum so far; it starts again from zero, with no layout
    __device__ __forceinline__ double take() {
        const bool neg = static_cast<int>(a3) < 0;
        unsigned long long h = (static_cast<unsigned long long>(a3) << 32) | a2, l = (static_cast<unsigned long long>(a1) << 32) | a0;
        if (neg) {
            l = ~l + 1ULL;
            h = ~h + (l == 0ULL ? 1ULL : 0ULL);
        }
        const double v = fma(__ull2double_rn(h), 18446744073709551616.0, __ull2double_rn(l));
        const int e = lim - kUnit;
        a0 = a1 = a2 = a3 = 0u;
        lim = 0;
        return v == 0.0 ? 0.0 : ldexp(neg ? -v : v, e);
    }
};

struct GradSum {
    FixedSum f;
    double acc;
};

// A product above the window, the first of its sum, or one that a layout made since its add has
// taken in (by value, out of line: its operands stay in registers elsewhere).
__device__ __noinline__ GradSum place_product(GradSum g, GradRow r, double d) {
    const int ed = (__double2hiint(d) >> 20) & 0x7ff;
    if (ed == 0 || ed == 0x7ff || r.ex < 0 || r.ex == kNotFinite) {
        g.acc = fma(-r.w.y, d, g.acc);
        return g;
    }
    if (g.f.lim - r.ex - ed < kMinShift) {
        g.acc += g.f.take();
        g.f.lim = r.ex + ed + kMinShift + kMargin;
    }
    g.f.add(r, d);
    return g;
}

// Whether a product that add left out belongs into the fixed-point sum (place_product); if not, it
// is below the window or not a normal number and goes to the FP64 accumulator.
__device__ __forceinline__ bool to_place(const GradSum& g, const GradRow& r, double d) {
    const int ed = (__double2hiint(d) >> 20) & 0x7ff;
    return g.f.lim - r.ex - ed < 64 && ed != 0 && ed != 0x7ff;
}

// One CTA: 256 >> shift consecutive columns of one chunk of rows, the rows dealt over
// 1 << shift groups of its threads, whose sums are added in a fixed order.  The chunk's
// weights are staged in shared memory; every thread walks its rows of its column, kGradLoads
// loads in flight.
__global__ void __launch_bounds__(kGradThreads, 4)
    grad_contract_kernel(const double2* __restrict__ eloc, const long long* __restrict__ counts,
                         const double2* __restrict__ w, long long n, const qc_eloc_summary* __restrict__ sum,
                         const double2* __restrict__ D, long long P, long long rows_per_chunk, int shift,
                         double* __restrict__ part) {
    __shared__ GradRow ws[kGradRowsMax];
    const int cols = kGradThreads >> shift, groups = 1 << shift;
    const int col = threadIdx.x & (cols - 1), grp = threadIdx.x / cols;
    const long long p = static_cast<long long>(blockIdx.x) * cols + col;
    const long long r0 = static_cast<long long>(blockIdx.y) * rows_per_chunk;
    const long long r1 = r0 + rows_per_chunk < n ? r0 + rows_per_chunk : n;
    GradSum g{};
    for (long long b = r0; b < r1; b += kGradRowsMax) {
        const int nb = static_cast<int>(r1 - b < kGradRowsMax ? r1 - b : kGradRowsMax);
        __syncthreads();
        for (int t = threadIdx.x; t < nb; t += kGradThreads)
            ws[t] = grad_row(w != nullptr ? w[b + t] : weight(eloc[b + t], counts[b + t], sum));
        __syncthreads();
        if (p < P) {
            const double2* row = D + (b + grp) * P + p;
            const long long step = static_cast<long long>(groups) * P;
            int t = grp;
            for (; t + (kGradLoads - 1) * groups < nb; t += kGradLoads * groups) {
                double2 d[kGradLoads];
#pragma unroll
                for (int k = 0; k < kGradLoads; ++k) {
                    d[k] = __ldcs(row);
                    row += step;
                }
                if (t == grp) {  // a stage's first rows: the sum is laid out by the largest of them
                    int top = 0;
#pragma unroll
                    for (int k = 0; k < kGradLoads; ++k) {
                        const int ex = ws[t + k * groups].ex, ed = (__double2hiint(d[k].y) >> 20) & 0x7ff;
                        if (ex > 0 && ex < kNotFinite && ed != 0 && ed != 0x7ff && ex + ed > top) top = ex + ed;
                    }
                    if (top != 0) g.f.lim = top + kMinShift + kMargin;
                }
                bool ok[kGradLoads];
#pragma unroll
                for (int k = 0; k < kGradLoads; ++k) {
                    const GradRow r = ws[t + k * groups];
                    g.acc = fma(r.w.x, d[k].x, g.acc);
                    ok[k] = g.f.add(r, d[k].y);
                }
                if (!(ok[0] && ok[1] && ok[2] && ok[3])) {
#pragma unroll
                    for (int k = 0; k < kGradLoads; ++k)
                        if (!ok[k]) {
                            const GradRow& r = ws[t + k * groups];
                            if (to_place(g, r, d[k].y)) g = place_product(g, r, d[k].y);
                            else g.acc = fma(-r.w.y, d[k].y, g.acc);
                        }
                }
            }
            for (; t < nb; t += groups) {
                const double2 d = __ldcs(row);
                row += step;
                const GradRow r = ws[t];
                g.acc = fma(r.w.x, d.x, g.acc);
                if (!g.f.add(r, d.y)) {
                    if (to_place(g, r, d.y)) g = place_product(g, r, d.y);
                    else g.acc = fma(-r.w.y, d.y, g.acc);
                }
            }
            g.acc += g.f.take();
        }
    }
    if (groups > 1) {
        __syncthreads();
        double* sh = reinterpret_cast<double*>(ws);
        sh[threadIdx.x] = g.acc;
        __syncthreads();
        if (grp != 0) return;
        for (int k = 1; k < groups; ++k) g.acc += sh[k * cols + col];
    }
    if (p < P) part[static_cast<long long>(blockIdx.y) * P + p] = g.acc;
}

// One CTA: 32 columns, each chunk's partials coalesced; 32 groups of threads take chunks
// g, g + 32, .. and are added by halves (one thread a column walked all 512 chunks in 40 us).
constexpr int kFinishGroups = 32;
__global__ void __launch_bounds__(32 * kFinishGroups) grad_finish_kernel(const double* __restrict__ part, int chunks,
                                                                        long long P, double* __restrict__ g) {
    __shared__ double sh[kFinishGroups][32];
    const int col = threadIdx.x & 31, grp = threadIdx.x >> 5;
    const long long p = static_cast<long long>(blockIdx.x) * 32 + col;
    double s = 0.0;
    if (p < P)
#pragma unroll 4
        for (int r = grp; r < chunks; r += kFinishGroups) s += part[static_cast<long long>(r) * P + p];
    sh[grp][col] = s;
    __syncthreads();
    for (int h = kFinishGroups / 2; h > 0; h >>= 1) {
        if (grp < h) sh[grp][col] += sh[grp + h][col];
        __syncthreads();
    }
    if (grp == 0 && p < P) g[p] = 2.0 * sh[0][col];
}

// The contraction's split: columns per CTA (256 >> shift), rows per chunk and chunks.  A function
// of the sizes only (not of the GPU), so the summation order, and the result, are the same
// everywhere.  Up to 128 columns the CTA's threads share the rows; the chunks fill whole waves of
// kGradWave CTAs (four on each of 152 SMs) with at most 256 rows a CTA (more only beyond
// kGradChunksMax x 256 rows) and at least 8 a thread, as a CTA starts and ends with some twenty
// FP64 operations a thread (5,723 x 2,816: 64-row chunks of 256 columns 80 us, of 32 columns
// 126 us).
constexpr long long kGradWave = 608, kGradChunksMax = 512;
struct GradSplit {
    int shift, chunks;
    long long tiles, rows;
};
GradSplit grad_split(long long n, long long P) {
    GradSplit g{};
    while (g.shift < 3 && P <= (kGradThreads >> (g.shift + 1))) ++g.shift;
    const long long cols = kGradThreads >> g.shift;
    g.tiles = (P + cols - 1) / cols;
    const long long waves = std::max<long long>(1, (g.tiles * ((n + 255) / 256) + kGradWave - 1) / kGradWave);
    const long long most = std::min<long long>(kGradChunksMax, (n + (8LL << g.shift) - 1) / (8LL << g.shift));
    const long long chunks = std::max<long long>(1, std::min(most, kGradWave * waves / g.tiles));
    g.rows = (n + chunks - 1) / chunks;
    g.chunks = static_cast<int>((n + g.rows - 1) / g.rows);
    return g;
}

// The most chunks that a call of up to n rows splits into, whatever its columns: the partials'
// buffer is sized by it, so that a later call that is no larger in rows and columns fits (the
// split itself is not monotone: 2,433 x 300 has 271 chunks, 2,432 x 300 has 304).
long long grad_chunks_bound(long long n) { return std::min<long long>(kGradChunksMax, (n + 7) / 8); }

}  // namespace

extern "C" qc_status qc_eloc_grad(qc_eloc* H, const double* eloc, const int64_t* counts, int64_t n_u,
                                  const double* dconj, int64_t n_par, double* w_out, double* g_out,
                                  void* stream) {
    if (!H) return QC_ERR_ARG;
    auto fail = [&](qc_status st, const char* m) {
        H->err = m;
        return st;
    };
    if (n_u < 0 || n_par < 0) return fail(QC_ERR_ARG, "negative size");
    if (n_u > 0 && (!eloc || !counts)) return fail(QC_ERR_ARG, "eloc or counts is NULL");
    if (g_out && n_par > 0 && !dconj) return fail(QC_ERR_ARG, "g_out needs dconj");
    auto mis = [](const void* q, unsigned a) { return q && (reinterpret_cast<uintptr_t>(q) & (a - 1)) != 0; };
    if (mis(eloc, 16) || mis(dconj, 16) || mis(w_out, 16) || mis(counts, 8) || mis(g_out, 8))
        return fail(QC_ERR_ARG, "device arrays must be 16-byte aligned (counts, g_out: 8)");
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != H->device) return fail(QC_ERR_ARG, "handle belongs to another device");
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const double2* e2 = reinterpret_cast<const double2*>(eloc);
    const long long* c = reinterpret_cast<const long long*>(counts);
    cudaError_t e = cudaSuccess;
    if (w_out && n_u > 0) {
        const long long blocks = std::min<long long>((n_u + 255) / 256, 4096);
        grad_weights_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(e2, c, n_u, H->d_sum,
                                                                          reinterpret_cast<double2*>(w_out));
        e = cudaGetLastError();
    }
    if (e == cudaSuccess && g_out && n_par > 0) {
        if (n_u == 0) {
            e = cudaMemsetAsync(g_out, 0, static_cast<size_t>(n_par) * sizeof(double), s);
        } else {
            const GradSplit sp = grad_split(n_u, n_par);
            const int chunks = sp.chunks;
            const size_t need = static_cast<size_t>(grad_chunks_bound(n_u)) * static_cast<size_t>(n_par);
            if (need > H->gpart_cap) {
                if (H->d_gpart) cudaFree(H->d_gpart);
                H->d_gpart = nullptr;
                H->gpart_cap = 0;
                e = qc::dev_alloc(&H->d_gpart, need * sizeof(double));
                if (e == cudaSuccess) H->gpart_cap = need;
            }
            if (e == cudaSuccess) {
                if (sp.tiles > 0x7fffffffLL) return fail(QC_ERR_CAPACITY, "n_par too large");
                grad_contract_kernel<<<dim3(static_cast<unsigned>(sp.tiles), static_cast<unsigned>(chunks)), kGradThreads,
                                       0, s>>>(e2, c, reinterpret_cast<const double2*>(w_out), n_u, H->d_sum,
                                               reinterpret_cast<const double2*>(dconj), n_par, sp.rows, sp.shift,
                                               H->d_gpart);
                e = cudaGetLastError();
            }
            if (e == cudaSuccess) {
                grad_finish_kernel<<<static_cast<unsigned>((n_par + 31) / 32), 32 * kFinishGroups, 0, s>>>(
                    H->d_gpart, chunks, n_par, g_out);
                e = cudaGetLastError();
            }
        }
    }
    if (e != cudaSuccess) {
        H->err = std::string("qc_eloc_grad: ") + cudaGetErrorString(e);
        return e == cudaErrorMemoryAllocation ? QC_ERR_OOM : QC_ERR_CUDA;
    }
    return QC_OK;
}
