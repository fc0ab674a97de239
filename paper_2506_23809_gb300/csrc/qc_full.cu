// qc_full.cu -- the "accurate energy" of Sec. IV-C-4 at scale: the full connected set of
// every sample is handed to the caller (whose network evaluates psi on it), and Eq. 5 is
// then reduced against those values.
//   K8 eloc_export_kernel  every single and double excitation x' of each sample, its signed
//                          Slater-Condon element <x|H|x'> (Eq. 2, Sec. III-B (ii)) and the
//                          diagonal <x|H|x>, written in a fixed order (below)
//   K9 eloc_apply_kernel   E_loc(x) = <x|H|x> + sum_j <x|H|x'_j> psi(x'_j) / psi(x)
// followed by the Eq. 1 reduction (K3) over the chunk.
//
// Order of the connected set of one sample (P = pairs per sample, position = class offset
// + u * n2 + w): alpha singles, beta singles (w = occupied index * empty count + empty
// index, both over the spin's ascending lists), alpha-alpha and beta-beta doubles (u an
// occupied pair, w an empty pair; the pair (p < q) has index q (q - 1) / 2 + p), then
// alpha-beta doubles (u an alpha single, w a beta single).
//
// Both kernels stream HBM: the export writes 24 B per pair (key and element), the apply
// reads 24 B per pair (element and psi) plus two FP64 fused multiply-adds.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "qc_device.cuh"
#include "qc_eloc.h"
#include "qc_handle.h"
#include "qc_internal.h"

namespace qc {
namespace {

// ------------------------------------------------------------------------------------
// K8: export of the connected sets
// ------------------------------------------------------------------------------------
// The export writes 24 B per pair, so its floor is HBM's write rate; what bounds it below that
// is the work per pair.  One CTA takes a contiguous range of one sample's output (a work item
// from a device cursor).  For each double class the part of an excitation that its outer entry u
// fixes and the part that its inner entry w fixes are each formed once per item, in shared
// memory, as a record:
//   u: the key with u's orbitals flipped, the mask of orbitals strictly between u's two, its
//      share of the phase and of the integral indexes
//   w: the key bits of w's orbitals, their positions, share of the phase, integral offset
// A pair is then two key XORs, one or two integral loads, one subtraction for equal spins and
// three phase bits: the pairs [i < j] .. [b < a] of the phase reduce to "is w's first (second)
// orbital between u's two".  Consecutive pairs go to consecutive lanes, so keys and elements
// leave in whole sectors, and the integrals are read with w's fastest index innermost
// ((ai|jb); (jb|ia) and (ib|ja) for equal spins: the 8-fold symmetry of (pq|rs)), neighbouring
// lanes in neighbouring words.  Before, every lane decoded its excitation from scratch (193 warp
// instructions per 32 pairs, the FP64 pipe 59% busy with negations, gathers over strides of K^3).
// N=52, 10,000 samples: 1.72 ms (3.5 TB/s); now 1.03 ms (5.9 TB/s; 48 registers and five CTAs of
// 256 threads an SM; 61 registers and four: 1.09); N=120, 100 samples 2.67 -> 0.60 ms; N=104,
// 70 electrons, 12 samples 1.22 -> 0.065 ms.
constexpr long long kExpItemPairs = 10240;  // pairs of a work item (a single counts as export_single_weight)
constexpr int kExpUTile = 256;  // outer entries whose records are in shared memory at a time

struct ExportOut {
    ulonglong2* keys;   // [n_u * P] or null
    double* elems;      // [n_u * P] or null
    double* diag;       // [n_u] or null
};

struct alignas(16) ExpU {
    ulonglong2 key;            // x with u's orbitals flipped
    unsigned long long between;  // spatial orbitals (of w's spin) strictly between u's two
    unsigned d1;               // integral index share of (ai|bj), phase share in bit 31
    unsigned d2;               // of (aj|bi) (equal spins)
};

// shared memory of an item: occupation lists, u records, w key bits, w words
__host__ __device__ inline int exp_max_w(const SysParams& sp) {
    int n = sp.nsb;
    if (sp.npoa > 0 && sp.npva > n) n = sp.npva;
    if (sp.npob > 0 && sp.npvb > n) n = sp.npvb;
    return n;
}
constexpr size_t kExpOffList = kOffVar;
constexpr size_t kExpOffU = kExpOffList + 256;
constexpr size_t kExpOffW = kExpOffU + kExpUTile * sizeof(ExpU);
inline size_t export_smem_bytes(const SysParams& sp) { return kExpOffW + static_cast<size_t>(exp_max_w(sp)) * (16 + 4); }
constexpr size_t kExpSmemMax = kExpOffW + kPairLut * (16 + 4);  // a spin's 64 orbitals all empty: 2,016 pairs

__device__ __forceinline__ ulonglong2 key_bits(int p, int q) {
    ulonglong2 k = make_ulonglong2(0ULL, 0ULL);
    flip(k, p);
    flip(k, q);
    return k;
}

// One class of doubles over the output positions [lo, hi) of the class (the block's threads).
// ab: an alpha-beta class (u an alpha single, w a beta single), else equal spins (u an occupied
// pair, w an empty pair of spin `spin`).
template <int PREC, int T, bool AB>
__device__ __forceinline__ void export_doubles(const SysParams& sp, const ExportOut& out, ulonglong2 x, ulonglong2 px,
                                               int spin, int n2, int lo, int hi, long long base, unsigned char* smem) {
    const unsigned short* lut = reinterpret_cast<const unsigned short*>(smem + kOffLut);
    const unsigned char* divA = smem + kOffDiv;
    const unsigned char* divB = divA + 1024;
    const unsigned char* wl = smem + kExpOffList;
    const unsigned char* occ = wl + (AB ? 0 : 128 * spin);
    const unsigned char* vir = wl + 64 + (AB ? 0 : 128 * spin);
    ExpU* U = reinterpret_cast<ExpU*>(smem + kExpOffU);
    ulonglong2* WK = reinterpret_cast<ulonglong2*>(smem + kExpOffW);
    unsigned* WI = reinterpret_cast<unsigned*>(WK + exp_max_w(sp));
    const int K = sp.K;
    const unsigned K2 = static_cast<unsigned>(K) * K;
    __syncthreads();  // the previous class's records are read no more
    for (int w = threadIdx.x; w < n2; w += T) {
        int k1, k2;  // w's spatial orbitals: (empty, occupied) beta or the empty pair a < b
        unsigned off, par;
        if (AB) {
            const int jo = divB[w];
            k2 = wl[128 + jo];
            k1 = wl[192 + (w - jo * sp.vb)];
            off = static_cast<unsigned>(k2 * K + k1);  // (ai|jb): kj K + kb
            par = pbit(px, 2 * k2 + 1) ^ pbit(px, 2 * k1 + 1) ^ (k2 < k1 ? 1 : 0);
            WK[w] = key_bits(2 * k2 + 1, 2 * k1 + 1);
        } else {
            const unsigned p = lut[w];
            k1 = vir[p & 255u];
            k2 = vir[p >> 8];
            off = static_cast<unsigned>(k2) * K2 + k1;  // (jb|ia) and (ib|ja): kb K^2 + ka
            par = pbit(px, 2 * k1 + spin) ^ pbit(px, 2 * k2 + spin);
            WK[w] = key_bits(2 * k1 + spin, 2 * k2 + spin);
        }
        WI[w] = static_cast<unsigned>(k1) | (static_cast<unsigned>(k2) << 6) | (par << 12) | (off << 13);
    }
    const int u_end = (hi - 1) / n2 + 1;
    const int sq = T / n2, sr = T - sq * n2;  // a step of the block in (u, w)
    for (int ut = lo / n2; ut < u_end; ut += kExpUTile) {
        const int nu = u_end - ut < kExpUTile ? u_end - ut : kExpUTile;
        if (ut != lo / n2) __syncthreads();
        for (int k = threadIdx.x; k < nu; k += T) {
            const int u = ut + k;
            ExpU r;
            r.key = x;
            int p, q;  // u's spatial orbitals
            unsigned par;
            if (AB) {
                const int io = divA[u];
                p = occ[io];
                q = vir[u - io * sp.va];
                flip(r.key, 2 * p);
                flip(r.key, 2 * q);
                par = pbit(px, 2 * p) ^ pbit(px, 2 * q) ^ (p < q ? 1 : 0);
                // beta orbitals between the alpha orbitals 2p and 2q: spatial min .. max - 1
                const int l = p < q ? p : q, h = p < q ? q : p;
                r.between = (1ULL << h) - (1ULL << l);
                r.d1 = (static_cast<unsigned>(q) * K + p) * K2;
                r.d2 = 0u;
            } else {
                const unsigned pu = lut[u];
                p = occ[pu & 255u];
                q = occ[pu >> 8];
                flip(r.key, 2 * p + spin);
                flip(r.key, 2 * q + spin);
                par = pbit(px, 2 * p + spin) ^ pbit(px, 2 * q + spin) ^ 1;  // [i < j] holds
                r.between = (1ULL << q) - (1ULL << (p + 1));
                r.d1 = static_cast<unsigned>(q) * K2 * K + static_cast<unsigned>(p) * K;  // (jb|ia)
                r.d2 = static_cast<unsigned>(p) * K2 * K + static_cast<unsigned>(q) * K;  // (ib|ja)
            }
            r.d1 |= par << 31;
            U[k] = r;
        }
        __syncthreads();
        const int t_end = hi < (ut + nu) * n2 ? hi : (ut + nu) * n2;
        int t = (lo > ut * n2 ? lo : ut * n2) + static_cast<int>(threadIdx.x);
        int u = t / n2 - ut, w = t - (t / n2) * n2;
        for (; t < t_end; t += T) {
            const ExpU r = U[u];
            const unsigned wi = WI[w];
            if (out.elems) {
                const unsigned off = wi >> 13, d = (r.d1 & 0x7fffffffu) + off;
                const unsigned neg = (r.d1 >> 31) ^ (wi >> 12) ^ static_cast<unsigned>(r.between >> (wi & 63u)) ^
                                     static_cast<unsigned>(r.between >> ((wi >> 6) & 63u));
                double val;
                if (PREC == QC_FP64) {
                    double e = __ldg(sp.eri + QC_IX(d, QC_K4(sp), sp.err));
                    if (!AB) e -= __ldg(sp.eri + QC_IX(r.d2 + off, QC_K4(sp), sp.err));
                    val = with_sign(e, (neg & 1u) != 0u);
                } else {
                    float e = __ldg(sp.eri32 + QC_IX(d, QC_K4(sp), sp.err));
                    if (!AB) e -= __ldg(sp.eri32 + QC_IX(r.d2 + off, QC_K4(sp), sp.err));
                    val = static_cast<double>(with_sign(e, (neg & 1u) != 0u));
                }
                __stcs(out.elems + base + t, val);
            }
            if (out.keys) {
                const ulonglong2 k = WK[w];
                __stcs(out.keys + base + t, make_ulonglong2(r.key.x ^ k.x, r.key.y ^ k.y));
            }
            u += sq;
            w += sr;
            if (w >= n2) {
                w -= n2;
                ++u;
            }
        }
    }
}

// A single's element sums 3 n_elec / 2 integrals: it weighs as much as a quarter as many doubles, and
// items are cut by weight, so that a sample's singles spread over several (N=104, 70 electrons, 12
// samples: 130 us when the first item of a sample held all its singles, 65 us so).
__host__ __device__ inline long long export_single_weight(const SysParams& sp) {
    const long long w = 3LL * (sp.oa + sp.ob) / 8;
    return w > 1 ? w : 1;
}

// Output position of weight v of a sample's weighted order (singles w each, then doubles 1 each).
__host__ __device__ inline long long export_position(const SysParams& sp, long long v) {
    const long long w = export_single_weight(sp), n = sp.nsa + sp.nsb;
    return v < n * w ? (v + w - 1) / w : n + (v - n * w);
}

// Work item (sample s, part c of C): weights [c Q, (c + 1) Q) of the sample's output.
template <int PREC, int T>
__global__ void __launch_bounds__(T, 1280 / T) eloc_export_kernel(const __grid_constant__ SysParams sp,
                                                                  const ulonglong2* __restrict__ samples, long long n_u,
                                                                  const unsigned long long* __restrict__ Tg,
                                                                  const ExportOut out, long long C, long long Q,
                                                                  unsigned long long* __restrict__ cursor) {
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ unsigned long long item;
    __shared__ int valid;
    fill_cta_tables(sp, Tg, smem);
    unsigned char* wl = smem + kExpOffList;
    const unsigned long long* T64 = reinterpret_cast<const unsigned long long*>(smem + kOffT);
    const long long P = sp.pairs;
    const unsigned long long items = static_cast<unsigned long long>(n_u) * C;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    while (true) {
        __syncthreads();  // the tables are there; the previous item's lists are read no more
        if (threadIdx.x < 32) {
            unsigned long long it = 0;
            if (threadIdx.x == 0) it = atomicAdd(cursor, 1ULL);
            it = __shfl_sync(QC_FULLMASK, it, 0);
            if (it < items) {
                const long long s = static_cast<long long>(it / C);
                unsigned long long hx, As, Bs, hxa;
                double ediag = 0.0;
                const bool first = it == static_cast<unsigned long long>(s) * C && out.diag != nullptr;
                const bool ok = sample_setup(sp, samples[s], threadIdx.x, wl, T64, hx, ediag, As, Bs, hxa, first);
                if (threadIdx.x == 0) {
                    if (first) out.diag[s] = ok ? ediag : nan;
                    valid = ok ? 1 : 0;
                }
            }
            if (threadIdx.x == 0) item = it;
        }
        __syncthreads();
        if (item >= items) break;
        const long long s = static_cast<long long>(item / C);
        const long long v0 = (static_cast<long long>(item) - s * C) * Q;
        const long long p0 = export_position(sp, v0), p1 = export_position(sp, v0 + Q) < P ? export_position(sp, v0 + Q) : P;
        const ulonglong2 x = samples[s];
        const long long off = s * P;
        if (!valid) {  // not a determinant of this system: no connected set
            for (long long p = p0 + threadIdx.x; p < p1; p += T) {
                if (out.keys) __stcs(out.keys + off + p, make_ulonglong2(0ULL, 0ULL));
                if (out.elems) __stcs(out.elems + off + p, nan);
            }
            continue;
        }
        const ulonglong2 px = prefix_parity(x);
        // singles: the general path (a small share of the pairs)
        for (long long p = p0 + threadIdx.x; p < p1 && p < sp.nsa + sp.nsb; p += T) {
            const unsigned code = p < sp.nsa ? static_cast<unsigned>(p)
                                             : (1u << 24) | static_cast<unsigned>(p - sp.nsa);
            const unsigned orbs = decode(code, sp, wl, smem, nullptr, nullptr);
            if (out.keys) __stcs(out.keys + off + p, excited_key(orbs, x));
            if (out.elems) {
                double h64 = 0.0;
                float h32 = 0.f;
                bool sneg = false;
                single_element<PREC>(orbs, px, sp, wl, nullptr, h64, h32, sneg);
                __stcs(out.elems + off + p, PREC == QC_FP64 ? h64 : static_cast<double>(h32));
            }
        }
        // doubles, class by class: the item's share of each (a class holds fewer than 2^31 pairs)
        long long c0 = sp.nsa + sp.nsb;
#pragma unroll
        for (int cls = 2; cls < 5; ++cls) {
            const int n2 = cls == 2 ? sp.npva : cls == 3 ? sp.npvb : sp.nsb;
            const long long n = static_cast<long long>(cls == 2 ? sp.npoa : cls == 3 ? sp.npob : sp.nsa) * n2;
            const long long a = p0 > c0 ? p0 - c0 : 0, b = p1 - c0 < n ? p1 - c0 : n;
            if (a < b) {
                if (cls == 4)
                    export_doubles<PREC, T, true>(sp, out, x, px, 0, n2, static_cast<int>(a), static_cast<int>(b),
                                               off + c0, smem);
                else
                    export_doubles<PREC, T, false>(sp, out, x, px, cls - 2, n2, static_cast<int>(a),
                                                static_cast<int>(b), off + c0, smem);
            }
            c0 += n;
        }
    }
}

// E_loc of one sample from its sum of products, and the reports of a sample that has none.
__device__ __forceinline__ void apply_finish(double re, double im, double2 p, double d, double2* __restrict__ eloc,
                                             Counters* __restrict__ ctr) {
    const double n2 = p.x * p.x + p.y * p.y;
    double2 out;
    if (n2 == 0.0 || !isfinite(d)) {
        out.x = out.y = __longlong_as_double(0x7ff8000000000000LL);
        atomicAdd(&ctr->bad, 1ULL);
        if (n2 == 0.0) atomicOr(&ctr->flags, QC_FLAG_ZERO_PSI);
        else {
            atomicAdd(&ctr->invalid, 1ULL);
            atomicOr(&ctr->flags, QC_FLAG_NELEC);
        }
    } else {
        const double inv = 1.0 / n2;
        out.x = d + (re * p.x + im * p.y) * inv;
        out.y = (im * p.x - re * p.y) * inv;
    }
    *eloc = out;
}

// One lane's share of the products elems[j] psi[j], j = j0, j0 + step, ... < j1: kAppUnroll
// independent partial sums (their loads in flight together), added in a fixed order.
constexpr int kAppUnroll = 4;
__device__ __forceinline__ double2 apply_products(const double* __restrict__ e, const double2* __restrict__ q,
                                                  long long j0, long long j1, long long step) {
    double re[kAppUnroll], im[kAppUnroll];
#pragma unroll
    for (int k = 0; k < kAppUnroll; ++k) re[k] = im[k] = 0.0;
    long long j = j0;
    for (; j + (kAppUnroll - 1) * step < j1; j += kAppUnroll * step) {
        double h[kAppUnroll];
        double2 v[kAppUnroll];
#pragma unroll
        for (int k = 0; k < kAppUnroll; ++k) {
            h[k] = __ldcs(e + j + k * step);
            v[k] = __ldcs(q + j + k * step);
        }
#pragma unroll
        for (int k = 0; k < kAppUnroll; ++k) {
            re[k] = fma(h[k], v[k].x, re[k]);
            im[k] = fma(h[k], v[k].y, im[k]);
        }
    }
    for (; j < j1; j += step) {
        const double h = __ldcs(e + j);
        const double2 v = __ldcs(q + j);
        re[0] = fma(h, v.x, re[0]);
        im[0] = fma(h, v.y, im[0]);
    }
    return make_double2((re[0] + re[1]) + (re[2] + re[3]), (im[0] + im[1]) + (im[2] + im[3]));
}

// Many samples or short connected sets: one warp per sample.  The P products are summed
// lane-wise in FP64 (fixed lanes, fixed shuffle tree: deterministic).
__global__ void __launch_bounds__(256) eloc_apply_kernel(const double* __restrict__ elems,
                                                         const double* __restrict__ diag,
                                                         const double2* __restrict__ psi_conn,
                                                         const double2* __restrict__ psi, long long n_u,
                                                         long long P, double2* __restrict__ eloc,
                                                         Counters* __restrict__ ctr) {
    const int lane = threadIdx.x & 31;
    const long long warps = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
    for (long long s = static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); s < n_u;
         s += warps) {
        const double2 t = apply_products(elems + s * P, psi_conn + s * P, lane, P, 32);
        const double re = warp_sum(t.x), im = warp_sum(t.y);
        if (lane == 0) apply_finish(re, im, psi[s], diag[s], eloc + s, ctr);
    }
}

// Long connected sets: 128 threads, or a cluster of R CTAs of 512, per sample.  The stream is
// bound by HBM and, a close second, by the FP64 pipe (24 B and two fused multiply-adds per
// pair), so what matters is that every SM has loads in flight whatever the number of samples:
// a chunk of a large molecule is a few hundred samples of 10^6 pairs, and a warp per sample
// left all but 200 warps of the chip idle (N=120, 200 samples, 5.7 GB: 11.1 ms; now 0.98 ms,
// 5.9 TB/s).  Each CTA sums a contiguous share of the sample's pairs; the CTA sums are read
// over distributed shared memory by the first CTA in rank order, so the result is
// deterministic and needs no workspace.
template <int T>
__global__ void __launch_bounds__(T) eloc_apply_wide_kernel(const double* __restrict__ elems,
                                                            const double* __restrict__ diag,
                                                            const double2* __restrict__ psi_conn,
                                                            const double2* __restrict__ psi, long long P,
                                                            double2* __restrict__ eloc, Counters* __restrict__ ctr) {
    __shared__ double2 warp_part[T / 32];
    __shared__ double2 cta_part;
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const unsigned R = cl.num_blocks(), r = cl.block_rank();
    const long long s = blockIdx.x / R;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double2 t = apply_products(elems + s * P, psi_conn + s * P, P * r / R + threadIdx.x, P * (r + 1) / R, T);
    const double re = warp_sum(t.x), im = warp_sum(t.y);
    if (lane == 0) warp_part[warp] = make_double2(re, im);
    __syncthreads();
    double sr = 0.0, si = 0.0;
    if (warp == 0) {
        const double2 v = lane < T / 32 ? warp_part[lane] : make_double2(0.0, 0.0);
        sr = warp_sum(v.x);
        si = warp_sum(v.y);
        if (R > 1 && lane == 0) cta_part = make_double2(sr, si);
    }
    if (R > 1) {
        cl.sync();
        if (r == 0 && threadIdx.x == 0) {
            for (unsigned k = 1; k < R; ++k) {
                const double2 v = *cl.map_shared_rank(&cta_part, k);
                sr += v.x;
                si += v.y;
            }
        }
        cl.sync();  // the other CTAs' sums stay in place until the first CTA has read them
    }
    if (r == 0 && threadIdx.x == 0) apply_finish(sr, si, psi[s], diag[s], eloc + s, ctr);
}

// Threads per sample: two full waves of the chip's threads over the samples; 32 (a warp), 128, or
// R x 512 with R up to the portable cluster size.  With many samples a CTA's fixed cost (block
// sum, launch) pays only for long sums (10,000 samples, P = 2,220: 140 us with a warp, 167 us with
// 128 threads; P = 5,040: 277 against 311 us; P = 7,875: 381 against 361; P = 25,137: 1,102 against 983);
// with few, idle SMs cost more (300 samples, P = 25,137: 270 us with a warp, 106 us).
int apply_threads(long long n_u, long long P, int sm_count) {
    const long long cap = n_u >= 8LL * sm_count ? P / 160 : P / 8;
    const long long want = std::min(2LL * 2048 * sm_count / n_u, cap);
    if (want <= 48) return 32;
    if (want < 256 || (want < 512 && P < 32768)) return 128;
    int t = 512;
    while (t < 8 * 512 && want >= 2 * t) t *= 2;
    return t;
}

template <int T>
cudaError_t launch_apply_wide(const double* elems, const double* diag, const double2* conn, const double2* psi,
                              long long n_u, long long P, double2* eloc, Counters* ctr, int R, cudaStream_t s) {
    // a grid holds fewer than 2^31 blocks: longer chunks go out in several launches
    const long long most = 0x7fffffffLL / R;
    cudaError_t e = cudaSuccess;
    for (long long lo = 0; lo < n_u && e == cudaSuccess; lo += most) {
        const long long n = std::min(most, n_u - lo);
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(static_cast<unsigned>(n * R));
        cfg.blockDim = dim3(T);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = static_cast<unsigned>(R);
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, eloc_apply_wide_kernel<T>, elems + lo * P, diag + lo, conn + lo * P, psi + lo, P,
                               eloc + lo, ctr);
    }
    return e;
}

qc_status ffail(qc_eloc* H, qc_status st, const std::string& m) {
    H->err = m;
    return st;
}

}  // namespace

// The export kernels' shared-memory limit belongs to the function, not to a launch: it is set once,
// to the most any handle needs (set per call to the handle's own size, threads exporting with
// different handles lowered it between each other's call and launch).
cudaError_t prepare_export() {
    cudaError_t e = cudaSuccess;
    for (const void* f : {(const void*)eloc_export_kernel<QC_FP64, 128>, (const void*)eloc_export_kernel<QC_FP32_COMP, 128>,
                          (const void*)eloc_export_kernel<QC_FP64, 256>, (const void*)eloc_export_kernel<QC_FP32_COMP, 256>}) {
        const cudaError_t r =
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kExpSmemMax));
        if (r != cudaSuccess) e = r;
    }
    return e;
}

}  // namespace qc

extern "C" qc_status qc_eloc_export(qc_eloc* H, const uint64_t* samples, int64_t n_u, uint64_t* keys_out,
                                    double* elems_out, double* diag_out, void* stream) {
    if (!H) return QC_ERR_ARG;
    if (n_u < 0) return qc::ffail(H, QC_ERR_ARG, "negative n_u");
    if (n_u > 0 && !samples) return qc::ffail(H, QC_ERR_ARG, "samples is NULL");
    auto mis = [](const void* p, unsigned a) { return p && (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0; };
    if (mis(samples, 16) || mis(keys_out, 16) || mis(elems_out, 8) || mis(diag_out, 8))
        return qc::ffail(H, QC_ERR_ARG, "alignment: samples and keys 16 bytes, elements and diagonal 8");
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != H->device) return qc::ffail(H, QC_ERR_ARG, "handle belongs to another device");
    if (n_u == 0 || (!keys_out && !elems_out && !diag_out)) return QC_OK;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    qc::ExportOut out{reinterpret_cast<ulonglong2*>(keys_out), elems_out, diag_out};
    const size_t smem = qc::export_smem_bytes(H->sp);
    using Kernel = void (*)(qc::SysParams, const ulonglong2*, long long, const unsigned long long*, qc::ExportOut,
                            long long, long long, unsigned long long*);
    const bool f64 = H->precision == QC_FP64;
    // an item's fixed part (cursor, occupation lists, records) costs a small CTA less: 128 threads
    // for short connected sets (P = 2,220, 20,000 samples: 437 us with 256, 328 with 128; P = 609: 108
    // and 79; P = 25,137: 1,029 and 1,118)
    const int T = H->sp.pairs < 8192 ? 128 : 256;
    const Kernel f = T == 128 ? (f64 ? qc::eloc_export_kernel<QC_FP64, 128> : qc::eloc_export_kernel<QC_FP32_COMP, 128>)
                              : (f64 ? qc::eloc_export_kernel<QC_FP64, 256> : qc::eloc_export_kernel<QC_FP32_COMP, 256>);
    int per_sm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, T, smem);
    if (e != cudaSuccess || per_sm < 1)
        return qc::ffail(H, QC_ERR_CUDA, std::string("export: ") + cudaGetErrorString(e));
    // pairs per work item: about kExpItemPairs, fewer when that leaves the chip's CTAs short of work
    const long long resident = static_cast<long long>(per_sm) * H->sm_count;
    const long long V = H->sp.pairs + (qc::export_single_weight(H->sp) - 1) * (H->sp.nsa + H->sp.nsb);
    long long C = std::max<long long>(1, (V + qc::kExpItemPairs / 2) / qc::kExpItemPairs);
    while (n_u * C < 2 * resident && V / (2 * C) >= 1024) C *= 2;
    const long long Q = (V + C - 1) / C;
    const long long blocks = std::min<long long>(n_u * C, resident);
    unsigned long long* cursor = &H->d_ctr->next;  // the handle's counters are free between evaluations
    e = cudaMemsetAsync(cursor, 0, sizeof(unsigned long long), s);
    if (e != cudaSuccess) return qc::ffail(H, QC_ERR_CUDA, std::string("export: ") + cudaGetErrorString(e));
    const ulonglong2* sk = reinterpret_cast<const ulonglong2*>(samples);
    const unsigned grid = static_cast<unsigned>(blocks);
    f<<<grid, T, smem, s>>>(H->sp, sk, n_u, H->d_T, out, C, Q, cursor);
    e = cudaGetLastError();
    if (e != cudaSuccess) return qc::ffail(H, QC_ERR_CUDA, std::string("export launch: ") + cudaGetErrorString(e));
    return QC_OK;
}

extern "C" qc_status qc_eloc_apply(qc_eloc* H, const double* psi, const int64_t* counts, int64_t n_u,
                                   const double* elems, const double* diag, const double* psi_conn,
                                   double* eloc_out, qc_eloc_summary* summary, void* stream) {
    if (!H) return QC_ERR_ARG;
    if (n_u < 0) return qc::ffail(H, QC_ERR_ARG, "negative n_u");
    if (n_u > 0 && (!psi || !counts || !elems || !diag || !psi_conn || !eloc_out))
        return qc::ffail(H, QC_ERR_ARG, "NULL pointer");
    auto mis = [](const void* p, unsigned a) { return p && (reinterpret_cast<uintptr_t>(p) & (a - 1)) != 0; };
    if (mis(psi, 16) || mis(psi_conn, 16) || mis(eloc_out, 16) || mis(elems, 8) || mis(diag, 8) || mis(counts, 8))
        return qc::ffail(H, QC_ERR_ARG, "alignment: complex arrays 16 bytes, the others 8");
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev != H->device) return qc::ffail(H, QC_ERR_ARG, "handle belongs to another device");
    qc_status st = qc::ensure_workspace(H, std::max<int64_t>(n_u, 1), 1, 0);
    if (st != QC_OK) return st;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e = cudaMemsetAsync(H->d_ctr, 0, sizeof(qc::Counters), s);
    if (e == cudaSuccess && n_u > 0) {
        const double2* conn = reinterpret_cast<const double2*>(psi_conn);
        const double2* p2 = reinterpret_cast<const double2*>(psi);
        double2* el = reinterpret_cast<double2*>(eloc_out);
        const int t = qc::apply_threads(n_u, H->sp.pairs, H->sm_count);
        if (t >= 512) {
            e = qc::launch_apply_wide<512>(elems, diag, conn, p2, n_u, H->sp.pairs, el, H->d_ctr, t / 512, s);
        } else if (t == 128) {
            e = qc::launch_apply_wide<128>(elems, diag, conn, p2, n_u, H->sp.pairs, el, H->d_ctr, 1, s);
        } else {
            const long long blocks = std::min<long long>((n_u + 7) / 8, static_cast<long long>(H->sm_count) * 16);
            qc::eloc_apply_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(elems, diag, conn, p2, n_u,
                                                                              H->sp.pairs, el, H->d_ctr);
            e = cudaGetLastError();
        }
    }
    if (e == cudaSuccess) {
        qc::EvalParams ep{};
        ep.psi = reinterpret_cast<const double2*>(psi);
        ep.counts = reinterpret_cast<const long long*>(counts);
        ep.n_u = n_u;
        ep.eloc = reinterpret_cast<double2*>(eloc_out);
        ep.ctr = H->d_ctr;
        ep.T = H->d_T;
        ep.mode = QC_FULL;
        e = qc::launch_reduce(ep, H->d_part, qc::reduce_blocks(n_u), H->d_sum, H->sp.pairs, s);
    }
    if (e == cudaSuccess && summary)
        e = cudaMemcpyAsync(summary, H->d_sum, sizeof(qc_eloc_summary), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) return qc::ffail(H, QC_ERR_CUDA, std::string("apply: ") + cudaGetErrorString(e));
    return QC_OK;
}
