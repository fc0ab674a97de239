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
        if (out.keys == nullptr && out.elems == nullptr) continue;  // the diagonal alone
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

// The sum of one sample's P products elems[j] psi[j] has one order, given by P alone, so a sample's
// E_loc has the same bits whatever else its call holds.  Runs of `run` products are dealt to
// `blocks` blocks in turn; a block is summed by 128 accumulators (accumulator a takes products a,
// a + 128, .. of each of its runs, one after another) or, in long blocks, twice as many (added in
// pairs a, a + 128); then, for each accumulator, the blocks are added by fours and the fours one after
// another; then the accumulators by a fixed tree.  Accumulators and blocks go to lanes, warps or
// CTAs as the call's size asks.  (A split by the threads at hand gave a chunk's last samples other
// bits than the whole call's.)
constexpr int kAppAcc = 128, kAppBlocks = 32, kAppFour = 4;
struct AppOrder {
    int P, run, blocks;
    bool pairs;
};
// One block up to 8,192 products (a warp's or 128 threads' work); beyond, one per run of 2,048 (a block
// more is two FP64 additions an accumulator, against 32 for its products) until they are as many as
// a cluster has groups of 128 threads.  From 64 products an accumulator on, a thread's four products
// in flight go to two accumulators, half as long a chain of additions: N=120, 200 samples 1,019 ->
// 994 us.
AppOrder apply_order(long long P) {
    const int run = P <= 8192 ? 8192 : 2048;
    const long long n = std::max<long long>(1, (P + run - 1) / run);
    return AppOrder{static_cast<int>(P), run, static_cast<int>(std::min<long long>(n, kAppBlocks)),
                    P >= 64LL * kAppBlocks * kAppAcc};
}

// Adds v to a sum, or begins it.
__device__ __forceinline__ void add_to(double2& sum, double2 v, bool first) {
    sum.x = first ? v.x : sum.x + v.x;
    sum.y = first ? v.y : sum.y + v.y;
}

// Products j, j + step, .. below end, U loads in flight, to ACC accumulators in turn.  APART: the last
// few by code of their own, so that the loop needs no predicates and fewer registers.
template <int ACC, int U, int UNROLL, bool APART>
__device__ __forceinline__ void add_products(const double* __restrict__ e, const double2* __restrict__ q, int j,
                                             int step, int end, double2 (&v)[ACC]) {
    double h[U];
    double2 w[U];
#pragma unroll UNROLL
    for (; j + (APART ? (U - 1) * step : 0) < end; j += U * step) {
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (APART || j + k * step < end) {
                h[k] = __ldcs(e + j + k * step);
                w[k] = __ldcs(q + j + k * step);
            }
#pragma unroll
        for (int k = 0; k < U; ++k)
            if (APART || j + k * step < end) {
                v[k % ACC].x = fma(h[k], w[k].x, v[k % ACC].x);
                v[k % ACC].y = fma(h[k], w[k].y, v[k % ACC].y);
            }
    }
    if (APART && j < end) {
#pragma unroll
        for (int k = 0; k < U - 1; ++k)
            if (j + k * step < end) {
                h[k] = __ldcs(e + j + k * step);
                w[k] = __ldcs(q + j + k * step);
            }
#pragma unroll
        for (int k = 0; k < U - 1; ++k)
            if (j + k * step < end) {
                v[k % ACC].x = fma(h[k], w[k].x, v[k % ACC].x);
                v[k % ACC].y = fma(h[k], w[k].y, v[k % ACC].y);
            }
    }
}

// The sum of 128 accumulators, four to a lane.
__device__ __forceinline__ double2 add_accumulators(double2 a, double2 b, double2 c, double2 d) {
    return make_double2(warp_sum((a.x + b.x) + (c.x + d.x)), warp_sum((a.y + b.y) + (c.y + d.y)));
}

// Many samples of one block: one warp per sample, a lane four accumulators.  A warp takes `run`
// consecutive samples and finishes them together, a lane each: one at a time their divisions kept the
// FP64 pipe (16 cycles an instruction of a warp, however few its lanes) longer than P = 204 products
// do (300,000 samples 836 -> 630 us).  APART, with five CTAs an SM, from 1,024 products on (P = 2,220,
// 20,000 samples 232 us, 258 without; P = 609 138, 119 without).
template <bool APART>
__global__ void __launch_bounds__(256, APART ? 5 : 4) eloc_apply_kernel(const double* __restrict__ elems,
                                                                        const double* __restrict__ diag,
                                                                        const double2* __restrict__ psi_conn,
                                                                        const double2* __restrict__ psi,
                                                                        long long n_u, int run, int P,
                                                                        double2* __restrict__ eloc,
                                                                        Counters* __restrict__ ctr) {
    constexpr int U = kAppAcc / 32;
    const int lane = threadIdx.x & 31;
    const long long warps = static_cast<long long>(gridDim.x) * (blockDim.x >> 5);
    for (long long s0 = (static_cast<long long>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5)) * run; s0 < n_u;
         s0 += warps * run) {
        const int m = n_u - s0 < run ? static_cast<int>(n_u - s0) : run;
        double2 mine = make_double2(0.0, 0.0);
        for (int i = 0; i < m; ++i) {
            double2 v[U];
#pragma unroll
            for (int k = 0; k < U; ++k) v[k] = make_double2(0.0, 0.0);
            add_products<U, 4, APART ? 1 : 2, APART>(elems + (s0 + i) * P, psi_conn + (s0 + i) * P, lane, 32, P, v);
            const double2 t = add_accumulators(v[0], v[1], v[2], v[3]);
            if (lane == i) mine = t;
        }
        if (lane < m) apply_finish(mine.x, mine.y, psi[s0 + lane], diag[s0 + lane], eloc + s0 + lane, ctr);
    }
}

// Accumulator a's sum of block b (ACC = 2: accumulators a's and a + 128's).
template <int ACC, int U, int UNROLL>
__device__ __forceinline__ double2 block_products(const double* __restrict__ e, const double2* __restrict__ q,
                                                  const AppOrder& o, int b, int a) {
    double2 v[ACC];
#pragma unroll
    for (int k = 0; k < ACC; ++k) v[k] = make_double2(0.0, 0.0);
    for (int c = b * o.run; c < o.P; c += o.blocks * o.run)
        add_products<ACC, U, UNROLL, true>(e, q, c + a, kAppAcc, min(c + o.run, o.P), v);
    if (ACC == 2) add_to(v[0], v[ACC - 1], false);
    return v[0];
}

// Long connected sets: a thread one accumulator (PAIRS: two), 128 threads (G = 1), or a cluster of R
// CTAs of four times 128 (G = 4), per sample.  The stream is bound by HBM and, a close second, by the
// FP64 pipe (24 B and two fused multiply-adds per pair), so what matters is that every SM has loads
// in flight whatever the number of samples: a chunk of a large molecule is a few hundred samples of
// 10^6 pairs, and a warp per sample left all but 200 warps of the chip idle (N=120, 200 samples,
// 5.7 GB: 11.1 ms; now 0.95 ms, 6.0 TB/s).  With G = 4 a CTA's groups take the four blocks of a four; the
// fours' sums stay in shared memory and the first CTA adds all of the sample's in order, over
// distributed shared memory.  No workspace.  G = 1 has eight CTAs an SM with eight loads a thread in
// flight, or ten with four (kept for calls of several waves: P = 11,340, 20,000 samples 908 us, 931
// with eight loads; 40 samples of 5,040 41 and 35 us).
template <int G, bool PAIRS, int PER_SM>
__global__ void __launch_bounds__(kAppAcc * G, PER_SM) eloc_apply_wide_kernel(const double* __restrict__ elems,
                                                                      const double* __restrict__ diag,
                                                                      const double2* __restrict__ psi_conn,
                                                                      const double2* __restrict__ psi,
                                                                      const AppOrder o, double2* __restrict__ eloc,
                                                                      Counters* __restrict__ ctr) {
    static_assert(G == kAppFour || (G == 1 && !PAIRS), "a CTA takes whole fours of blocks");
    constexpr int kFours = kAppBlocks / kAppFour;
    __shared__ double2 acc[kAppAcc];
    __shared__ double2 part[G > 1 ? 2 : 1][G][kAppAcc], fours[G > 1 ? kFours : 1][kAppAcc];
    cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int R = static_cast<int>(cl.num_blocks()), r = static_cast<int>(cl.block_rank());
    const long long s = blockIdx.x / R;
    const double* e = elems + s * o.P;
    const double2* q = psi_conn + s * o.P;
    const int a = threadIdx.x % kAppAcc, g = threadIdx.x / kAppAcc;
    double2 total = make_double2(0.0, 0.0);
    if (G == 1) {
        double2 four = total;
        for (int b = 0; b < o.blocks; ++b) {
            add_to(four, block_products<1, PER_SM == 8 ? 8 : 4, PER_SM == 8 ? 1 : 2>(e, q, o, b, a), b % kAppFour == 0);
            if (b % kAppFour == kAppFour - 1 || b == o.blocks - 1) add_to(total, four, b < kAppFour);
        }
    } else {
        const int n = (o.blocks + kAppFour - 1) / kAppFour, own = (n + R - 1) / R;  // fours, and of one CTA
        for (int f = r * own; f < (r + 1) * own && f < n; ++f) {
            if (f * kAppFour + g < o.blocks) part[f & 1][g][a] = block_products<PAIRS ? 2 : 1, 4, 1>(e, q, o, f * kAppFour + g, a);
            __syncthreads();  // (the other half of part is read before the next one)
            if (g == 0) {
                double2 four = part[f & 1][0][a];
#pragma unroll
                for (int k = 1; k < kAppFour; ++k)
                    if (f * kAppFour + k < o.blocks) add_to(four, part[f & 1][k][a], false);
                fours[f - r * own][a] = four;
            }
        }
        if (R > 1) cl.sync();
        if (r == 0 && g == 0)
            for (int f = 0; f < n; ++f) {
                const double2 v = R > 1 ? cl.map_shared_rank(&fours[0][0], f / own)[f % own * kAppAcc + a] : fours[f][a];
                add_to(total, v, f == 0);
            }
        if (R > 1) cl.sync();  // the other CTAs' sums stay in place until the first CTA has read them
    }
    if (r != 0) return;
    if (g == 0) acc[a] = total;
    __syncthreads();
    if (threadIdx.x < 32) {
        const double2 t = add_accumulators(acc[a], acc[a + 32], acc[a + 64], acc[a + 96]);
        if (a == 0) apply_finish(t.x, t.y, psi[s], diag[s], eloc + s, ctr);
    }
}

// Threads per sample: 32 (a warp), 128, or R x 512 with R up to the portable cluster size and the fours
// of blocks.  One block: 128 while they are resident together, then a warp (P = 2,220, 1,300 samples
// 48 us against 54, 10,000 148 against 139; from 6,144 products 128 always: P = 7,875, 5,000 samples 201
// against 224).  Above 16,384 products 512 R by how the samples fill waves of three CTAs an SM: few
// take the whole cluster, up to three an SM one CTA each (300 samples: P = 25,137 65 us, 79 with R = 4;
// 599,360 682, 730 with R = 8), then 128 threads or R = 4, whose waves are finer (500 samples: P = 25,137
// 96 us, 109 with R = 1; 294,750 629, 816 with R = 1), and many again one CTA each (P = 25,137, 10,000
// samples 990 us, 1,040 with 128 threads).
int apply_threads(long long n_u, const AppOrder& o, int sm_count) {
    const long long sm = sm_count;
    if (o.blocks == 1) return n_u <= 9 * sm || o.P >= 6144 ? 128 : 32;
    if (o.P <= 16384 && n_u > 2 * sm) return 128;
    int R;
    if (o.P < 65536)
        R = n_u <= sm * 4 / 5 ? 4 : n_u <= 3 * sm || n_u > 8 * sm ? 1 : 0;
    else
        R = n_u <= sm * 8 / 5 ? 8 : n_u <= 3 * sm || n_u > 8 * sm ? 1 : 4;
    if (R == 0) return 128;
    const int fours = (o.blocks + kAppFour - 1) / kAppFour;
    while (R > fours) R /= 2;
    return 512 * R;
}

template <int G, bool PAIRS, int PER_SM>
cudaError_t launch_apply_wide(const double* elems, const double* diag, const double2* conn, const double2* psi,
                              long long n_u, const AppOrder& o, double2* eloc, Counters* ctr, int R, cudaStream_t s) {
    // a grid holds fewer than 2^31 blocks: longer chunks go out in several launches
    const long long most = 0x7fffffffLL / R;
    cudaError_t e = cudaSuccess;
    for (long long lo = 0; lo < n_u && e == cudaSuccess; lo += most) {
        const long long n = std::min(most, n_u - lo);
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(static_cast<unsigned>(n * R));
        cfg.blockDim = dim3(kAppAcc * G);
        cfg.stream = s;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = static_cast<unsigned>(R);
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, eloc_apply_wide_kernel<G, PAIRS, PER_SM>, elems + lo * o.P, diag + lo, conn + lo * o.P, psi + lo, o,
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
    if (!keys_out && !elems_out) C = 1;  // the diagonal alone (N=40, 10 electrons, 20,000 samples:
                                         // 193 us when every pair was walked for it, 48)
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
        const qc::AppOrder o = qc::apply_order(H->sp.pairs);
        const int t = qc::apply_threads(n_u, o, H->sm_count);
        if (t >= 512) {
            // two CTAs an SM with pairs (N=120, 200 samples 992 us, 1,043 with three) but where three
            // hold every CTA at once (40 samples 309, 346 with two), and three without pairs but where
            // two fill their second wave better
            const long long ctas = n_u * (t / 512), sm = H->sm_count;
            const auto f = o.pairs ? ctas > 2 * sm && ctas <= 3 * sm ? qc::launch_apply_wide<4, true, 3>
                                                                     : qc::launch_apply_wide<4, true, 2>
                           : ctas > 3 * sm && ctas <= 4 * sm ? qc::launch_apply_wide<4, false, 2>
                                                             : qc::launch_apply_wide<4, false, 3>;
            e = f(elems, diag, conn, p2, n_u, o, el, H->d_ctr, t / 512, s);
        } else if (t == 128) {
            const auto f = n_u <= 5LL * H->sm_count ? qc::launch_apply_wide<1, false, 8> : qc::launch_apply_wide<1, false, 10>;
            e = f(elems, diag, conn, p2, n_u, o, el, H->d_ctr, 1, s);
        } else {
            const long long warps = std::min<long long>(n_u, static_cast<long long>(H->sm_count) * 128);
            const int run = static_cast<int>(std::min<long long>(32, (n_u + warps - 1) / warps));
            const auto f = o.P < 1024 ? qc::eloc_apply_kernel<false> : qc::eloc_apply_kernel<true>;
            f<<<static_cast<unsigned>((warps + 7) / 8), 256, 0, s>>>(elems, diag, conn, p2, n_u, run, o.P, el, H->d_ctr);
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
