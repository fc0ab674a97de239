// qc_kernels.cu -- the single-molecule kernels of libqc_eloc (sm_103a) and their launchers:
// K0 table build, K2 local-energy kernel (filtered and unfiltered; the template is in
// qc_main_kernel.cuh, its diagnostic instantiations in qc_kernels_diag.cu), K3 reduction.  The
// device code they share with the batch kernels is in qc_device.cuh.
#include <cstdint>
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "qc_main_kernel.cuh"

namespace qc {

namespace cg = cooperative_groups;

int reduce_blocks(long long n) {
    // two rows per thread: enough blocks that every SM has a few (latency-bound loads)
    long long b = (n + kRedThreads * 2 - 1) / (kRedThreads * 2);
    if (b < 1) b = 1;
    if (b > 1024) b = 1024;
    return static_cast<int>(b);
}

size_t smem_fixed_bytes() { return kOffVar; }

size_t filtered_smem_bytes(const SysParams& sp, int warps, int fw, bool lean, bool join, int acap) {
    return kOffVar + (static_cast<size_t>(4) << fw) +
           static_cast<size_t>(warps) * main_warp_bytes(sp, true, lean, join, join ? acap : 0);
}
size_t direct_smem_bytes(const SysParams& sp, int warps) {
    return kOffVar + static_cast<size_t>(warps) * main_warp_bytes(sp, false);
}

__global__ void __launch_bounds__(256) build_table_kernel(TableParams tp, int n_orb, int na, int nb,
                                                          const unsigned long long* __restrict__ T,
                                                          unsigned long long* slots,
                                                          uint32_t* filter, unsigned long long* aset,
                                                          unsigned long long* bset, Counters* ctr,
                                                          unsigned* jkey, unsigned* jlen) {
    let_next_start();
    wait_previous();
    const long long r = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (r < tp.n) build_one(tp, n_orb, na, nb, T, slots, filter, aset, bset, ctr, r, jkey, jlen, 0u,
                            2u * (tp.set_mask + 1u));
}

__global__ void __launch_bounds__(kRedThreads) reduce_pass1(EvalParams ep, double* part) {
    let_next_start();
    wait_previous();
    reduce_pass1_body(ep, part, blockIdx.x, gridDim.x, 0, ep.n_u);
}
__global__ void __launch_bounds__(kRedThreads) reduce_pass2(EvalParams ep, double* part,
                                                            qc_eloc_summary* out, long long pairs_per_sample) {
    wait_previous();
    reduce_pass2_body(ep, part, out, pairs_per_sample, blockIdx.x, gridDim.x, 0, ep.n_u);
}

// Both passes of a small sample set in one launch: a cluster of CTAs keeps its rows in registers
// and exchanges its sums through distributed shared memory.  Each CTA stands for two blocks of the
// grid-wide passes and every sum is added in their order, so the summary has the same bits
// as theirs (a batch reduces its molecules by the passes).  Up to kRedSmallRows rows, two a thread;
// above, the few SMs' FP64 rate (some ten operations a row at two per clock and SM) costs more
// than the second launch.
constexpr int kRedCluster = 8, kRedVirtual = 2;
constexpr long long kRedSmallRows = static_cast<long long>(kRedCluster) * kRedVirtual * kRedThreads * 2;

__global__ void __cluster_dims__(kRedCluster, 1, 1) __launch_bounds__(kRedThreads)
    reduce_small_kernel(EvalParams ep, qc_eloc_summary* out, long long pairs_per_sample, int nblk) {
    __shared__ RedSums sh[kRedWarps];
    __shared__ double shd[kRedWarps];
    __shared__ RedSums mine[kRedVirtual], total;
    __shared__ double mine_var[kRedVirtual];
    cg::cluster_group cl = cg::this_cluster();
    wait_previous();
    const int lane = threadIdx.x & 31;
    double2 e[kRedVirtual][2];
    long long c[kRedVirtual][2];
#pragma unroll
    for (int b = 0; b < kRedVirtual; ++b)
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const int vb = b * kRedCluster + static_cast<int>(blockIdx.x);
            const long long i = static_cast<long long>(vb + k * nblk) * kRedThreads + threadIdx.x;
            const bool in = vb < nblk && i < ep.n_u;
            // a row past the end is left out like one of a NaN energy
            e[b][k] = in ? ep.eloc[i] : make_double2(__longlong_as_double(0x7ff8000000000000LL), 0.0);
            c[b][k] = in ? ep.counts[i] : 0;
        }
    bool neg = false;
#pragma unroll
    for (int b = 0; b < kRedVirtual; ++b) {
        RedSums v{};
        red_row(e[b][0], c[b][0], v, neg);
        red_row(e[b][1], c[b][1], v, neg);
        v = block_sums(v, sh);
        if (threadIdx.x == 0) mine[b] = v;
    }
    if (neg) {
        atomicOr(&ep.ctr->flags, QC_FLAG_NEG_COUNT);
        __threadfence();  // for the CTA that writes the summary
    }
    cl.sync();
    if (threadIdx.x < 32) {
        RedSums t{};
        if (lane < nblk) t = cl.map_shared_rank(mine, lane % kRedCluster)[lane / kRedCluster];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            red_add(t, RedSums{__shfl_down_sync(QC_FULLMASK, t.re, o), __shfl_down_sync(QC_FULLMASK, t.im, o),
                               __shfl_down_sync(QC_FULLMASK, t.w, o), __shfl_down_sync(QC_FULLMASK, t.used, o)});
        red_add(t, RedSums{});
        if (lane == 0) total = t;
    }
    __syncthreads();
    const double mr = total.re / static_cast<double>(total.w), mi = total.im / static_cast<double>(total.w);
#pragma unroll
    for (int b = 0; b < kRedVirtual; ++b) {
        double q = red_row_var(e[b][0], c[b][0], mr, mi, 0.0);
        q = block_sum(red_row_var(e[b][1], c[b][1], mr, mi, q), shd);
        if (threadIdx.x == 0) mine_var[b] = q;
    }
    cl.sync();
    if (blockIdx.x == 0 && threadIdx.x < 32) {
        double tv = lane < nblk ? cl.map_shared_rank(mine_var, lane % kRedCluster)[lane / kRedCluster] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) tv += __shfl_down_sync(QC_FULLMASK, tv, o);
        if (lane == 0) {
            write_means(ep.ctr, total);
            write_summary(ep.ctr, out, tv, ep.n_u, pairs_per_sample);
        }
    }
    cl.sync();  // no CTA leaves while its sums are read
}

// Zeroes up to ClearList::kMax ranges (the tables and counters an evaluation starts from): one
// launch in the place of four to six memsets.
__global__ void __launch_bounds__(256) clear_kernel(const __grid_constant__ ClearList list) {
    let_next_start();
    const size_t step = static_cast<size_t>(gridDim.x) * blockDim.x;
    for (int k = 0; k < list.n; ++k) {
        uint4* p = static_cast<uint4*>(list.p[k]);
        for (size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < list.bytes[k] / 16; i += step)
            p[i] = make_uint4(0u, 0u, 0u, 0u);
    }
}

// ------------------------------------------------------------------------------------
// host launchers
// ------------------------------------------------------------------------------------
cudaError_t launch_clear(const ClearList& list, int sm_count, cudaStream_t s) {
    size_t most = 0;
    for (int k = 0; k < list.n; ++k) most = list.bytes[k] > most ? list.bytes[k] : most;
    // up to two 16-byte stores a thread and range, at most eight CTAs an SM
    const size_t cap = static_cast<size_t>(sm_count) * 8;
    size_t blocks = (most / 16 + 511) / 512;
    blocks = blocks < 1 ? 1 : blocks > cap ? cap : blocks;
    clear_kernel<<<static_cast<unsigned>(blocks), 256, 0, s>>>(list);
    return cudaGetLastError();
}

cudaError_t launch_build_table(const TableParams& tp, int n_orb, int na, int nb,
                               const unsigned long long* T, unsigned long long* slots,
                               uint32_t* filter, unsigned long long* aset,
                               unsigned long long* bset, Counters* ctr, cudaStream_t s, unsigned* jkey,
                               unsigned* jlen, bool early) {
    if (tp.n <= 0) return cudaSuccess;
    const long long blocks = (tp.n + 255) / 256;
    return launch_early(build_table_kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, s, early, tp, n_orb, na,
                        nb, T, slots, filter, aset, bset, ctr, jkey, jlen);
}

cudaError_t launch_eloc_main(const SysParams& sp, const TableParams& tp, const EvalParams& ep,
                             const LaunchCfg& c, cudaStream_t s) {
    if (ep.n_u <= 0) return cudaSuccess;
    // per-sample digests, hit lists or work counters asked for: the diagnostic instantiations
    // (qc_kernels_diag.cu)
    if (ep.hit_count != nullptr || ep.hit_rowsum != nullptr || ep.hit_signsum != nullptr || ep.hit_list != nullptr ||
        ep.work != nullptr)
        return launch_eloc_main_diag(sp, tp, ep, c, s);
    return launch_main_variant<false>(sp, tp, ep, c, s);
}

cudaError_t launch_reduce(const EvalParams& ep, double* partials, int nblk, void* summary_dev,
                          long long pairs_per_sample, cudaStream_t s, bool early) {
    qc_eloc_summary* out = static_cast<qc_eloc_summary*>(summary_dev);
    if (ep.n_u <= kRedSmallRows) {
        return launch_early(reduce_small_kernel, dim3(kRedCluster), dim3(kRedThreads), 0, s, early, ep, out,
                            pairs_per_sample, nblk);
    }
    const cudaError_t e = launch_early(reduce_pass1, dim3(nblk), dim3(kRedThreads), 0, s, early, ep, partials);
    if (e != cudaSuccess) return e;
    return launch_early(reduce_pass2, dim3(nblk), dim3(kRedThreads), 0, s, early, ep, partials, out, pairs_per_sample);
}

int max_active_ctas(int kernel, int precision, int unroll, int threads, size_t smem, int lean, int join, int seg) {
    const void* f = precision == QC_FP64 ? main_kernel_ptr<QC_FP64, false>(kernel, unroll, lean, join, seg)
                                         : main_kernel_ptr<QC_FP32_COMP, false>(kernel, unroll, lean, join, seg);
    int n = 0;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, f, threads, smem) == cudaSuccess ? n : 0;
}

cudaError_t prepare_kernels(size_t max_smem) {
    const cudaError_t e = prepare_variant<false>(max_smem);
    const cudaError_t d = prepare_kernels_diag(max_smem);
    return e != cudaSuccess ? e : d;
}

}  // namespace qc
