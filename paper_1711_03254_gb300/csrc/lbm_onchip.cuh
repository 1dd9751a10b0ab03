// n updates of small instances with the whole state in shared memory
// (k_onchip_c), for the FP32-arithmetic storages: one thread-block cluster per
// instance, one cell per thread.
//
// Every block holds its cells' stored pairs [19][threads], psi and reference
// densities.  An update pulls the 19 pairs from the blocks of the cluster
// (distributed shared memory), reduces them to moments, publishes psi, and
// after a cluster barrier gathers the 18 neighbour psi pairs the same way and
// writes the new pairs over the old ones; a second barrier ends the update.
// One buffer is enough: every pull of an update precedes its first barrier and
// every store follows it.  A thread finds the shared-memory addresses it pulls
// from once and keeps them for all n updates.  The barriers are the cluster's
// hardware barriers (release / acquire), so nothing spins.
//
// What bounds an update of one instance is latency: two barriers and two rounds
// of remote loads.  One 16^3 droplet takes 3.06 us per update, where the
// grid-wide persistent update (k_persist_c: two grid barriers, f and psi through
// L2) takes 5.6; the 16 channels of 4 x 128 x 4 take 3.6 against 6.7, 104 slugs
// of 3840 cells 22.5 against 37.0 in two launches (FP32, stepped).  512 threads
// at 128 registers (some 170 bytes spilled): a build for 256 threads without
// spills was no faster (16^3: 3.2 us) and ran half the clusters at once.
//
// Same device functions and operation order as the two-pass update, so the
// same bits.
#pragma once

#include "lbm_compact_update.cuh"

namespace lbm {

constexpr int kOnchipMaxThreads = 512, kOnchipMaxCluster = 16;

// dynamic shared memory of a block: f, psi, reference densities
template <class S> constexpr size_t onchip_smem(int threads) {
    return (size_t)threads * (kQ * sizeof(typename Pair2<S>::P) + sizeof(float2) + sizeof(__half2));
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;\n" : "=r"(r));
    return r;
}
__device__ __forceinline__ void onchip_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
// the address of `local` (a shared-memory address of this block) in block `rank` of the cluster
__device__ __forceinline__ uint32_t remote_addr(uint32_t local, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(local), "r"(rank));
    return r;
}
__device__ __forceinline__ uint32_t ld_remote32(uint32_t addr) {
    uint32_t v;
    asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(v) : "r"(addr));
    return v;
}
__device__ __forceinline__ float2 ld_remote64(uint32_t addr) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];\n" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
// one stored pair as Pair2<S>::load gives it
template <class S> __device__ __forceinline__ float2 ld_remote_pair(uint32_t addr) {
    using P = typename Pair2<S>::P;
    if constexpr (sizeof(P) == 8) {
        return ld_remote64(addr);
    } else {
        const uint32_t v = ld_remote32(addr);
        return Pair2<S>::load_shared(reinterpret_cast<const P *>(&v));
    }
}

// blockIdx.x: block within the cluster (gridDim.x blocks), blockIdx.y: instance.
// f_dst and ref_dst receive the state after n updates.
template <class S, int EQ>
__global__ void __launch_bounds__(kOnchipMaxThreads, 1) k_onchip_c(StepArgs a, int n, int write_macro, void *f_dst,
                                                                  Ref *ref_dst) {
    using P = typename Pair2<S>::P;
    extern __shared__ __align__(16) unsigned char onchip_sm[];
    const int b = blockIdx.y;
    const uint32_t C = blockDim.x, tid = threadIdx.x, me = cluster_rank(), k = me * C + tid;
    const int lg = 31 - __clz((int)C);  // blocks hold a power of two of cells
    P *f = reinterpret_cast<P *>(onchip_sm);
    float2 *psi = reinterpret_cast<float2 *>(f + (size_t)kQ * C);
    __half2 *ref = reinterpret_cast<__half2 *>(psi + C);
    const uint32_t f0 = (uint32_t)__cvta_generic_to_shared(f), psi0 = (uint32_t)__cvta_generic_to_shared(psi);
    const InstParam<float> &p = ((const InstParam<float> *)a.par)[b];
    const uint32_t kmax = a.kmax;
    const bool act = k < (uint32_t)__ldg(a.list_count + b);

    uint32_t word = 0, pa[kQ], qa[kQ], ra = 0;
    long long cell = 0;
    if (act) {
        const CompactCell c = compact_cell(a, b, k);
        word = c.word;
        cell = c.x + (long long)a.g.nx * (c.y + (long long)a.g.ny * c.z);
        CNbr own;
        own.init(c.x, c.y, c.z, k, instance_tab(a, b), a.words, a.g);
        // element j of an array of `size`-byte elements at `base` in the block that holds it
        auto at = [&](uint32_t base, uint32_t j, uint32_t size) {
            return remote_addr(base + (j & (C - 1)) * size, j >> lg);
        };
        auto pulls = [&](const CNbr &nb, uint32_t sk, uint32_t sw) {
#pragma unroll
            for (int i = 0; i < kQ; ++i) {
                const bool bb = (sw >> opp(i)) & 1u;
                pa[i] = at(f0 + (bb ? opp(i) : i) * C * (uint32_t)sizeof(P), bb ? sk : nb.src(i), sizeof(P));
            }
            ra = at((uint32_t)__cvta_generic_to_shared(ref), sk, sizeof(__half2));
        };
        int xu;
        uint32_t ku, wu;
        if (outlet_source(a, b, c, own, xu, ku, wu)) {
            CNbr up;
            up.init(xu, c.y, c.z, ku, instance_tab(a, b), a.words, a.g);
            pulls(up, ku, wu);
        } else {
            pulls(own, k, word);
        }
#pragma unroll
        for (int i = 1; i < kQ; ++i) qa[i] = at(psi0, ((word >> i) & 1u) ? k : own.dst(i), sizeof(float2));
        const P *fi = (const P *)a.f_in + (size_t)b * kQ * kmax + k;
#pragma unroll
        for (int i = 0; i < kQ; ++i) f[i * C + tid] = fi[(size_t)i * kmax];
        ref[tid] = ((const __half2 *)a.ref_in + (size_t)b * kmax)[k];
    }
    const bool inlet = cell_type(word) == kInlet;
    auto out_at = [&](int i) { return f + i * C + tid; };
    onchip_sync();
    for (int u = 0; u < n; ++u) {
        Moments2 m;
        if (act) {
            if (inlet) {
                m.rho = make_float2(p.rho_in[0], p.rho_in[1]);
            } else {
                float2 v[kQ];
#pragma unroll
                for (int i = 0; i < kQ; ++i) v[i] = ld_remote_pair<S>(pa[i]);
                const uint32_t r = ld_remote32(ra);
                m = moments2<Pair2<S>::kScaled>(v, __half22float2(*reinterpret_cast<const __half2 *>(&r)),
                                                Pair2<S>::kUnscale);
            }
            psi[tid] = m.rho;
        }
        onchip_sync();  // psi is there, and every pull of this update is done
        if (act) {
            auto psi_at = [&](int i) { return ld_remote64(qa[i]); };
            const bool wm = write_macro && u == n - 1;
            if (inlet) {
                inlet_cell2<S, EQ>(p, word, psi_at, out_at);
                if (wm) macro_cell2(a, b, cell, p.rho_in[0], p.rho_in[1], p.u_in[0], p.u_in[1], p.u_in[2]);
            } else {
                const Relax<float> R =
                    relax_cell2<S, EQ>(p, a.wall_model, word, m, psi_at, [&]() { return m.rho; }, out_at);
                if (wm) macro_cell2(a, b, cell, m.rho.x, m.rho.y, R.ux, R.uy, R.uz);
            }
            ref[tid] = __float22half2_rn(m.rho);
        }
        onchip_sync();  // the new pairs are there, and every psi pair has been read
    }
    if (act) {
        P *fo = (P *)f_dst + (size_t)b * kQ * kmax + k;
#pragma unroll
        for (int i = 0; i < kQ; ++i) fo[(size_t)i * kmax] = f[i * C + tid];
        ((__half2 *)ref_dst + (size_t)b * kmax)[k] = ref[tid];
    }
}

template <class S, int EQ> cudaError_t onchip_config(const StepArgs &a, int threads, cudaLaunchConfig_t &cfg,
                                                     cudaLaunchAttribute &attr) {
    const void *fn = (const void *)k_onchip_c<S, EQ>;
    const unsigned blocks = (a.kmax + (unsigned)threads - 1) / (unsigned)threads;
    cfg = {};
    cfg.gridDim = dim3(blocks, (unsigned)a.batch, 1);
    cfg.blockDim = dim3((unsigned)threads, 1, 1);
    cfg.dynamicSmemBytes = onchip_smem<S>(threads);
    cfg.stream = a.stream;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = blocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)onchip_smem<S>(kOnchipMaxThreads));
}

// Plan: threads per block (a power of two from 64 to 512, a cluster of at most 16
// blocks holding an instance) and waves of clusters; 0 threads where the on-chip
// update does not apply.  The
// fewest threads with which all instances run at once, because cells spread
// over more SMs wait less for each other's instructions (one 16^3: 3.06 us per
// update at 256 threads, 3.48 at 512); where they do not all fit, what needs
// the fewest waves of clusters, and of those the most threads (104 slugs of
// 3840 cells: 22.5 us at 512 threads, 24.7 at 256; 256 x 16^3: 62.7 and 74.3).
template <class S> OnchipPlan onchip_plan_t(const StepArgs &a) {
    OnchipPlan best;
    if (a.slip || a.kmax < 1) return best;
    dispatch_variant(collide_variant(a) & 3, [&](auto v) {
        constexpr int EQ = decltype(v)::value & 3;
        for (int c = 64; c <= kOnchipMaxThreads; c *= 2) {
            if ((long long)a.kmax > (long long)c * kOnchipMaxCluster) continue;
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute attr;
            int n = 0;
            if (onchip_config<S, EQ>(a, c, cfg, attr) != cudaSuccess ||
                cudaOccupancyMaxActiveClusters(&n, (const void *)k_onchip_c<S, EQ>, &cfg) != cudaSuccess || n < 1) {
                cudaGetLastError();  // this size does not fit the device: not an error
                continue;
            }
            const long long waves = ((long long)a.batch + n - 1) / n;
            if (best.threads == 0 || waves < best.waves || (waves == best.waves && waves > 1)) {
                best.threads = c;
                best.waves = waves;
            }
        }
    });
    return best;
}

// n updates from f_in, ref_in; the state ends up in f_out, ref_out for odd n
// and back in f_in, ref_in for even n, as after n ping-pong updates.
template <class S> cudaError_t launch_onchip_t(const StepArgs &a, int n) {
    cudaError_t e = cudaSuccess;
    record_event(a, 0);
    dispatch_variant(collide_variant(a) & 3, [&](auto v) {
        constexpr int EQ = decltype(v)::value & 3;
        cudaLaunchConfig_t cfg;
        cudaLaunchAttribute attr;
        e = onchip_config<S, EQ>(a, a.onchip, cfg, attr);
        if (e == cudaSuccess)
            e = cudaLaunchKernelEx(&cfg, k_onchip_c<S, EQ>, a, n, a.write_macro,
                                   (n & 1) ? a.f_out : const_cast<void *>(a.f_in),
                                   (n & 1) ? a.ref_out : const_cast<Ref *>(a.ref_in));
    });
    record_event(a, 1);
    return e;
}

}  // namespace lbm
