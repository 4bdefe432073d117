// k_cluster.cu -- resident PHIA kernel for dense instances past one CTA's registers, on
// warp-level tensor-core MMAs over a thread-block cluster, all iterations in one launch.
//
// As in k_warp.cu the chain of an iteration is what bounds these sizes, and J stays in
// registers as MMA fragments; here the rows of J are spread over the CTAs of a cluster, 8 or 12
// warps of 16 spins each, and a cluster owns 8 replicas.  The only thing that
// crosses CTAs in an iteration are the signs: every warp sends its 16 spins' fragments to all
// CTAs of the cluster with st.async, which counts the bytes on the receiver's mbarrier, so a
// CTA goes on the moment that all spins of the iteration have arrived and there is no barrier.
//
// The spin buffers alternate by iteration parity.  A warp sends the spins of iteration it + 1
// after its MMAs of iteration it, and no warp anywhere can have them all before every warp has
// sent its own; so whoever writes slot it % 2 again (the spins of it + 2) does so after every
// warp has read it.
//
// The energy terms of iteration it go, a phase later, to the cluster's first CTA (rank 0), whose
// eight warps settle a replica each in the phase after (Table 3, state 5) and send every CTA
// whether it improved; the warps take that in phase it + 4, having kept the signs of their
// elements that long, and hold the best states, a bit per element.  The lag makes both
// exchanges' slots (four, by iteration) safe: a phase takes the mask of four iterations ago, so
// a slot's next use comes after its last one was read.  Every wait is bounded; one that runs
// out sets the run's error flag and the warp winds down.
//
// bf16 fragments up to 512 spins; above, e4m3 ones, as bf16 rows of J no longer fit in registers.
// Per iteration (us): N = 512 x 256 replicas 1.15 against 10.9 with one launch per iteration,
// 600 x 128 1.68 against 11.2, 1000 x 64 2.35 against 11.7; 333 x 500 1.54.  (With plain remote stores, a fence and an
// arrival on every CTA's mbarrier in the place of st.async, N = 512 took 1.8.)
#include <algorithm>
#include <atomic>
#include <climits>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "device_common.cuh"
#include "phia_internal.h"
#include "warp_mma.cuh"

namespace phia {

namespace {

constexpr int kLag = 4;              // phases until an iteration's improved mask is taken
constexpr int kMaxWarps = 64;        // warps of a cluster (N <= 1024)

template <int KS>
struct ClusterShared {
    uint2 B[2][KS][32];                           // spins of iteration t in slot t % 2, as B fragments
    int32_t epart[4][8][kMaxWarps];            // rank 0: per-warp sums of s (I + h), by iteration
    uint32_t improved[4][8];                      // by iteration
    uint64_t full[2];                             // all spins of an iteration have arrived
    uint64_t ebar[4];                             // rank 0: all energy sums of an iteration
    uint64_t ibar[4];                             // whether the eight replicas improved at an iteration
    int32_t timed_out;
};

__device__ __forceinline__ uint32_t map_rank(uint32_t saddr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(saddr), "r"(rank));
    return r;
}
// Asynchronous stores into a CTA of the cluster, counted in bytes on its mbarrier.
__device__ __forceinline__ void st_async_u32(uint32_t addr, uint32_t v, uint32_t mbar) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v), "r"(mbar)
                 : "memory");
}
__device__ __forceinline__ void st_async_u64(uint32_t addr, uint2 v, uint32_t mbar) {
    const uint64_t w = (uint64_t)v.x | ((uint64_t)v.y << 32);
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(w), "r"(mbar)
                 : "memory");
}
// KS: MMA K-steps of 32 bytes (every spin of the instance); CW: warps per CTA; BATCHED: the cluster's
// instance is its entry of a batch's table (a.small_cta).
template <int KS, int OP, int CW, bool BATCHED>
__global__ void __launch_bounds__(32 * CW, 1) cluster_small_kernel(const RunArgs a, int cl) {
    using Sh = ClusterShared<KS>;
    extern __shared__ __align__(16) uint8_t smem[];
    Sh *sm = reinterpret_cast<Sh *>(smem);
    volatile int32_t *tout = &sm->timed_out;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, q = lane & 3;
    SmallCta ic;
    if constexpr (BATCHED) ic = a.small_cta[blockIdx.x / cl];
    else ic = SmallCta{a.Jk, a.hk, a.N, a.W, a.inst, a.q, (int32_t)(blockIdx.x / cl) * 8, 0, 0, a.target};
    const int N = ic.N, nit = (int)a.nsteps;
    const int rank = (int)cluster_ctarank();
    const int rbase = ic.rbase;
    const int nwarps = (N + 15) / 16;                 // warps of the cluster that own spins
    const uint64_t kWaitNs = a.wait_ns > 0 ? (uint64_t)a.wait_ns : kWaitTimeoutNs;
    const uint32_t bytes = (uint32_t)(nwarps * 32) * (OP == kOpE4M3 ? 4u : 8u);   // an iteration's spins
    const uint32_t ebytes = (uint32_t)nwarps * 32;    // and energy sums

    for (int e = tid; e < 2 * KS * 32; e += blockDim.x) (&sm->B[0][0][0])[e] = make_uint2(0u, 0u);
    if (tid == 0) {
        for (int s = 0; s < 2; ++s) mbar_init(&sm->full[s], 1);
        for (int s = 0; s < 4; ++s) {
            mbar_init(&sm->ebar[s], 1);
            mbar_init(&sm->ibar[s], 1);
        }
        sm->timed_out = 0;
        fence_mbarrier_init();
        for (int s = 0; s < 2; ++s) mbar_arrive_expect_tx(&sm->full[s], bytes);
        for (int s = 0; s < 4; ++s) {
            mbar_arrive_expect_tx(&sm->ebar[s], ebytes);
            mbar_arrive_expect_tx(&sm->ibar[s], 32);
        }
    }
    __syncthreads();
    cluster_sync_all();          // every CTA's buffers are cleared and its barriers exist

    const int gw = rank * CW + warp;                  // this warp among the cluster's
    if (gw < nwarps) {
        const int i[2] = {16 * gw + g, 16 * gw + g + 8};
        uint32_t af[KS][4];
        load_fragments<OP, KS>(af, ic.Jk, N, i, q);
        Elems s;
        float hf[2];
        int32_t h2c[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int32_t h = i[u] < N ? ic.hk[i[u]] : 0;
            hf[u] = (float)h;
            h2c[u] = 2 * h - (int32_t)kMagicBits;
        }
        // This lane's place in a spin buffer: slot 0 in this CTA's addresses.
        const uint32_t spin0 = OP == kOpE4M3 ? smem_u32(&sm->B[0][gw >> 1][lane]) + 4 * (gw & 1) : smem_u32(&sm->B[0][gw][lane]);
        const uint32_t full0 = smem_u32(&sm->full[0]);
        auto send_spins = [&](int slot) {
            const uint32_t addr = spin0 + (uint32_t)(slot * KS * 32 * 8), bar = full0 + 8 * slot;
            if constexpr (OP == kOpE4M3) {
                const uint32_t b = spin_fragment_e4m3(s.m);
                for (int c = 0; c < cl; ++c) st_async_u32(map_rank(addr, c), b, map_rank(bar, c));
            } else {
                const uint2 b = spin_fragment_bf16(s.m);
                for (int c = 0; c < cl; ++c) st_async_u64(map_rank(addr, c), b, map_rank(bar, c));
            }
        };
        const int r0 = rbase + 2 * q;
        initial_state(s, a, ic, r0, i);
        send_spins(0);
        const float inv_tm1 = inv_tm1_of(a.T_total), gq = a.gamma * ic.q, eps = a.eps, gamma = a.gamma;
        const int refresh = a.refresh, deriv = a.deriv, t0 = (int)a.t0;
        int rc = refresh > 0 ? (t0 + 1) % refresh : 1;
        // Energy terms of iteration it (d: its field, m: its spins) to rank 0.
        const uint32_t epart0 = map_rank(smem_u32(&sm->epart[0][0][0]), 0), ebar0 = map_rank(smem_u32(&sm->ebar[0]), 0);
        auto put_energy = [&](int it, const float (&d)[2][2], const uint32_t (&m)[2][2]) {
            int32_t es[2];
            energy_terms(d, m, h2c, es);
            const int32_t sum = sum_rows(es, lane);
            if (lane < 8)
                st_async_u32(epart0 + 4u * (uint32_t)(((it & 3) * 8 + 2 * q + (lane >> 2)) * kMaxWarps + gw), (uint32_t)sum,
                             ebar0 + 8 * (it & 3));
        };
        Record rec;
        rec.live = false;
        const bool records = rank == 0 && warp < 8;
        if (records) rec.load(a, ic.rec_off, rbase + warp);
        const uint32_t imp0 = smem_u32(&sm->improved[0][0]), ibar0 = smem_u32(&sm->ibar[0]);
        // Rank 0: record of iteration it, replica `warp`, and word of it to every CTA.
        auto settle = [&](int it) -> bool {
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&sm->ebar[it & 3], (uint32_t)(it >> 2) & 1u, kWaitNs))) return false;
            if (tid == 0) mbar_arrive_expect_tx(&sm->ebar[it & 3], ebytes);      // for it + 4
            const volatile int32_t *e = sm->epart[it & 3][warp];
            const int32_t e0 = lane < nwarps ? e[lane] : 0, e1 = lane + 32 < nwarps ? e[lane + 32] : 0;
            const long long twice = (long long)__reduce_add_sync(0xffffffffu, (e0 & 0xffff) + (e1 & 0xffff)) +
                                    ((long long)__reduce_add_sync(0xffffffffu, (e0 >> 16) + (e1 >> 16)) << 16);
            bool first_hit;
            const bool imp = rec.settle(a, ic.target, t0 + it, twice, first_hit);
            if (lane < cl)
                st_async_u32(map_rank(imp0 + (uint32_t)((it & 3) * 8 + warp) * 4, (uint32_t)lane), imp,
                             map_rank(ibar0 + 8 * (it & 3), (uint32_t)lane));
            return true;
        };
        uint32_t hist[kLag] = {0u, 0u, 0u, 0u};
        BestBits best;
        auto take = [&](int it, uint32_t was) -> bool {
            if (!__all_sync(0xffffffffu, mbar_wait_bounded(&sm->ibar[it & 3], (uint32_t)(it >> 2) & 1u, kWaitNs))) return false;
            if (tid == 0) mbar_arrive_expect_tx(&sm->ibar[it & 3], 32);          // for it + 4
            const volatile uint32_t *w = &sm->improved[it & 3][2 * q];
            best.take(w[0] | (w[1] << 8), was);
            return true;
        };
        // Phase it: iteration it itself and its energies, the records of it - 2, the best spins of
        // it - kLag; kLag more phases finish the last iteration.  What the next iteration waits for
        // comes first: the energies and records follow the phase's spins.
        bool ok = true;
        for (int it = 0; it < nit + kLag; ++it) {
            const bool runs = it < nit;
            if (runs) ok = mbar_wait_bounded(&sm->full[it & 1], (uint32_t)(it >> 1) & 1u, kWaitNs);
            ok = __all_sync(0xffffffffu, ok && !*tout);
            if (!ok) break;
            const uint32_t now = sign_bits(s);
            if (runs) {
                if (tid == 0) mbar_arrive_expect_tx(&sm->full[it & 1], bytes);   // for it + 2
                float acc[2][4], f[2][2], d[2][2];
                uint32_t m[2][2];
#pragma unroll
                for (int e = 0; e < 8; ++e) acc[e >> 2][e & 3] = 0.0f;
#pragma unroll
                for (int ks = 0; ks < KS; ++ks) mma_step<OP>(acc[ks & 1], af[ks], lds_fragment(&sm->B[it & 1][ks][lane]));
                factors(s, f, deriv, beta_at(t0 + it, inv_tm1, a.beta0, a.beta1) * gq, gamma);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    m[e >> 1][e & 1] = s.m[e >> 1][e & 1];
                    d[e >> 1][e & 1] = __fadd_rn(acc[0][e], acc[1][e]);
                }
                momentum_step(s, d, f, hf, eps);
                if (it + 1 < nit) {
                    if (refresh > 0 && rc == 0) refresh_step(s, a.seed, ic.inst, (uint32_t)r0, i, (uint32_t)(t0 + it + 1));
                    position_step(s, eps);
                    send_spins((it + 1) & 1);
                }
                rc = rc + 1 == refresh ? 0 : rc + 1;
                // The mask of four iterations ago has been read by this warp before its energies of this
                // one let rank 0 write that slot again.
                if (it >= kLag) ok = take(it - kLag, hist[kLag - 1]);
                if (ok) put_energy(it, d, m);
            } else if (it >= kLag) {
                ok = take(it - kLag, hist[kLag - 1]);
            }
            if (ok && records && it >= 2 && it - 2 < nit) ok = settle(it - 2);
#pragma unroll
            for (int k = kLag - 1; k > 0; --k) hist[k] = hist[k - 1];
            hist[0] = now;
        }
        if (ok) {
            best.store(a.best_bits + ic.bits_off, rbase, a.R, ic.W, gw, N, lane);
            if (a.x_out) export_state(s, a, N, r0, i);
        } else {
            *tout = 1;
        }
        if (records && lane == 0) rec.store(a, ic.rec_off, rbase + warp);
        if (gw == 0 && lane == 0)
            atomicAdd(a.replica_iters, (unsigned long long)((long long)min(8, a.R - rbase) * nit));
    }
    __syncthreads();
    if (tid == 0 && sm->timed_out) atomicExch(a.err, 1);
    cluster_sync_all();          // no CTA leaves while another may still write into it
}

// Launch of a run (a) on `clusters` clusters, or with a null the number of clusters that the GPU
// holds at once.
template <int KS, int OP, int CW, bool BATCHED>
cudaError_t launch_cfg(const RunArgs *a, int N, int clusters, cudaStream_t st, int *resident) {
    constexpr size_t smem = sizeof(ClusterShared<KS>);
    const int cl = (N + 16 * CW - 1) / (16 * CW);
    auto k = cluster_small_kernel<KS, OP, CW, BATCHED>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[1];
    cfg.gridDim = dim3((unsigned)cl * (unsigned)clusters);
    cfg.blockDim = dim3(32 * CW);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cl;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (!a) {
        // A property of the device and the kernel, asked for once: runs ask before every launch.
        constexpr int kDevices = 16, kSizes = 9;
        static std::atomic<int> known[kDevices][kSizes];
        int dev = 0;
        e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        const bool keep = dev < kDevices && cl < kSizes;
        *resident = keep ? known[dev][cl].load() : 0;
        if (*resident > 0) return cudaSuccess;
        e = cudaOccupancyMaxActiveClusters(resident, reinterpret_cast<const void *>(k), &cfg);
        if (e == cudaSuccess && keep) known[dev][cl].store(*resident);
        return e;
    }
    e = cudaLaunchKernelEx(&cfg, k, *a, cl);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// bf16 fragments up to 512 spins (the warp-level e4m3 MMA runs as conversions and two FP16 MMAs),
// e4m3 ones above, where bf16 would not fit the registers.  8 warps per CTA, 12 between 257 and
// 384 spins (two CTAs instead of three).
template <bool BATCHED>
cudaError_t dispatch(const RunArgs *a, int N, int clusters, cudaStream_t st, int *resident) {
    if constexpr (!BATCHED)
        if (N <= 256) return launch_cfg<16, kOpBF16, 8, false>(a, N, clusters, st, resident);
    if (N <= 384) return launch_cfg<24, kOpBF16, 12, BATCHED>(a, N, clusters, st, resident);
    if (N <= 512) return launch_cfg<32, kOpBF16, 8, BATCHED>(a, N, clusters, st, resident);
    if constexpr (!BATCHED) {
        if (N <= 768) return launch_cfg<24, kOpE4M3, 8, false>(a, N, clusters, st, resident);
        return launch_cfg<32, kOpE4M3, 8, false>(a, N, clusters, st, resident);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

int cluster_small_min_n() { return 128; }          // rank 0 settles a replica per warp
int cluster_small_max_n(int op) { return op == kOpE4M3 ? 1024 : 512; }

double cluster_small_estimate(int N, int R, int op, int sms, double limit) {
    if (N < cluster_small_min_n() || N > cluster_small_max_n(op)) return 1e30;
    const double wave = N <= 512 ? 0.8 + 0.0009 * N : 0.8 + 0.0016 * N;
    // The number of clusters that the GPU holds is asked of the kernel, which loads its code once per
    // process (a first run at N = 600 x 2000 replicas 1.0 ms without it, 2.1 with it): not where CTAs on all
    // SMs, one on each (168 registers a thread and more), would not be fast enough.
    const int cl = (N + 127) / 128, most = std::max(1, N > 256 && N <= 384 ? sms / 2 : sms / cl);
    if (((R + 7) / 8 + most - 1) / most * wave >= limit) return 1e30;
    int resident = 0;
    if (dispatch<false>(nullptr, N, 1, nullptr, &resident) != cudaSuccess || resident < 1) {
        cudaGetLastError();
        return 1e30;
    }
    const int waves = ((R + 7) / 8 + resident - 1) / resident;
    return waves * wave;
}

cudaError_t launch_cluster_small(const RunArgs &a, int op, cudaStream_t st, int *launches) {
    if (a.N < cluster_small_min_n() || a.N > cluster_small_max_n(op)) return cudaErrorInvalidValue;
    if (launches) *launches += 1;
    return dispatch<false>(&a, a.N, (a.R + 7) / 8, st, nullptr);
}

int cluster_batch_max_n() { return 512; }

cudaError_t launch_cluster_batch(const RunArgs &a, int nmax, cudaStream_t st) {
    if (a.small_ctas < 1) return cudaSuccess;
    if (nmax > cluster_batch_max_n()) return cudaErrorInvalidValue;
    return dispatch<true>(&a, nmax, a.small_ctas, st, nullptr);
}

}  // namespace phia
