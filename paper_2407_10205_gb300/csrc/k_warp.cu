// k_warp.cu -- resident PHIA kernel for small dense instances (N <= 256) on warp-level
// tensor-core MMAs (mma.sync m16n8k16 bf16, FP32 accumulation of integer products), all
// iterations in one launch.
//
// What bounds these sizes is not a rate but the chain of one iteration: the next field needs
// every spin of this one.  A tcgen05 iteration pays for its hand-overs (an MMA chain of
// about 70 cycles an instruction, a commit, an mbarrier wait, a tensor-memory load, a proxy
// fence) before any of its arithmetic; a warp-level MMA leaves its sum in the registers of the
// threads that use it, so an iteration here is shared-memory loads of the spins, ceil(N/16)
// MMAs in two chains and the update.
//
// One CTA owns 8 replicas; warp w owns the spins [16w, 16w + 16):
//  - A = the warp's 16 rows of J as MMA fragments (bf16, exact for every int8 k), held in
//    registers for the whole run.  (e4m3 fragments would take half the registers, but the
//    warp-level e4m3 MMA runs as conversions and two FP16 MMAs here: 12 more instructions a
//    K-step, N = 200: 0.99 us an iteration against 0.76.)
//  - B = the spins of the CTA's replicas in shared memory, stored as the fragments that the
//    MMA reads: 8 bytes per lane and K-step, so a K-step is one conflict-free 8-byte load.
//    Warp w writes its 16 spins: its signs sit in the accumulator layout (lane = spin,
//    register pair = replicas) and two movmatrix turn them;
//  - D = J s lands in registers: lane (g, q) holds spins 16w + g and 16w + g + 8 for replicas
//    2q and 2q + 1; |D| <= 127 x 256 < 2^24, so the FP32 sum is exact.
// x and v of those (spin, replica) pairs stay in registers.  Per iteration and warp: barrier;
// loads and MMAs, and while they run the derivative factors (they need the position alone) and
// the sums of the previous iteration's energy terms; then field (Eq. 6), momentum (Eqs. 5, 8,
// A7), refresh, position, signs into the next B.  (With mbarriers in the barrier's place and the
// energies behind the spins, N = 64 took 0.55 us an iteration against 0.37.)
// A records warp settles iteration it - 2 meanwhile (Table 3, state 5) and says which replicas
// improved; a phase later the warps, which remember the signs of their elements for three
// iterations, take them over into the best state that they hold, a bit per element.  (With the
// records spread over the compute warps instead, N = 200 took 1.25 us an iteration against
// 0.77: a replica's record is some 50 instructions.)
//
// Per iteration, 256 replicas, this kernel and the tcgen05 resident one (us): N = 16 0.31 / 0.85,
// 64 0.34 / 0.83, 128 0.50 / 0.86, 200 0.80 / 1.12, 230 0.82 / 1.18; at N = 256 the registers of
// 17 warps run short and it loses.  (Factors and energies between the MMAs instead of after them:
// N = 64 0.44 against 0.33, 200 0.88 against 0.79; the MMAs are the longer chain.)
#include <algorithm>
#include <climits>

#include "device_common.cuh"
#include "phia_internal.h"
#include "warp_mma.cuh"

namespace phia {

namespace {

template <int KW>
struct WarpShared {
    uint2 B[2][KW][32];                    // spins of iteration t in slot t % 2, as MMA B fragments
    int32_t epart[2][8][KW];               // per-warp sums of s (I + h), by iteration parity
    alignas(8) uint8_t improved[2][8];     // replicas that improved at the iteration settled in a phase
    int32_t stop[2];                       // by phase parity
};

// KW: compute warps, 16 spins each; CTAS: how many of them an SM has to hold.
template <int KW, bool BATCHED, int CTAS>
__global__ void __launch_bounds__(32 * (KW + 1), CTAS) warp_small_kernel(const RunArgs a) {
    __shared__ WarpShared<KW> sm;
    // The instance: the run's own, or the CTA's entry of a batch's table.
    SmallCta ic;
    if constexpr (BATCHED) ic = a.small_cta[blockIdx.x];
    else ic = SmallCta{a.Jk, a.hk, a.N, a.W, a.inst, a.q, (int32_t)blockIdx.x * 8, 0, 0, a.target};
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int g = lane >> 2, q = lane & 3;
    const int N = ic.N;
    const int nk = (N + 15) / 16;          // K-steps with spins (a batch's launch is sized for its largest member)
    const int nit = (int)a.nsteps, t0 = (int)a.t0;
    const bool stops = a.stop_at_target && !BATCHED;
    if (tid < 16) sm.improved[tid >> 3][tid & 7] = 0;
    if (tid < 2) sm.stop[tid] = 0;

    // Phase it: iteration it itself, the energies of it - 1, the records of it - 2, the best spins
    // of it - 3; three more phases finish the last iteration.
    if (warp == KW) {
        // Records warp: lane l keeps the record of replica l % 8 (four lanes alike).
        const int c = lane & 7, part = lane >> 3, r = ic.rbase + c;
        Record rec;
        rec.load(a, ic.rec_off, r);
        int it = 0;
        bool stopped = false;
        for (; it < nit + 3; ++it) {
            __syncthreads();
            if (stops && it > 0 && sm.stop[(it - 1) & 1]) {
                stopped = true;
                break;
            }
            const int ir = it - 2;                     // the iteration to settle
            bool imp = false;
            if (ir >= 0 && ir < nit) {
                long long twice = 0;
#pragma unroll
                for (int w = 0; w < KW; w += 4)
                    if (w + part < KW) twice += sm.epart[ir & 1][c][w + part];
                if constexpr (KW > 1) {
                    twice += __shfl_xor_sync(0xffffffffu, twice, 8);
                    twice += __shfl_xor_sync(0xffffffffu, twice, 16);
                } else {
                    twice = __shfl_sync(0xffffffffu, twice, c);
                }
                bool first_hit;
                imp = rec.settle(a, ic.target, t0 + ir, twice, first_hit);
                if (stops && first_hit && part == 0) atomicMin(a.min_hit, (unsigned long long)(t0 + ir));
            }
            if (part == 0) sm.improved[it & 1][c] = imp;
            // Early stop: once the records of iteration t = it - 3 (settled a phase ago) reach the
            // earliest hit, t + 1 is the last iteration that is recorded and the next phase ends the run.
            if (stops && lane == 0)
                sm.stop[it & 1] = it >= 3 && it - 3 <= nit - 2 &&
                                  *(volatile unsigned long long *)a.min_hit <= (unsigned long long)(t0 + it - 3);
        }
        if (part == 0) rec.store(a, ic.rec_off, r);
        if (lane == 0)
            atomicAdd(a.replica_iters, (unsigned long long)((long long)min(8, a.R - ic.rbase) * (stopped ? it - 2 : nit)));
        return;
    }
    const int i[2] = {16 * warp + g, 16 * warp + g + 8};       // this thread's two spins
    uint32_t af[KW][4];
    load_fragments<kOpBF16, KW>(af, ic.Jk, N, i, q);
    Elems s;
    float hf[2];
    int32_t h2c[2];                         // 2 h, less the bits of the rounding constant
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const int32_t h = i[u] < N ? ic.hk[i[u]] : 0;
        hf[u] = (float)h;
        h2c[u] = 2 * h - (int32_t)kMagicBits;
    }
    const int r0 = ic.rbase + 2 * q;
    initial_state(s, a, ic, r0, i);
    sm.B[0][warp][lane] = spin_fragment_bf16(s.m);
    const float inv_tm1 = inv_tm1_of(a.T_total), gq = a.gamma * ic.q, eps = a.eps, gamma = a.gamma;
    const int refresh = a.refresh, deriv = a.deriv;
    int rc = refresh > 0 ? (t0 + 1) % refresh : 1;             // (t + 1) mod refresh
    // The field and spins of the previous iteration, whose energy terms are still to be summed.
    float d[2][2];
    uint32_t mp[2][2];
    // Signs of the last iterations, newest first, and those of the best state.
    uint32_t hist[3] = {0u, 0u, 0u};
    BestBits best;
    bool stopped = false;
    for (int it = 0; it < nit + 3; ++it) {
        __syncthreads();
        const uint32_t imp2 = *reinterpret_cast<const uint16_t *>(&sm.improved[(it + 1) & 1][2 * q]);   // at it - 3
        if (stops && it > 0 && sm.stop[(it - 1) & 1]) {
            best.take(imp2, hist[2]);
            stopped = true;
            break;
        }
        const bool runs = it < nit;
        float acc[2][4], f[2][2];
        if (runs) {
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e >> 2][e & 3] = 0.0f;
#pragma unroll
            for (int ks = 0; ks < KW; ++ks) {
                if (BATCHED && ks >= nk) break;
                // At 17 warps the registers are short: the loads stay with their MMAs.
                const uint2 b = KW > 15 ? lds_fragment(&sm.B[it & 1][ks][lane]) : sm.B[it & 1][ks][lane];
                mma_step<kOpBF16>(acc[ks & 1], af[ks], b);
            }
            // While they run: the derivative factors, the previous iteration's energies.
            factors(s, f, deriv, beta_at(t0 + it, inv_tm1, a.beta0, a.beta1) * gq, gamma);
        }
        if (it > 0 && it <= nit) {
            int32_t es[2];
            energy_terms(d, mp, h2c, es);
            const int32_t sum = sum_rows(es, lane);
            if (lane < 8) sm.epart[(it - 1) & 1][2 * q + (lane >> 2)][warp] = sum;
        }
        best.take(imp2, hist[2]);
        hist[2] = hist[1];
        hist[1] = hist[0];
        hist[0] = sign_bits(s);
        if (!runs) continue;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            mp[e >> 1][e & 1] = s.m[e >> 1][e & 1];
            d[e >> 1][e & 1] = KW > 1 ? __fadd_rn(acc[0][e], acc[1][e]) : acc[0][e];
        }
        momentum_step(s, d, f, hf, eps);
        if (it + 1 < nit) {
            if (refresh > 0 && rc == 0) refresh_step(s, a.seed, ic.inst, (uint32_t)r0, i, (uint32_t)(t0 + it + 1));
            position_step(s, eps);
            sm.B[(it + 1) & 1][warp][lane] = spin_fragment_bf16(s.m);
        }
        rc = rc + 1 == refresh ? 0 : rc + 1;
    }
    best.store(a.best_bits + ic.bits_off, ic.rbase, a.R, ic.W, warp, N, lane);
    if (!stopped && a.x_out) export_state(s, a, N, r0, i);
}

template <int KW, bool BATCHED, int CTAS = KW <= 8 ? 2 : 1>
cudaError_t launch_cfg(const RunArgs &a, unsigned ctas, cudaStream_t st) {
    warp_small_kernel<KW, BATCHED, CTAS><<<ctas, 32 * (KW + 1), 0, st>>>(a);
    return cudaGetLastError();
}

template <bool BATCHED>
cudaError_t launch_n(const RunArgs &a, int n, unsigned ctas, cudaStream_t st) {
    const int kw = (n + 15) / 16;
    if constexpr (!BATCHED) {
        if (kw <= 1) return launch_cfg<1, false>(a, ctas, st);
        if (kw <= 2) return launch_cfg<2, false>(a, ctas, st);
        // Two CTAs of 9 warps on an SM leave a thread 96 registers, which cost an iteration 0.1 us:
        // only where there are more CTAs than SMs (N = 128: 0.49 against 0.65 us up to 1216
        // replicas, 1.04 against 0.79 at 2048).
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        if (kw > 6 && kw <= 8 && (int)ctas <= sms) return launch_cfg<8, false, 1>(a, ctas, st);
        if (kw > 4 && kw <= 6) return launch_cfg<6, false>(a, ctas, st);
        if (kw == 16) return launch_cfg<16, false>(a, ctas, st);
    }
    if (kw <= 4) return launch_cfg<4, BATCHED>(a, ctas, st);
    if (kw <= 8) return launch_cfg<8, BATCHED>(a, ctas, st);
    // By the size of its largest member in a batch too: built for 16 warps, whose registers run short, 32
    // members of 150 spins x 512 replicas took 19.8 us an iteration.
    if (kw <= 10) return launch_cfg<10, BATCHED>(a, ctas, st);
    if (kw <= 13) return launch_cfg<13, BATCHED>(a, ctas, st);
    return launch_cfg<15, BATCHED>(a, ctas, st);
}

}  // namespace

int warp_small_max_n() { return 256; }

int warp_small_auto_n() { return 240; }

double warp_small_estimate(int N, int R, int sms) {
    const int kw = (N + 15) / 16, per_sm = kw <= 6 ? 16 / (kw + 1) : kw <= 8 ? 2 : 1;
    const int waves = ((R + 7) / 8 + sms * per_sm - 1) / (sms * per_sm);
    return waves * (0.35 + 0.0023 * N);
}

cudaError_t launch_warp_small(const RunArgs &a, cudaStream_t st, int *launches) {
    if (a.N > warp_small_max_n()) return cudaErrorInvalidValue;
    if (launches) *launches += 1;
    return launch_n<false>(a, a.N, (unsigned)((a.R + 7) / 8), st);
}

cudaError_t launch_warp_small_batch(const RunArgs &a, int nmax, cudaStream_t st) {
    if (a.small_ctas < 1) return cudaSuccess;
    if (nmax > warp_small_auto_n()) return cudaErrorInvalidValue;
    return launch_n<true>(a, nmax, (unsigned)a.small_ctas, st);
}

}  // namespace phia
