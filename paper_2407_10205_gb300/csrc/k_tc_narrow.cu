// k_tc_narrow.cu -- overlapped tensor-core PHIA path for few replicas of dense instances: one
// tile of 128 replicas x 32 or 64 output spins per CTA, x and v in registers, every iteration
// of a call in one cooperative launch.
//
// The field I = J s + h (Eq. 6) is computed with the replicas in the rows of the MMA:
//   A = spins of this iteration [Rpad][Kbytes] (128 replicas per tile), one of 4 rotating
//       buffers (iteration t reads buffer t % 4 and writes t + 1 % 4),
//   B = couplings k re-encoded exactly (e4m3 or bf16), [Mpad][Kpad], BN spins per tile (J is
//       symmetric, so the row of output spin i serves as column i),
//   D = s J in tensor memory: lane = replica, column = output spin (FP32, integer-valued,
//       exact below 2^24).
// So an epilogue thread owns one replica and BN / 2 spins for the whole run: its x and v stay
// in registers, its energy terms add up in a register, its spins are consecutive bytes of one
// operand row, and everything that belongs to a spin (h, the end of the row, the masking of N)
// is the same for the whole warp.
//
// What bounds it: the chain of one iteration.  A replica tile's spins are the A operand of all
// its output tiles, so no tile can begin t + 1 before all have finished t: a counter ready[n]
// per replica tile counts the output tiles that have (about 2 us from the last store to the next
// MMA: counter, copies, accumulator), the operands come at about 90 bytes per ns and SM (the
// couplings of the first stages, which do not depend on the iteration, are copied before the
// wait), and the epilogue is 16 or 32 elements a thread.  The wide tiles of k_tc_large.cu (128 x
// 128 .. 256) leave most SMs idle here and carry x and v through global memory: per
// iteration 11.8 us at N = 700 x 1000 replicas against 5.3 here, 14.5 against 8.2 at 1001 x
// 600 (bf16).  With more tiles than SMs the wide ones win (N = 2000 x 4096: 23.4 us against
// 25.8 for this form with wide tiles), so it is not built for that.
//
// Warp roles: warp 0 issues TMA, warp 1 the MMAs (one thread each), warps 2-9 run the epilogue,
// a records warp settles energies and copies best spins, and a signal warp counts the finished
// tile off the epilogue's path.  Between calls x and v live in a spin-interleaved layout
// [Mp/4][Rpad][4] (FP32): the 4 spins of one group sit together for each replica, so a thread
// moves its values as 16-byte vectors and a warp's vector covers 512 contiguous bytes.
//
// Reuse of the rotating buffers is guarded: the m = 0 tile is counted for iteration t only
// after its records warp settled t - 1 (the energy sums of t - 1 share a slot with t + 1), and
// a tile writes the spins of iteration t + 1 into the buffer of t - 3 only after its records
// warp copied t - 3; the improved flags rotate over four slots.  The accumulator needs no guard
// of its own: the MMAs of t + 1 wait for spins that the epilogue counts after it has read t.
// Every wait is bounded; a wait that runs out sets the run's error flag and the CTA winds
// down.  The dependency graph is acyclic: every wait points to an earlier iteration, or to an
// earlier stage of the same one.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>

#include "device_common.cuh"
#include "phia_internal.h"

namespace phia {

namespace {

constexpr int kBM = 128;       // replicas per tile (TMEM lanes)
constexpr int kBKB = 128;      // bytes of K per pipeline stage (one 128-byte swizzle row)
constexpr int kEpiWarps = 8;   // two per TMEM lane quadrant, each half of the columns
constexpr int kThreads = 32 * (2 + kEpiWarps + 2);
constexpr int kChunk = 16;     // output spins per epilogue step (four x/v groups)
constexpr int kStages = 8;
constexpr uint32_t kStageA = kBM * kBKB;

struct NarrowShared {
    uint64_t full[kStages];
    uint64_t empty[kStages];
    uint64_t accf;                // the accumulator holds an iteration's fields
    uint64_t tiledone;            // the epilogue warps finished an iteration
    uint64_t drain;               // every MMA issued has completed
    alignas(16) float h[64];      // field of the tile's spins, 0 past N
    uint32_t tmem_base;
    int32_t timed_out;
    int64_t rec_settled;          // last iteration the records warp settled
    int64_t rec_copied;           // ... and whose best spins it copied
};

// BN output spins per tile: two column groups of BN / 32 chunks.
template <int BN>
struct NarrowTile {
    static constexpr uint32_t kStageB = BN * kBKB;
    static constexpr uint32_t kTmemCols = BN;
    static constexpr int kColsPerWarp = BN / 2;
    static constexpr int kChunks = kColsPerWarp / kChunk;
    static constexpr size_t kSmemBytes = 1024 + kStages * (kStageA + kStageB) + sizeof(NarrowShared);
    static_assert(BN == 32 || BN == 64, "tile width");
    static_assert(kSmemBytes <= 232448, "shared memory over the per-CTA limit");
};

struct NarrowArgs {
    RunArgs a;
    uint8_t *S;         // [4][Rpad][Kbytes] spin operand buffers
    int64_t *Epart;     // [2][Rpad] sums of s (I + h) over output tiles, by iteration parity
    int8_t *flags;      // [4][Rpad] improved at an iteration, by iteration slot
    float *X, *V;       // [Mp/4][Rpad][4] state: replica r, spin i at ((i/4) Rpad + r) 4 + i%4
    int32_t Kbytes, Rpad, Mp;
    int32_t mtiles;     // output-spin tiles
    int32_t rtiles;     // replica tiles
    uint32_t *ready;    // [rtiles] output tiles finished per replica tile, then [rtiles]
                        // iterations settled per replica tile
    uint32_t *sbits;    // [4][Mp/32][Rpad] packed spins by iteration slot, word-major (bit i % 32
                        // of word i / 32 set: s_i = +1)
    int64_t f0, f1;     // this launch's iterations [f0, f1) of the call's
};

// The operand bytes of 4 consecutive spins (e4m3: +1 / -1 = 0x38 / 0xB8) or 2 (bf16: 0x3F80 /
// 0xBF80) from bits [b0, ..) of a mask with a bit set for +1.
__device__ __forceinline__ uint32_t spins4_e4m3(uint32_t plus, int b0) {
    return 0xB8B8B8B8u ^ (((((plus >> b0) & 0xFu) * 0x00204081u) & 0x01010101u) << 7);
}
__device__ __forceinline__ uint32_t spins2_bf16_bits(uint32_t plus, int b0) {
    const uint32_t b = plus >> b0;
    return 0xBF80BF80u ^ (((b & 1u) << 15) | ((b & 2u) << 30));
}

// 32 lanes x 16 consecutive accumulator columns: the load without its wait, and the wait (the
// registers pass through it, so that no use is scheduled before it).
__device__ __forceinline__ void tmem_ld_x16_issue(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait_x16(uint32_t (&r)[16]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// Momentum draw d = t1 of a chunk (out of line: once per trajectory).
__device__ __noinline__ void refresh_chunk(float *v, uint64_t seed, uint32_t inst, uint32_t r, uint32_t i0, uint32_t t1) {
#pragma unroll 1
    for (int j = 0; j < kChunk; ++j) v[j] = draw_v(seed, inst, r, i0 + j, t1);
}

// Record step for K replicas r0 + 32 k of one lane at iteration tt (Table 3, state 5): E from
// the sum that the output tiles accumulated, best / target records, improved flag; the sum
// slot is cleared for iteration tt + 2.  Every load is issued before any store, so that the
// K replicas' round trips overlap.
template <int K>
__device__ __forceinline__ void settle_lane(const NarrowArgs &L, int r0, int64_t tt) {
    const RunArgs &a = L.a;
    unsigned long long *slots = reinterpret_cast<unsigned long long *>(L.Epart) + (size_t)(tt & 1) * L.Rpad;
    long long tw[K], be[K], hs[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int r = r0 + 32 * k;
        const bool live = r < a.R;
        tw[k] = live ? (long long)slots[r] : 0;
        be[k] = live ? (long long)a.best_e[r] : 0;
        hs[k] = live ? (long long)a.hit_step[r] : 0;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int r = r0 + 32 * k;
        if (r >= L.Rpad) continue;
        slots[r] = 0ull;
        int imp = 0;
        if (r < a.R) {
            const long long E = -tw[k] / 2;
            if (!(a.stop_at_target && hs[k] >= 0) && E < be[k]) {
                a.best_e[r] = E;
                a.best_step[r] = tt;
                imp = 1;
            }
            if (a.has_target && hs[k] < 0 && E <= a.target) {
                a.hit_step[r] = tt;
                if (a.hit_ns) a.hit_ns[r] = globaltimer_ns();
            }
        }
        L.flags[(size_t)(tt & 3) * L.Rpad + r] = (int8_t)imp;
    }
}

// Best spins of iteration tt, output spins i0 .. i0 + BN - 1, of the replicas of tile n that
// improved at tt, from the packed spins that the epilogue wrote: a replica to a lane, so that
// the four replicas of a lane load their words side by side and every load is coalesced over
// the lanes.  (Early in a run nearly every replica improves in every iteration: reading the
// operand rows instead, a replica to a warp, took 20 us a tile then and set the pace.)
template <int BN>
__device__ __forceinline__ void copy_best(const NarrowArgs &L, int n, int i0, int64_t tt, int lane) {
    const RunArgs &a = L.a;
    constexpr int K = kBM / 32;
    const int8_t *F = L.flags + (size_t)(tt & 3) * L.Rpad;
    const uint32_t *B = L.sbits + (size_t)(tt & 3) * (L.Mp / 32) * L.Rpad;
    const int w0 = i0 >> 5, r0 = n * kBM + lane;
    bool f[K];
#pragma unroll
    for (int k = 0; k < K; ++k) f[k] = r0 + 32 * k < a.R && __ldcg(F + r0 + 32 * k) != 0;
#pragma unroll
    for (int w = 0; w < BN / 32; ++w) {
        const int left = a.N - (w0 + w) * 32;                  // spins of this word
        if (left <= 0) break;
        const uint32_t valid = left >= 32 ? 0xffffffffu : (1u << left) - 1u;
        uint32_t v[K];
#pragma unroll
        for (int k = 0; k < K; ++k) v[k] = f[k] ? __ldcg(B + (size_t)(w0 + w) * L.Rpad + r0 + 32 * k) : 0u;
#pragma unroll
        for (int k = 0; k < K; ++k)
            if (f[k]) a.best_bits[(size_t)(r0 + 32 * k) * a.W + w0 + w] = v[k] & valid;
    }
}

template <int OP, int BN>
__global__ void __launch_bounds__(kThreads, 1)
    tc_narrow_run(const __grid_constant__ CUtensorMap tmS, const __grid_constant__ CUtensorMap tmJ, const NarrowArgs L) {
    using T = NarrowTile<BN>;
    constexpr int ESZ = OP == kOpE4M3 ? 1 : 2;
    constexpr uint32_t IDESC = make_idesc(OP == kOpE4M3 ? 0u : 1u, kBM, BN);
    constexpr int kColsPerWarp = T::kColsPerWarp;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *sA = smem;
    uint8_t *sB = smem + kStages * kStageA;
    NarrowShared *sh = reinterpret_cast<NarrowShared *>(sB + kStages * T::kStageB);
    volatile int32_t *tout = &sh->timed_out;
    volatile int64_t *rec_settled = &sh->rec_settled, *rec_copied = &sh->rec_copied;

    const RunArgs &a = L.a;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int mt = L.mtiles;
    const int m = (int)blockIdx.x % mt, n = (int)blockIdx.x / mt;     // this CTA's tile
    const int64_t t0 = L.f0, t_end = L.f1, t_call_end = a.t0 + a.nsteps;
    const int KB = L.Kbytes / kBKB;
    const int N = a.N;
    const uint64_t kWaitNs = a.wait_ns > 0 ? (uint64_t)a.wait_ns : kWaitTimeoutNs;
    // A chunk's 16 energy terms s (I + h) add up exactly in FP32 while |I + h| <= 2^20.
    const int32_t h_mine = tid < BN && m * BN + tid < N ? a.hk[m * BN + tid] : 0;
    const bool h_small = (int64_t)a.max_abs_k * (N - 1) + 2 * (int64_t)abs(h_mine) <= (int64_t)1 << 20;
    if (tid < BN) sh->h[tid] = (float)h_mine;
    uint32_t *ready = L.ready, *settled = L.ready + L.rtiles;

    if (warp == 0) {
        tmem_alloc(&sh->tmem_base, T::kTmemCols);
        tmem_relinquish();
    }
    if (tid == 32) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sh->full[s], 1);
            mbar_init(&sh->empty[s], 1);
        }
        mbar_init(&sh->accf, 1);
        mbar_init(&sh->tiledone, kEpiWarps);
        mbar_init(&sh->drain, 1);
        sh->timed_out = 0;
        sh->rec_settled = t0 - 1;
        sh->rec_copied = t0 - 1;
        fence_mbarrier_init();
    }
    tc_fence_before();
    const bool exact_sums = __syncthreads_and(h_small) != 0;
    tc_fence_after();
    const uint32_t tmem = sh->tmem_base;

    if (warp == 0) {
        // TMA producer.
        if (lane == 0 && !a.stall_producer) {
            int64_t kg = 0;
            int64_t armed = 0;          // stages whose couplings are on their way (kg .. armed - 1)
            bool ok = true;
            // Stage k: free, expecting both operands, couplings requested.
            auto arm = [&](int64_t k, int kb) -> bool {
                const int s = (int)(k % kStages);
                if (k >= kStages && (*tout || !mbar_wait_bounded(&sh->empty[s], (uint32_t)((k / kStages) - 1) & 1u, kWaitNs)))
                    return false;
                mbar_arrive_expect_tx(&sh->full[s], kStageA + T::kStageB);
                tma_load_2d(sB + s * T::kStageB, &tmJ, &sh->full[s], kb * (kBKB / ESZ), m * BN);
                return true;
            };
            for (int64_t t = t0; t < t_end && ok; ++t) {
                // The couplings of the first k-blocks go out before the spins are known to be
                // complete: they are what the stages that are free by now wait for.
                const int pre = min(KB, kStages);
                for (int kb = 0; kb < pre && ok; ++kb) {
                    ok = arm(armed, kb);
                    if (ok) ++armed;
                }
                // the spins of iteration t of replica tile n: all its output tiles finished t - 1
                if (!ok || !wait_counter_at_least(ready + n, (uint32_t)(mt * (t - t0)), kWaitNs, tout)) {
                    ok = false;
                    break;
                }
                fence_proxy_async_global();
                const int ybuf = (int)(t & 3) * L.Rpad + n * kBM;
                for (int kb = 0; kb < KB; ++kb, ++kg) {
                    if (kg == armed) {
                        ok = arm(armed, kb);
                        if (!ok) break;
                        ++armed;
                    }
                    const int s = (int)(kg % kStages);
                    tma_load_2d(sA + s * kStageA, &tmS, &sh->full[s], kb * (kBKB / ESZ), ybuf);
                }
            }
            if (!ok) *tout = 1;
            // Copies still in flight (only after a timeout) land before the CTA exits: stages
            // complete in full, and those armed with couplings alone once their missing half
            // is brought in.
            for (; kg < armed; ++kg) {
                const int s = (int)(kg % kStages);
                tma_load_2d(sA + s * kStageA, &tmS, &sh->full[s], 0, 0);
            }
            for (int64_t k = kg > kStages ? kg - kStages : 0; k < kg; ++k)
                mbar_wait_bounded(&sh->full[k % kStages], (uint32_t)(k / kStages) & 1u, kWaitNs);
        }
    } else if (warp == 1) {
        // MMA issuer: 4 K-steps of 32 bytes per stage.
        if (lane == 0) {
            int64_t kg = 0;
            bool ok = true;
            for (int64_t t = t0; t < t_end && ok; ++t) {
                for (int kb = 0; kb < KB; ++kb, ++kg) {
                    const int s = (int)(kg % kStages);
                    if (*tout || !mbar_wait_bounded(&sh->full[s], (uint32_t)(kg / kStages) & 1u, kWaitNs)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint64_t ad = smem_desc_sw128(smem_u32(sA + s * kStageA));
                    const uint64_t bd = smem_desc_sw128(smem_u32(sB + s * T::kStageB));
#pragma unroll
                    for (int k = 0; k < kBKB / 32; ++k) {
                        if constexpr (OP == kOpE4M3) mma_e4m3(tmem, ad + 2 * k, bd + 2 * k, IDESC, (kb | k) != 0);
                        else mma_bf16(tmem, ad + 2 * k, bd + 2 * k, IDESC, (kb | k) != 0);
                    }
                    mma_commit(&sh->empty[s]);
                }
                if (ok) mma_commit(&sh->accf);
            }
            if (!ok) *tout = 1;
            mma_commit(&sh->drain);
            mbar_wait_bounded(&sh->drain, 0, kWaitNs);
        }
    } else if (warp < 2 + kEpiWarps) {
        // Epilogue warps: warp w reads TMEM lane quadrant w % 4 (32 replicas, one per lane) and
        // column group (w - 2) / 4 (half of the tile's spins, in chunks of 16).
        const int q4 = warp & 3;
        const int cg = (warp - 2) >> 2;
        const size_t gs = (size_t)L.Rpad * 4;              // floats between groups of 4 spins
        const int i_base = m * BN + cg * kColsPerWarp;     // this warp's first spin
        const int r = n * kBM + q4 * 32 + lane;            // this thread's replica
        // its first 4 values of chunk c; chunks past N stay out
        auto xv_offset = [&](int c) -> size_t { return ((size_t)((i_base >> 2) + 4 * c) * L.Rpad + r) * 4; };
        const int nch = min(T::kChunks, max(0, (N - i_base + kChunk - 1) / kChunk));
        struct Chunk {
            float x[kChunk], v[kChunk];
        };
        Chunk st[T::kChunks];
#pragma unroll
        for (int c = 0; c < T::kChunks; ++c) {
            if (c >= nch) break;
            const size_t off = xv_offset(c);
#pragma unroll
            for (int k = 0; k < kChunk / 4; ++k) {
                const float4 x4 = __ldcg(reinterpret_cast<const float4 *>(L.X + off + k * gs));
                const float4 v4 = __ldcg(reinterpret_cast<const float4 *>(L.V + off + k * gs));
                st[c].x[4 * k] = x4.x; st[c].x[4 * k + 1] = x4.y; st[c].x[4 * k + 2] = x4.z; st[c].x[4 * k + 3] = x4.w;
                st[c].v[4 * k] = v4.x; st[c].v[4 * k + 1] = v4.y; st[c].v[4 * k + 2] = v4.z; st[c].v[4 * k + 3] = v4.w;
            }
        }
        const float inv_tm1 = inv_tm1_of(a.T_total), eps = a.eps, gamma = a.gamma;
        const uint32_t tbase = tmem + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(cg * kColsPerWarp);
        bool ok = true;
        for (int64_t t = t0; t < t_end && ok; ++t) {
            const float bgq = beta_at(t, inv_tm1, a.beta0, a.beta1) * (gamma * a.q), bgq4 = 4.0f * bgq;
            const bool more = t + 1 < t_call_end;
            const bool refresh_next = more && refresh_at(t + 1, a.refresh);
            uint8_t *srow = L.S + ((size_t)((t + 1) & 3) * L.Rpad + r) * L.Kbytes + (size_t)i_base * ESZ;
            uint16_t *bword = reinterpret_cast<uint16_t *>(L.sbits + (size_t)((t + 1) & 3) * (L.Mp / 32) * L.Rpad + r);
            // The spins of t + 1 overwrite those of t - 3: their best copy must be done.
            if (more && t - 3 >= t0) {
                const uint64_t ts = globaltimer_ns();
                while (*rec_copied < t - 3) {
                    if (*tout || globaltimer_ns() - ts > kWaitNs) {
                        ok = false;
                        break;
                    }
                    __nanosleep(64);
                }
            }
            // Warp-uniform, as the TMEM loads below are warp-collective.
            ok = __all_sync(0xffffffffu, ok && !*tout && mbar_wait_bounded(&sh->accf, (uint32_t)(t - t0) & 1u, kWaitNs));
            if (!ok) {
                *tout = 1;
                break;
            }
            tc_fence_after();
            int32_t esum = 0;
#pragma unroll
            for (int c = 0; c < T::kChunks; ++c) {
                if (c >= nch) break;
                Chunk &cur = st[c];
                uint32_t acc[kChunk];
                tmem_ld_x16_issue(tbase + c * kChunk, acc);
                const int i0 = i_base + c * kChunk;
                float h[kChunk], f[kChunk];
#pragma unroll
                for (int k = 0; k < kChunk / 4; ++k) {
                    const float4 h4 = *reinterpret_cast<const float4 *>(&sh->h[cg * kColsPerWarp + c * kChunk + 4 * k]);
                    h[4 * k] = h4.x; h[4 * k + 1] = h4.y; h[4 * k + 2] = h4.z; h[4 * k + 3] = h4.w;
                }
                if (a.deriv == 1) {
#pragma unroll
                    for (int j = 0; j < kChunk; ++j) f[j] = factor_quad(cur.x[j], bgq, gamma);
                } else {
#pragma unroll
                    for (int j = 0; j < kChunk; ++j) f[j] = factor_exact(cur.x[j], bgq4, gamma);
                }
                tmem_ld_wait_x16(acc);
                // Field I = J s + h (Eq. 6): acc and h are exact integers, their FP32 sum rounds the
                // exact field.  Energy terms s (I + h) (Eq. 2 through Eq. 6) of the replica: where a
                // chunk's add up exactly in FP32 (the tile's max |h|, max |k| and N say so) they are
                // converted once, otherwise each by itself.  Spins past N have zero couplings, h = 0
                // and x = v = 0.
                float I[kChunk];
                if (exact_sums) {
                    float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
                    for (int j = 0; j < kChunk; ++j) {
                        I[j] = __fadd_rn(__uint_as_float(acc[j]), h[j]);
                        const float e = __fadd_rn(I[j], h[j]);
                        float &s = j & 1 ? s1 : s0;
                        s = __fadd_rn(s, cur.x[j] >= 0.0f ? e : -e);
                    }
                    esum += __float2int_rn(__fadd_rn(s0, s1));
                } else {
                    long long es = 0;
#pragma unroll
                    for (int j = 0; j < kChunk; ++j) {
                        I[j] = __fadd_rn(__uint_as_float(acc[j]), h[j]);
                        const int32_t e = __float2int_rn(__uint_as_float(acc[j])) + 2 * __float2int_rn(h[j]);
                        es += cur.x[j] >= 0.0f ? e : -e;
                    }
                    atomicAdd(reinterpret_cast<unsigned long long *>(L.Epart) + (size_t)(t & 1) * L.Rpad + r,
                              (unsigned long long)es);
                }
#pragma unroll
                for (int j = 0; j < kChunk; ++j) cur.v[j] = momentum_of(cur.v[j], cur.x[j], I[j], f[j], eps);
                if (refresh_next) {
                    float w[kChunk];
                    refresh_chunk(w, a.seed, a.inst, (uint32_t)r, (uint32_t)i0, (uint32_t)(t + 1));
#pragma unroll
                    for (int j = 0; j < kChunk; ++j) cur.v[j] = w[j];
                }
                if (more) {
                    uint32_t plus = 0;
#pragma unroll
                    for (int j = 0; j < kChunk; ++j) {
                        cur.x[j] = __fmaf_rn(eps, cur.v[j], cur.x[j]);
                        if (cur.x[j] >= 0.0f) plus |= 1u << j;
                    }
                    bword[(size_t)(i0 >> 5) * L.Rpad * 2 + ((i0 >> 4) & 1)] = (uint16_t)plus;
                    uint4 *d4 = reinterpret_cast<uint4 *>(srow + c * kChunk * ESZ);
                    if constexpr (OP == kOpE4M3) {
                        d4[0] = make_uint4(spins4_e4m3(plus, 0), spins4_e4m3(plus, 4), spins4_e4m3(plus, 8),
                                           spins4_e4m3(plus, 12));
                    } else {
                        d4[0] = make_uint4(spins2_bf16_bits(plus, 0), spins2_bf16_bits(plus, 2), spins2_bf16_bits(plus, 4),
                                           spins2_bf16_bits(plus, 6));
                        d4[1] = make_uint4(spins2_bf16_bits(plus, 8), spins2_bf16_bits(plus, 10),
                                           spins2_bf16_bits(plus, 12), spins2_bf16_bits(plus, 14));
                    }
                }
            }
            if (esum != 0)
                atomicAdd(reinterpret_cast<unsigned long long *>(L.Epart) + (size_t)(t & 1) * L.Rpad + r,
                          (unsigned long long)(long long)esum);
            // The tile is done: the signal warp publishes it (its arrival on tiledone carries
            // this warp's stores).
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sh->tiledone);
        }
#pragma unroll
        for (int c = 0; c < T::kChunks; ++c) {
            if (c >= nch || !ok) break;
            const size_t off = xv_offset(c);
#pragma unroll
            for (int k = 0; k < kChunk / 4; ++k) {
                __stcg(reinterpret_cast<float4 *>(L.X + off + k * gs),
                       make_float4(st[c].x[4 * k], st[c].x[4 * k + 1], st[c].x[4 * k + 2], st[c].x[4 * k + 3]));
                __stcg(reinterpret_cast<float4 *>(L.V + off + k * gs),
                       make_float4(st[c].v[4 * k], st[c].v[4 * k + 1], st[c].v[4 * k + 2], st[c].v[4 * k + 3]));
            }
        }
    } else if (warp == 2 + kEpiWarps) {
        // Records warp.
        for (int64_t t = t0; t < t_end && !*tout; ++t) {
            bool ok = true;
            if (m == 0) {
                ok = wait_counter_at_least(ready + n, (uint32_t)(mt * (t - t0 + 1)), kWaitNs, tout);
                ok = __all_sync(0xffffffffu, ok);
                if (ok) settle_lane<kBM / 32>(L, n * kBM + lane, t);
                __syncwarp();
                if (lane == 0 && ok) {
                    __threadfence();
                    st_release_gpu(settled + n, (uint32_t)(t - t0 + 1));
                }
                __syncwarp();
            }
            if (lane == 0) *rec_settled = t;
            ok = ok && wait_counter_at_least(settled + n, (uint32_t)(t - t0 + 1), kWaitNs, tout);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) {
                *tout = 1;
                break;
            }
            copy_best<BN>(L, n, m * BN, t, lane);
            __syncwarp();
            if (lane == 0) *rec_copied = t;
        }
    } else if (lane == 0) {
        // Signal warp: once the epilogue warps finished an iteration, make their spins and energy
        // terms visible to the GPU and count the tile in ready[n].
        for (int64_t t = t0; t < t_end; ++t) {
            bool go = !*tout && mbar_wait_bounded(&sh->tiledone, (uint32_t)(t - t0) & 1u, kWaitNs);
            if (go && m == 0 && t - 1 >= t0) {
                const uint64_t ts = globaltimer_ns();
                while (*rec_settled < t - 1) {
                    if (*tout || globaltimer_ns() - ts > kWaitNs) {
                        go = false;
                        break;
                    }
                    __nanosleep(32);
                }
            }
            if (!go) {
                *tout = 1;
                break;
            }
            __threadfence();
            atomicAdd(ready + n, 1u);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && sh->timed_out) atomicExch(a.err, 1);
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tmem, T::kTmemCols);
    }
}

// Initial state (or given), refresh at t0, first position update, spins of iteration t0.  A
// block takes 32 replicas x 64 spins: a given state is read along its rows and turned in
// shared memory, so that both sides move in whole sectors.
constexpr int kConvR = 32, kConvN = 64;

template <int OP>
__global__ void __launch_bounds__(256) narrow_prologue(const NarrowArgs L) {
    __shared__ float sx[kConvR][kConvN + 1], sv[kConvR][kConvN + 1];
    __shared__ uint32_t sw[kConvN / 32][kConvR];
    const RunArgs &a = L.a;
    const int nx = (L.Mp + kConvN - 1) / kConvN;
    const int r0 = (int)(blockIdx.x / nx) * kConvR, i0 = (int)(blockIdx.x % nx) * kConvN;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (warp < kConvN / 32) sw[warp][lane] = 0u;
    if (a.x_in) {
        for (int e = threadIdx.x; e < kConvR * kConvN; e += 256) {
            const int rr = e / kConvN, ii = e % kConvN;
            const bool live = r0 + rr < a.R && i0 + ii < a.N;
            const size_t src = (size_t)(r0 + rr) * a.N + i0 + ii;
            sx[rr][ii] = live ? a.x_in[src] : 0.0f;
            sv[rr][ii] = live ? a.v_in[src] : 0.0f;
        }
    }
    __syncthreads();
    const int r = r0 + lane;
    for (int gq = warp; gq < kConvN / 4; gq += 8) {        // a group of 4 spins of one replica
        const int i4 = i0 + gq * 4;
        if (i4 >= L.Mp) break;
        float x[4], v[4];
        uint32_t plus = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int i = i4 + k;
            x[k] = v[k] = 0.0f;
            if (r < a.R && i < a.N) {
                if (a.x_in) {
                    x[k] = sx[lane][gq * 4 + k];
                    v[k] = sv[lane][gq * 4 + k];
                } else {
                    const U4 o = draw_raw(a.seed, a.inst, (uint32_t)r, (uint32_t)i, 0u);
                    x[k] = box_muller(o.x, o.y);
                    v[k] = box_muller(o.z, o.w);
                }
                if (refresh_at(a.t0, a.refresh)) v[k] = draw_v(a.seed, a.inst, (uint32_t)r, (uint32_t)i, (uint32_t)a.t0);
                x[k] = x[k] + a.eps * v[k];
            }
            if (x[k] >= 0.0f) plus |= 1u << k;
        }
        const size_t off = ((size_t)(i4 >> 2) * L.Rpad + r) * 4;
        *reinterpret_cast<float4 *>(L.X + off) = make_float4(x[0], x[1], x[2], x[3]);
        *reinterpret_cast<float4 *>(L.V + off) = make_float4(v[0], v[1], v[2], v[3]);
        atomicOr(&sw[gq >> 3][lane], plus << (4 * (gq & 7)));
        if (r < a.R && i4 < a.N) {
            uint8_t *row = L.S + ((size_t)(a.t0 & 3) * L.Rpad + r) * L.Kbytes;
            if constexpr (OP == kOpE4M3) {
                *reinterpret_cast<uint32_t *>(row + i4) = spins4_e4m3(plus, 0);
            } else {
                *reinterpret_cast<uint2 *>(row + 2 * i4) = make_uint2(spins2_bf16_bits(plus, 0), spins2_bf16_bits(plus, 2));
            }
        }
    }
    __syncthreads();
    if (warp < kConvN / 32 && i0 + warp * 32 < L.Mp)
        L.sbits[((size_t)(a.t0 & 3) * (L.Mp / 32) + (i0 >> 5) + warp) * L.Rpad + r0 + lane] = sw[warp][lane];
}

// Final state back to the caller's [R][N] arrays.
__global__ void __launch_bounds__(256) narrow_export(const NarrowArgs L) {
    __shared__ float sx[kConvR][kConvN + 1], sv[kConvR][kConvN + 1];
    const RunArgs &a = L.a;
    const int nx = (L.Mp + kConvN - 1) / kConvN;
    const int r0 = (int)(blockIdx.x / nx) * kConvR, i0 = (int)(blockIdx.x % nx) * kConvN;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int gq = warp; gq < kConvN / 4; gq += 8) {
        const int i4 = i0 + gq * 4;
        if (i4 >= L.Mp) break;
        const size_t off = ((size_t)(i4 >> 2) * L.Rpad + r0 + lane) * 4;
        const float4 x = *reinterpret_cast<const float4 *>(L.X + off), v = *reinterpret_cast<const float4 *>(L.V + off);
        const float xa[4] = {x.x, x.y, x.z, x.w}, va[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            sx[lane][gq * 4 + k] = xa[k];
            sv[lane][gq * 4 + k] = va[k];
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kConvR * kConvN; e += 256) {
        const int rr = e / kConvN, ii = e % kConvN;
        if (r0 + rr >= a.R || i0 + ii >= a.N) continue;
        const size_t dst = (size_t)(r0 + rr) * a.N + i0 + ii;
        if (a.x_out) a.x_out[dst] = sx[rr][ii];
        if (a.v_out) a.v_out[dst] = sv[rr][ii];
    }
}

__global__ void narrow_count(unsigned long long *iters, unsigned long long n) {
    if (threadIdx.x == 0 && blockIdx.x == 0) atomicAdd(iters, n);
}

// The whole run in cooperative launches of tc_narrow_run (all CTAs resident at once, as CTAs
// wait on each other's tiles).  Runs whose tile counters could pass 2^31 go out in several
// launches; every launch settles and copies all of its iterations.
template <int OP, int BN>
cudaError_t run_narrow(const LargeBuffers &B, const RunArgs &a, cudaStream_t st, int *launches, int sms) {
    constexpr size_t kSmem = NarrowTile<BN>::kSmemBytes;
    NarrowArgs L;
    memset(&L, 0, sizeof L);
    L.a = a;
    L.S = B.S;
    L.Epart = B.Epart;
    L.flags = B.flags;
    L.X = B.X;
    L.V = B.V;
    L.Kbytes = B.Kbytes;
    L.Rpad = B.Rpad;
    L.Mp = B.Mpad;
    L.mtiles = (a.N + BN - 1) / BN;
    L.rtiles = (a.R + kBM - 1) / kBM;
    L.ready = B.ready;
    L.sbits = B.sbits;
    CUtensorMap tmS, tmJ;
    const int esz = OP == kOpE4M3 ? 1 : 2;
    if (!tc_operand_map(&tmJ, B.Jop, OP, (uint64_t)B.Kbytes / esz, (uint64_t)B.Mpad, (uint64_t)B.Kbytes, BN) ||
        !tc_operand_map(&tmS, B.S, OP, (uint64_t)B.Kbytes / esz, (uint64_t)4 * B.Rpad, (uint64_t)B.Kbytes, kBM))
        return cudaErrorInvalidValue;
    auto k = tc_narrow_run<OP, BN>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
    if (e != cudaSuccess) return e;
    int resident = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&resident, k, kThreads, kSmem);
    if (e != cudaSuccess) return e;
    if (L.mtiles * L.rtiles > resident * sms) return cudaErrorCooperativeLaunchTooLarge;   // a tile per CTA
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(L.mtiles * L.rtiles));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    e = cudaMemsetAsync(B.Epart, 0, 2 * (size_t)B.Rpad * sizeof(int64_t), st);   // energy sums start at 0
    if (e != cudaSuccess) return e;
    int n = 0;
    const unsigned conv = (unsigned)((B.Mpad + kConvN - 1) / kConvN) * (unsigned)(B.Rpad / kConvR);
    narrow_prologue<OP><<<conv, 256, 0, st>>>(L);
    ++n;
    const int64_t chunk = std::max<int64_t>(1, ((int64_t)1 << 31) / L.mtiles - 1);
    for (int64_t t = a.t0; t < a.t0 + a.nsteps; t += chunk) {
        NarrowArgs Lc = L;
        Lc.f0 = t;
        Lc.f1 = t + std::min(chunk, a.t0 + a.nsteps - t);
        Lc.a.x_in = Lc.a.v_in = nullptr;
        Lc.a.x_out = Lc.a.v_out = nullptr;
        e = cudaMemsetAsync(B.ready, 0, 2 * (size_t)L.rtiles * sizeof(uint32_t), st);
        if (e != cudaSuccess) return e;
        void *args[3] = {&tmS, &tmJ, &Lc};
        e = cudaLaunchKernelExC(&cfg, reinterpret_cast<const void *>(k), args);
        if (e != cudaSuccess) return e;
        ++n;
    }
    narrow_count<<<1, 32, 0, st>>>(a.replica_iters, (unsigned long long)((int64_t)a.R * a.nsteps));
    ++n;
    if (a.x_out || a.v_out) {
        narrow_export<<<conv, 256, 0, st>>>(L);
        ++n;
    }
    if (launches) *launches += n;
    return cudaGetLastError();
}

}  // namespace

double narrow_estimate(int N, int R, int Kbytes, int sms, int *width) {
    // One tile a CTA (x and v stay in registers): from a tile's spins to the next iteration's
    // first MMA 2 us (counter, copies, accumulator), the operands at 90 bytes per ns, an epilogue
    // of 0.5 us and 0.035 us per column (fitted to timings at N = 400 .. 3000).  With more tiles
    // than CTAs the wide tiles are the better split.
    double best = 1e30;
    for (int bn : {64, 32}) {
        if ((int64_t)((N + bn - 1) / bn) * ((R + kBM - 1) / kBM) > sms) continue;
        const double us = 0.5 + 0.035 * bn + 2.0 + (double)Kbytes * (kBM + bn) / 90000.0;
        if (us < best) {
            best = us;
            *width = bn;
        }
    }
    return best;
}

cudaError_t launch_tc_narrow(const LargeBuffers &B, const RunArgs &a, int op, int width, cudaStream_t st, int *launches,
                             int sms) {
    if (op == kOpE4M3)
        return width == 64 ? run_narrow<kOpE4M3, 64>(B, a, st, launches, sms) : run_narrow<kOpE4M3, 32>(B, a, st, launches, sms);
    return width == 64 ? run_narrow<kOpBF16, 64>(B, a, st, launches, sms) : run_narrow<kOpBF16, 32>(B, a, st, launches, sms);
}

}  // namespace phia
