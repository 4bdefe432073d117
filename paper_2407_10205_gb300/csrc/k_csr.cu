// k_csr.cu -- sparse PHIA path: many instances of uneven N, the field I = J s + h (Eq. 6)
// gathered from bit-packed spins with a row to a lane, fused with the update of Eqs. 5, 8 and
// A7; one launch per iteration, or one cooperative launch per run.
//
// Layout per instance b.  Rows (spins) are held in positions: sorted by their number of
// couplings, descending, so that the 32 rows of a slice have about equally many; Np = N
// rounded up to 32, positions past N are empty.  Replicas go in groups of 32.
//   spins     4 rotating buffers of uint32 [group][Np]: bit r of word p = (the spin at position
//             p of replica 32 group + r is +1); iteration t reads buffer t % 4, writes t+1 % 4
//   x, v      float32 [group][8][Np][4]: 4 replicas of one row sit together, so that a lane
//             moves them as one vector and a warp's vector covers 512 contiguous bytes
//   couplings per slice, for every 4 neighbours of its rows: 4 byte offsets of their positions in
//             a spin buffer (16 bits each while every Np <= 16384, else 32) and 4 x int8, one
//             entry per lane
//   best      uint32 [R][ceil(N/32)] bit-packed over spins in their own order
//
// A warp takes a slice (32 rows, one per lane) and a group of 32 replicas.  For 4 neighbours a
// lane reads 4 words (32 replicas each) from the block's shared-memory copy of the group's
// spins, turns them into 8-replica bytes (a 4 x 4 byte transpose) and adds, for each replica,
// (bytes & 2^b) . (4 couplings) with one 4-way dot product: acc_r = 2^b sum k [s = +1], b = r
// % 8.  With ksum the row's sum of couplings, I_r = 2 sum k [s = +1] - ksum + kh, exactly.
//
// What bounds it: the instructions of the gather (per 4 neighbours and 32 rows x 32 replicas
// 32 dot products, 32 masks, 8 byte permutes, 4 shared loads) and of the update, with the x, v
// stream (16 bytes per spin update) behind them.  The earlier form took a row to a warp and 8
// replicas to a lane: every neighbour cost the warp a load of 32 bytes, its address and its
// share of the byte permutes for 8 replicas a lane instead of 32.  Per iteration (us, 256 replicas),
// that form and this one: one Erdos-Renyi instance of 625 spins 20.9 / 7.0, of 1760 36.0 / 11.5, of
// 5000 27.1 / 10.5, where latencies in a row set the time; 12 instances of 100 .. 3000 spins
// 56.9 / 31.1, 48 of them 180 / 113, 256 of them 654 / 521.  For large instances of few couplings a
// row that form is the faster one and stays (k_csr_rows.cu).
//
// The instances go through their iterations in sets whose state fits in L2 together: a set runs
// all of its iterations before the next begins (the instances are independent), so x and v are
// read from L2 instead of the memory they would fall out to between two iterations of a batch
// (measured before x and v were staged in shared memory: 48 instances 117 us an iteration against
// 135 in one set, 256 of them 636 against 653).
//
// Records are lagged: the launch for iteration t settles t - 1 (the instance's last unit)
// and copies the best spins of t - 2 for the replicas that improved then.
#include <algorithm>
#include <type_traits>

#include "device_common.cuh"
#include "phia_internal.h"

namespace phia {

namespace {

constexpr int kWarps = 8;
constexpr int kBlk = 32 * kWarps;
constexpr size_t kTwo = 113 * 1024;            // shared memory of one of two blocks on an SM

// The word of position p and group g in a spin buffer: [group][Np], so that a group's spins are
// copied as one piece, or (C.by_pos) [Np][group], so that a neighbour's groups share a sector.
__device__ __forceinline__ size_t spin_word(const CsrArgs &C, const CsrInst &in, int g, int p) {
    return C.by_pos ? (size_t)p * (C.R / 32) + g : (size_t)g * in.Np + p;
}

__device__ __forceinline__ void settle_csr(const CsrArgs &C, const CsrInst &in, int b, int r, int64_t tt) {
    const RunArgs &a = C.a;
    const size_t rec = (size_t)in.rec_off + r;
    unsigned long long *slot =
        reinterpret_cast<unsigned long long *>(C.Esum) + (size_t)(tt & 1) * C.total_reps + rec;
    const long long twice = (long long)__ldcg(slot);
    *slot = 0ull;
    const long long E = -twice / 2;
    int imp = 0;
    const long long best = (long long)__ldcg(a.best_e + rec), hit = (long long)__ldcg(a.hit_step + rec);
    const bool frozen = a.stop_at_target && hit >= 0;
    if (!frozen && E < best) {
        a.best_e[rec] = E;
        a.best_step[rec] = tt;
        imp = 1;
    }
    const long long target = C.targets ? C.targets[b] : a.target;
    if (a.has_target && hit < 0 && E <= target) {
        a.hit_step[rec] = tt;
        if (a.hit_ns) a.hit_ns[rec] = globaltimer_ns();
    }
    C.flags[(size_t)(tt & 1) * C.total_reps + rec] = (int8_t)imp;
}

__device__ __forceinline__ uint32_t *spin_buf(const CsrArgs &C, const CsrInst &in, int64_t tt) {
    return C.S + (size_t)(tt & 3) * C.total_swords + in.s_off;
}

// Best spins of iteration tt for the replicas of group g that improved then: the words w0, w0 +
// step, .. of the best state.  A lane has the 32 replicas of one spin; transposed, the 32 spins of
// its replica, which are a word of that one's state.  Early in a run nearly every replica improves in
// every iteration: with a vote and a one-lane store per replica and word instead, 6000 spins x 256
// replicas took 13.6 us an iteration against 11.6 here (degree 60), 10000 x 256 18.9 against 14.5
// (degree 6), 20000 x 1024 117 against 101 (degree 20).
__device__ __forceinline__ void copy_best(const CsrArgs &C, const CsrInst &in, int g, int64_t tt, int w0, int step, int w_end) {
    const int lane = threadIdx.x & 31;
    const bool imp = __ldcg(C.flags + (size_t)(tt & 1) * C.total_reps + in.rec_off + g * 32 + lane) != 0;
    if (!__any_sync(0xffffffffu, imp)) return;
    const uint32_t *Sb = spin_buf(C, in, tt);
    const int W = (in.N + 31) / 32;
    for (int w = w0; w < w_end; w += step) {
        const int i = w * 32 + lane;
        uint32_t word = i < in.N ? __ldcg(Sb + spin_word(C, in, g, C.pos_of[in.inv_off + i])) : 0u;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) {
            const uint32_t m = d == 16 ? 0x0000ffffu : d == 8 ? 0x00ff00ffu : d == 4 ? 0x0f0f0f0fu : d == 2 ? 0x33333333u : 0x55555555u;
            const uint32_t other = __shfl_xor_sync(0xffffffffu, word, d);
            word = lane & d ? (word & ~m) | ((other >> d) & m) : (word & m) | ((other << d) & ~m);
        }
        if (imp) C.best_bits[in.bits_off + (size_t)(g * 32 + lane) * W + w] = word;
    }
}

// 4 x 4 byte transpose: byte b of word k of the result is byte k of word b of the input, i.e.
// word k holds the four neighbours' bytes of replicas 8k .. 8k + 7.
__device__ __forceinline__ void transpose4(const uint32_t (&w)[4], uint32_t (&B)[4]) {
    const uint32_t a = __byte_perm(w[0], w[1], 0x5140), b = __byte_perm(w[2], w[3], 0x5140);
    const uint32_t c = __byte_perm(w[0], w[1], 0x7362), d = __byte_perm(w[2], w[3], 0x7362);
    B[0] = __byte_perm(a, b, 0x5410);
    B[1] = __byte_perm(a, b, 0x7632);
    B[2] = __byte_perm(c, d, 0x5410);
    B[3] = __byte_perm(c, d, 0x7632);
}

// d + sum over 4 bytes of (unsigned byte of a) x (signed byte of b).
__device__ __forceinline__ int32_t dp4a_us(uint32_t a, uint32_t b, int32_t d) {
    asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(d) : "r"(a), "r"(b));
    return d;
}

// One entry of a lane's row: the byte offsets of 4 neighbours' spin words (16 or 32 bits each)
// and their couplings.
template <bool C16>
struct Entry {
    uint2 c;
    uint32_t k;
    __device__ __forceinline__ void load(const CsrArgs &C, int e, int lane) {
        c = __ldg(reinterpret_cast<const uint2 *>(C.col) + (size_t)e * 32 + lane);
        k = __ldg(C.val + (size_t)e * 32 + lane);
    }
    __device__ __forceinline__ uint32_t at(int n) const { return n & 1 ? (n & 2 ? c.y : c.x) >> 16 : (n & 2 ? c.y : c.x) & 0xffffu; }
};
template <>
struct Entry<false> {
    uint4 c;
    uint32_t k;
    __device__ __forceinline__ void load(const CsrArgs &C, int e, int lane) {
        c = __ldg(reinterpret_cast<const uint4 *>(C.col) + (size_t)e * 32 + lane);
        k = __ldg(C.val + (size_t)e * 32 + lane);
    }
    __device__ __forceinline__ uint32_t at(int n) const { return n == 0 ? c.x : n == 1 ? c.y : n == 2 ? c.z : c.w; }
};

// A lane's first entries of a slice: as many as gather_row keeps in flight.
template <bool C16>
struct Ahead {
    static constexpr int D = C16 ? 3 : 1;
    Entry<C16> nx[D];
    __device__ __forceinline__ void load(const CsrArgs &C, int e, int e_end, int lane) {
#pragma unroll
        for (int u = 0; u < D; ++u)
            if (e + u < e_end) nx[u].load(C, e + u, lane);
    }
};

// 4 neighbours of a lane's row: acc[r] += sum k [s = +1] over them.  SCALED: acc_r carries the
// factor 2^(r % 8) of its bit's place (one instruction less per replica); rows of over 2^16
// couplings take the bit down to place 0 instead, as the factor could leave 32 bits.
template <bool SCALED>
__device__ __forceinline__ void add_neighbours(const uint32_t (&w)[4], uint32_t k, int32_t (&acc)[32]) {
    uint32_t B[4];
    transpose4(w, B);
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const int bit = r & 7;
        if constexpr (SCALED) acc[r] = dp4a_us(B[r >> 3] & (0x01010101u << bit), k, acc[r]);
        else acc[r] = dp4a_us((B[r >> 3] >> bit) & 0x01010101u, k, acc[r]);
    }
}

// acc[r] of the lane's row over its couplings: entries [e, e_end) of the slice, 4 neighbours
// each; the next entries load meanwhile (three ahead with 16-bit offsets, whose registers allow
// it: an entry's L2 latency is several times its arithmetic).  Spins in shared memory.
template <bool C16, bool SCALED>
__device__ __forceinline__ void gather_smem(const CsrArgs &C, const char *spins, int e, int e_end, int lane,
                                            Ahead<C16> &ahead, int32_t (&acc)[32]) {
    constexpr int D = Ahead<C16>::D;
    Entry<C16>(&nx)[D] = ahead.nx;
#pragma unroll 1
    for (; e < e_end; e += D) {
#pragma unroll
        for (int u = 0; u < D; ++u) {
            if (u > 0 && e + u >= e_end) break;
            const Entry<C16> en = nx[u];
            if (e + u + D < e_end) nx[u].load(C, e + u + D, lane);
            uint32_t w[4];
#pragma unroll
            for (int n = 0; n < 4; ++n) w[n] = *reinterpret_cast<const uint32_t *>(spins + en.at(n));
            add_neighbours<SCALED>(w, en.k, acc);
        }
    }
}

// The same from global memory, spins by position (`groups` words each): the block's warps take
// the groups of a slice side by side, so that one of them brings a neighbour's sector to L1.  The
// next entry's words load while this one's are added.
// CACHED: through L1, which a launch finds empty; iterations within one launch read L2.
template <bool C16, bool SCALED, bool CACHED>
__device__ __forceinline__ void gather_global(const CsrArgs &C, const char *spins, uint32_t groups, int e, int e_end,
                                              int lane, Ahead<C16> &ahead, int32_t (&acc)[32]) {
    Entry<C16> nx = ahead.nx[0];
    uint32_t w[4] = {0u, 0u, 0u, 0u}, k = nx.k;
    auto words = [&]() {
#pragma unroll
        for (int n = 0; n < 4; ++n) {
            const uint32_t *p = reinterpret_cast<const uint32_t *>(spins + (size_t)nx.at(n) * groups);
            w[n] = CACHED ? *p : __ldcg(p);
        }
    };
    if (e < e_end) words();
    if (e + 1 < e_end) nx.load(C, e + 1, lane);
#pragma unroll 1
    for (; e < e_end; ++e) {
        const uint32_t c[4] = {w[0], w[1], w[2], w[3]}, ck = k;
        if (e + 1 < e_end) {
            words();
            k = nx.k;
            if (e + 2 < e_end) nx.load(C, e + 2, lane);
        }
        add_neighbours<SCALED>(c, ck, acc);
    }
}

// A block of a step launch with its place in the count of blocks that have read the iteration:
// the last one, whose count says that all have, advances it for the next launch.
__device__ __forceinline__ void step_done(IterCtl *c, unsigned ticket) {
    if (ticket != gridDim.x * gridDim.y - 1) return;
    c->done = 0;
    c->t = __ldcg(&c->t) + 1;
}

// Sums over a warp's rows of 8 replicas' terms: replica lane % 8 in every lane.  Three halving
// exchanges, then two whole ones (8 warp sums would take 8 cycles each).
__device__ __forceinline__ int32_t sum_rows8(const int32_t (&e)[8], int lane) {
    const bool h4 = lane & 4, h2 = lane & 2, h1 = lane & 1;
    int32_t a[4], b[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = (h4 ? e[4 + k] : e[k]) + __shfl_xor_sync(0xffffffffu, h4 ? e[k] : e[4 + k], 4);
#pragma unroll
    for (int k = 0; k < 2; ++k) b[k] = (h2 ? a[2 + k] : a[k]) + __shfl_xor_sync(0xffffffffu, h2 ? a[k] : a[2 + k], 2);
    int32_t s = (h1 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h1 ? b[0] : b[1], 1);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s;
}

// Momentum draws d = t1 of replicas r0 .. r0 + 7 of a spin (out of line: once per trajectory).
__device__ __noinline__ void refresh8(float *v, uint64_t seed, uint32_t inst, uint32_t r0, uint32_t i, uint32_t t1) {
#pragma unroll 1
    for (int k = 0; k < 8; ++k) v[k] = draw_v(seed, inst, r0 + k, i, t1);
}

// One work unit of iteration t: C.slices slices of an instance (block `bi` of the list) x
// C.gblock groups of 32 replicas (the y-th such set).  Uses the block's shared memory; every
// thread of the block calls it.  STEP: the unit of a step launch, which may start before the
// launch for t - 1 has ended: what no iteration changes (the block, its instance, the first
// entries) loads first, then it waits for that launch and reads its iteration.  SMEM: the spins are
// gathered from shared memory; STAGED: x and v of a slice pass through it.
template <bool SMEM, bool C16, bool STAGED, bool STEP>
__device__ __forceinline__ void csr_unit(const CsrArgs &C, int bi, int y, int64_t t, int64_t t_first, int64_t t_end,
                                         char *smem) {
    const RunArgs &a = C.a;
    const CsrBlock blk = C.blocks[bi];
    const CsrInst in = C.inst[blk.inst];
    const int b = blk.inst;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int G = C.gblock, groups = C.R / 32;
    const int gi = warp % G, sp = warp / G, spar = kWarps / G;     // group and slice lane of this warp
    const int g = y * G + gi;
    const bool active = g < groups;
    const int nsl = in.Np / 32;
    const int s_end = min(nsl, blk.s0 + C.slices);
    const int s_first = active ? blk.s0 + sp : s_end;              // this warp's first slice
    int e0 = 0, e1 = 0;
    Ahead<C16> ahead;
    if (s_first < s_end) {
        e0 = C.slice[in.slice_off + s_first];
        e1 = C.slice[in.slice_off + s_first + 1];
        ahead.load(C, e0, e1, lane);
    }
    if constexpr (STEP) {
        t_first = __ldcg(&C.ctl->t_first);
        t_end = __ldcg(&C.ctl->t_end);
        grid_dependency_wait();
        t = __ldcg(&C.ctl->t);
    }

    // The spins of this iteration of the block's groups into shared memory.
    const uint32_t *Sg = spin_buf(C, in, t);
    if constexpr (SMEM) {
        const int words = min(G, groups - y * G) * in.Np;          // consecutive in the buffer
        const uint32_t *src = Sg + (size_t)y * G * in.Np;
        for (int e = tid * 4; e < words; e += kBlk * 4) cp_async_16(smem + (size_t)e * 4, src + e);
        cp_async_commit();
    }
    // x and v of a slice load while the gather runs: all of it into the warp's part of shared memory
    // (a lane's own values, which nobody else reads), or the first 8 replicas into registers and
    // the others 8 replicas ahead of their use, which then waits for L2.
    const size_t qs = (size_t)in.Np * 4;               // floats between quads of replicas
    float4 *const stage = reinterpret_cast<float4 *>(smem + C.stage_off) + warp * (16 * 32) + lane;
    float4 xq[2], vq[2];
    auto fetch_state = [&](int s) {
        const size_t o = in.x_off + ((size_t)g * 8 * in.Np + s * 32 + lane) * 4;
        if constexpr (STAGED) {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                cp_async_16(stage + 64 * k, C.X + o + k * qs);
                cp_async_16(stage + 64 * k + 32, C.V + o + k * qs);
            }
        } else {
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                xq[k] = __ldcg(reinterpret_cast<const float4 *>(C.X + o + k * qs));
                vq[k] = __ldcg(reinterpret_cast<const float4 *>(C.V + o + k * qs));
            }
        }
    };
    if (s_first < s_end) fetch_state(s_first);
    if constexpr (STAGED) cp_async_commit();
    // (a) records of iteration t-1 (the last block of each instance, whose rows are the shortest).
    if (blk.s0 + C.slices >= nsl && t - 1 >= t_first) {
        for (int e = tid; e < G * 32; e += kBlk)
            if (y * G * 32 + e < C.R) settle_csr(C, in, b, y * G * 32 + e, t - 1);
    }
    // (b) best spins of iteration t-2: this block's share of the words of the best state.
    if (active && t - 2 >= t_first) copy_best(C, in, g, t - 2, blk.s0 + sp, spar, s_end);
    if constexpr (SMEM) cp_async_wait<STAGED ? 1 : 0>();
    if constexpr (SMEM || STEP) __syncthreads();
    unsigned ticket = 0;          // every thread of the block has read the iteration
    if constexpr (STEP)
        if (tid == 0) ticket = atomicAdd(&C.ctl->done, 1u);
    // (c) field and update.
    if (active) {
        const char *spins = SMEM ? smem + (size_t)gi * in.Np * 4 : reinterpret_cast<const char *>(Sg + g);
        uint32_t *Snext = spin_buf(C, in, t + 1);
        const float bgq = beta_at(t, inv_tm1_of(a.T_total), a.beta0, a.beta1) * (a.gamma * in.q);
        const float eps = a.eps, gamma = a.gamma, bgq4 = 4.0f * bgq;
        const bool more = t + 1 < t_end;
        const bool refresh_next = more && refresh_at(t + 1, a.refresh);
        long long esum = 0;                            // replica `lane` of the group
        for (int s = s_first; s < s_end; s += spar) {
            const int p = s * 32 + lane;
            float *X = C.X + in.x_off + ((size_t)g * 8 * in.Np + p) * 4;
            float *V = C.V + in.x_off + ((size_t)g * 8 * in.Np + p) * 4;
            if (s != s_first) {
                fetch_state(s);
                if constexpr (STAGED) cp_async_commit();
                e0 = C.slice[in.slice_off + s];
                e1 = C.slice[in.slice_off + s + 1];
                ahead.load(C, e0, e1, lane);
            }
            int32_t acc[32];
#pragma unroll
            for (int r = 0; r < 32; ++r) acc[r] = 0;
            if constexpr (SMEM) {
                if (in.wide) gather_smem<C16, false>(C, spins, e0, e1, lane, ahead, acc);
                else gather_smem<C16, true>(C, spins, e0, e1, lane, ahead, acc);
            } else {
                if (in.wide) gather_global<C16, false, STEP>(C, spins, groups, e0, e1, lane, ahead, acc);
                else gather_global<C16, true, STEP>(C, spins, groups, e0, e1, lane, ahead, acc);
            }
            const int2 hh = __ldg(reinterpret_cast<const int2 *>(C.hk) + in.pos_off + p);    // h, h - ksum
            const int row = refresh_next ? C.row_of[in.pos_off + p] : 0;
            uint32_t bits = 0;
            if constexpr (STAGED) cp_async_wait<0>();
            // 8 replicas at a time, their accumulators moved down to the front: one copy of the code
            // instead of four, as a straight line over all 32 replicas (with the draws of a refresh in it)
            // is fetched anew for every slice: its update took 8000 to 10000 cycles, most of them
            // waiting for instructions.
#pragma unroll 1
            for (int o = 0; o < 4; ++o) {
                float *Xo = X + 2 * o * qs, *Vo = V + 2 * o * qs;
                if constexpr (STAGED) {
                    const float4 *so = stage + 128 * o;
                    xq[0] = so[0];
                    vq[0] = so[32];
                    xq[1] = so[64];
                    vq[1] = so[96];
                }
                float xs[8] = {xq[0].x, xq[0].y, xq[0].z, xq[0].w, xq[1].x, xq[1].y, xq[1].z, xq[1].w}, If[8];
                float vn[8] = {vq[0].x, vq[0].y, vq[0].z, vq[0].w, vq[1].x, vq[1].y, vq[1].z, vq[1].w};
                if (!STAGED && o < 3) {
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        xq[k] = __ldcg(reinterpret_cast<const float4 *>(Xo + (2 + k) * qs));
                        vq[k] = __ldcg(reinterpret_cast<const float4 *>(Vo + (2 + k) * qs));
                    }
                }
                int32_t e8[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int32_t twice = (in.wide || k == 0) ? acc[k] << 1 : acc[k] >> (k - 1);
                    const int32_t I = twice + hh.y;                                   // Eq. 6, exact
                    const int32_t m = (int32_t)minus_mask(xs[k]);
                    e8[k] = ((I + hh.x) ^ m) - m;                                     // s (I + h)
                    If[k] = (float)I;
                }
                long long es;
                if (in.wide) {          // sums of such terms may leave 32 bits: halves apart
                    int32_t lo[8], hi[8];
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        lo[k] = e8[k] & 0xffff;
                        hi[k] = e8[k] >> 16;
                    }
                    es = (long long)sum_rows8(lo, lane) + ((long long)sum_rows8(hi, lane) << 16);
                } else {
                    es = sum_rows8(e8, lane);
                }
                if ((lane >> 3) == o) esum += es;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const float f = a.deriv == 1 ? factor_quad(xs[k], bgq, gamma) : factor_exact(xs[k], bgq4, gamma);
                    vn[k] = momentum_of(vn[k], xs[k], If[k], f, eps);
                }
                if (refresh_next && row >= 0) {
                    float w[8];
                    refresh8(w, a.seed, in.inst_id, (uint32_t)(g * 32 + 8 * o), (uint32_t)row, (uint32_t)(t + 1));
#pragma unroll
                    for (int k = 0; k < 8; ++k) vn[k] = w[k];
                }
                if (more) {
                    uint32_t plus = 0;
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        xs[k] = __fmaf_rn(eps, vn[k], xs[k]);
                        plus |= ~minus_mask(xs[k]) & (1u << k);
                    }
                    bits |= plus << (8 * o);
                    *reinterpret_cast<float4 *>(Xo) = make_float4(xs[0], xs[1], xs[2], xs[3]);
                    *reinterpret_cast<float4 *>(Xo + qs) = make_float4(xs[4], xs[5], xs[6], xs[7]);
                }
                *reinterpret_cast<float4 *>(Vo) = make_float4(vn[0], vn[1], vn[2], vn[3]);
                *reinterpret_cast<float4 *>(Vo + qs) = make_float4(vn[4], vn[5], vn[6], vn[7]);
#pragma unroll
                for (int r = 0; r < 24; ++r) acc[r] = acc[r + 8];
            }
            if (more) Snext[spin_word(C, in, g, p)] = bits;
        }
        atomicAdd(reinterpret_cast<unsigned long long *>(C.Esum) + (size_t)(t & 1) * C.total_reps + in.rec_off + g * 32 + lane,
                  (unsigned long long)esum);
    }
    if constexpr (SMEM && !STEP) __syncthreads();   // the shared spins are free for the next unit
    if constexpr (STEP)
        if (tid == 0) step_done(C.ctl, ticket);
}

// One launch per iteration of a set of instances: a block per work unit (the grid is that of
// the largest set); the iteration and the set come from C.ctl.  A launch lets the next one's
// blocks start as soon as its own have all started (they wait for its end before they read what
// it writes), so the boundary costs neither a launch nor the loads of what is the same in every
// iteration.
template <bool SMEM, bool C16, bool STAGED>
__global__ void __launch_bounds__(kBlk, 2) csr_step(const CsrArgs C) {
    extern __shared__ __align__(16) char smem[];
    grid_dependents_launch();
    const CsrSet set = C.sets[__ldcg(&C.ctl->set)];
    if ((int)blockIdx.x < set.len[C.list]) {
        csr_unit<SMEM, C16, STAGED, true>(C, set.off[C.list] + blockIdx.x, blockIdx.y, 0, 0, 0, smem);
    } else {
        grid_dependency_wait();
        if (threadIdx.x == 0) step_done(C.ctl, atomicAdd(&C.ctl->done, 1u));
    }
}

// Grid-wide barrier of a cooperative launch (every block resident): bar[0] counts the
// blocks arrived, bar[1] is the generation.  The wait is bounded; false when it expired.
__device__ bool grid_barrier(unsigned *bar, uint64_t timeout_ns) {
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        volatile unsigned *gen = bar + 1;
        const unsigned g0 = *gen;
        __threadfence();
        if (atomicAdd(bar, 1u) == gridDim.x - 1) {
            atomicExch(bar, 0u);
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            const uint64_t t_start = globaltimer_ns();
            while (*gen == g0) {
                if (globaltimer_ns() - t_start > timeout_ns) { ok = 0; break; }
                __nanosleep(64);
            }
        }
        __threadfence();
    }
    return __syncthreads_and(ok) != 0;
}

// All iterations of the run in one cooperative launch, set after set: per iteration every block
// takes work units from a counter (units of uneven cost balance themselves), then the grid
// meets at a barrier.  ctr[k & 1] hands out the units of the launch's k-th iteration; block 0
// clears it after that iteration's barrier, before it is used again.
template <bool SMEM, bool C16, bool STAGED>
__global__ void __launch_bounds__(kBlk, 2) csr_persistent(const CsrArgs C, unsigned *bar, unsigned *ctr) {
    extern __shared__ __align__(16) char smem[];
    __shared__ int unit;
    const int64_t t_first = C.a.t0, t_end = C.a.t0 + C.a.nsteps;
    const int ny = (C.R / 32 + C.gblock - 1) / C.gblock;
    int k = 0;
    for (int sidx = 0; sidx < C.nsets; ++sidx) {
        const CsrSet set = C.sets[sidx];
        const int nb = set.len[C.list], units = nb * ny;
        for (int64_t t = t_first; t < t_end; ++t, k ^= 1) {
            for (;;) {
                if (threadIdx.x == 0) unit = (int)atomicAdd(&ctr[k], 1u);
                __syncthreads();
                const int u = unit;
                __syncthreads();
                if (u >= units) break;
                csr_unit<SMEM, C16, STAGED, false>(C, set.off[C.list] + u % nb, u / nb, t, t_first, t_end, smem);
            }
            if (!grid_barrier(bar, kWaitTimeoutNs)) {
                if (threadIdx.x == 0) atomicExch(C.a.err, 1);
                return;
            }
            if (blockIdx.x == 0 && threadIdx.x == 0) ctr[k] = 0u;
        }
    }
}

// Iteration control back to the run's start, for the next set of instances.
__global__ void csr_next_set(IterCtl *ctl, int64_t t0, int64_t nsteps, int32_t set) {
    iter_ctl_start(ctl, t0, nsteps);
    ctl->set = set;
}

// The instance that holds global slice gs (slices are numbered instance after instance).
__device__ __forceinline__ int instance_of(const CsrArgs &C, int64_t gs) {
    int lo = 0, hi = C.count - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (C.inst[mid].slice_base <= gs) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Initial state (or given, [R][N] per instance), refresh at t0, first position update, spins
// of iteration t0.  A block per (slice, group): a warp per 4 replicas, a lane per row.
__global__ void __launch_bounds__(kBlk) csr_prologue(const CsrArgs C) {
    __shared__ uint32_t part[8][32];
    const RunArgs &a = C.a;
    const int groups = C.R / 32;
    const int64_t gs = blockIdx.x / groups;
    const int g = (int)(blockIdx.x % groups);
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        iter_ctl_start(C.ctl, a.t0, a.nsteps);
        C.ctl->set = 0;
    }
    const CsrInst in = C.inst[instance_of(C, gs)];
    const int qd = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = (int)(gs - in.slice_base) * 32 + lane;
    const int row = C.row_of[in.pos_off + p];
    float x[4] = {0.f, 0.f, 0.f, 0.f}, v[4] = {0.f, 0.f, 0.f, 0.f};
    uint32_t bits = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = g * 32 + qd * 4 + k;
        if (row >= 0) {
            if (C.x_in && r < C.R_real) {
                x[k] = C.x_in[in.xin_off + (size_t)r * in.N + row];
                v[k] = C.v_in[in.xin_off + (size_t)r * in.N + row];
            } else {
                const U4 o = draw_raw(a.seed, in.inst_id, (uint32_t)r, (uint32_t)row, 0u);
                x[k] = box_muller(o.x, o.y);
                v[k] = box_muller(o.z, o.w);
            }
            if (refresh_at(a.t0, a.refresh)) v[k] = draw_v(a.seed, in.inst_id, (uint32_t)r, (uint32_t)row, (uint32_t)a.t0);
            x[k] = x[k] + a.eps * v[k];
        }
        bits |= ~minus_mask(x[k]) & (1u << (qd * 4 + k));
    }
    const size_t off = in.x_off + ((size_t)(g * 8 + qd) * in.Np + p) * 4;
    *reinterpret_cast<float4 *>(C.X + off) = make_float4(x[0], x[1], x[2], x[3]);
    *reinterpret_cast<float4 *>(C.V + off) = make_float4(v[0], v[1], v[2], v[3]);
    part[qd][lane] = bits;
    __syncthreads();
    if (qd == 0) {
#pragma unroll
        for (int w = 1; w < 8; ++w) bits |= part[w][lane];
        spin_buf(C, in, a.t0)[spin_word(C, in, g, p)] = bits;
    }
}

// Final state back to [R][N] per instance (caller layout).
__global__ void __launch_bounds__(kBlk) csr_export(const CsrArgs C) {
    const int groups = C.R / 32;
    const int64_t gs = blockIdx.x / groups;
    const int g = (int)(blockIdx.x % groups);
    const CsrInst in = C.inst[instance_of(C, gs)];
    const int qd = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = (int)(gs - in.slice_base) * 32 + lane;
    const int row = C.row_of[in.pos_off + p];
    if (row < 0) return;
    const size_t off = in.x_off + ((size_t)(g * 8 + qd) * in.Np + p) * 4;
    const float4 x4 = *reinterpret_cast<const float4 *>(C.X + off), v4 = *reinterpret_cast<const float4 *>(C.V + off);
    const float x[4] = {x4.x, x4.y, x4.z, x4.w}, v[4] = {v4.x, v4.y, v4.z, v4.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int r = g * 32 + qd * 4 + k;
        if (r >= C.R_real) continue;
        C.x_out[in.xin_off + (size_t)r * in.N + row] = x[k];
        C.v_out[in.xin_off + (size_t)r * in.N + row] = v[k];
    }
}

__global__ void csr_settle_all(const CsrArgs C, int64_t tt) {
    const int b = blockIdx.x;
    const CsrInst in = C.inst[b];
    for (int r = threadIdx.x; r < C.R; r += blockDim.x) settle_csr(C, in, b, r, tt);
}

// Copies for iterations not handled by a later launch; a warp per (word of the best state, group).
__global__ void __launch_bounds__(kBlk) csr_copy_all(const CsrArgs C, int64_t t_from, int64_t t_last) {
    const CsrInst in = C.inst[blockIdx.y];
    const int W = (in.N + 31) / 32, groups = C.R / 32;
    const int64_t u = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (u >= (int64_t)W * groups) return;
    const int w = (int)(u / groups), g = (int)(u - (int64_t)w * groups);
    for (int64_t tt = t_from; tt <= t_last; ++tt) copy_best(C, in, g, tt, w, 1, w + 1);
}

// Field only: spins given as int8 [R][N] per instance -> field int32 [R][N], energy [R].
__global__ void csr_field_only(const CsrArgs C) {
    const RunArgs &a = C.a;
    const int64_t gidx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;   // over (slice, row, replica)
    const int R = C.R;
    const int64_t gp = gidx / R;
    if (gp >= C.total_slices * 32) return;
    const int r = (int)(gidx - gp * R);
    const CsrInst in = C.inst[instance_of(C, gp / 32)];
    const int p = (int)(gp - in.slice_base * 32), lane = p & 31;
    const int row = C.row_of[in.pos_off + p];
    if (row < 0 || r >= C.R_real) return;
    const int8_t *s = a.spins_in + in.xin_off + (size_t)r * in.N;
    const int32_t h = C.hk[2 * (in.pos_off + p)];
    int32_t I = h;
    for (int e = C.slice[in.slice_off + p / 32]; e < C.slice[in.slice_off + p / 32 + 1]; ++e) {
        Entry<true> e16;
        Entry<false> e32;
        if (C.col16) e16.load(C, e, lane);
        else e32.load(C, e, lane);
        const uint32_t kk = C.col16 ? e16.k : e32.k;
        // no look at the couplings first: the four ways from position to spin to sign run side by side
        // (entries that pad a row are position 0 with k = 0)
        int j[4];
#pragma unroll
        for (int n = 0; n < 4; ++n) j[n] = C.row_of[in.pos_off + (C.col16 ? e16.at(n) : e32.at(n)) / 4];
#pragma unroll
        for (int n = 0; n < 4; ++n) I += (int8_t)(kk >> (8 * n)) * s[j[n]];
    }
    if (a.field_out) a.field_out[in.xin_off + (size_t)r * in.N + row] = I;
    atomicAdd(reinterpret_cast<unsigned long long *>(C.Esum) + in.rec_off + r,
              (unsigned long long)((long long)s[row] * (I + h)));
}

__global__ void csr_field_energy(const CsrArgs C) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= C.total_reps) return;
    unsigned long long *slot = reinterpret_cast<unsigned long long *>(C.Esum) + idx;
    const int b = (int)(idx / C.R), r = (int)(idx - (int64_t)b * C.R);
    if (C.a.energy_out && r < C.R_real) C.a.energy_out[(size_t)b * C.R_real + r] = -((long long)*slot) / 2;
    *slot = 0ull;
}

__global__ void csr_count(const CsrArgs C) {
    if (threadIdx.x == 0 && blockIdx.x == 0)
        atomicAdd(C.a.replica_iters, (unsigned long long)((long long)C.total_reps * C.a.nsteps));
}

template <bool SMEM, bool C16, bool STAGED>
cudaError_t launch_iterations(const CsrArgs &C, size_t smem, StepGraphCache *graphs, cudaStream_t st, int sms,
                              int max_blocks, int *launches) {
    const int ny = (C.R / 32 + C.gblock - 1) / C.gblock;
    CsrArgs Cs = C;
    Cs.x_in = Cs.v_in = nullptr;
    Cs.x_out = Cs.v_out = nullptr;
    if (C.persistent) {
        // Every iteration in one cooperative launch: as many blocks as can be resident.
        auto k = csr_persistent<SMEM, C16, STAGED>;
        cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTwo);
        int per_sm = 0;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kBlk, smem);
        if (e != cudaSuccess) return e;
        const int64_t units = (int64_t)max_blocks * ny;
        const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(units, (int64_t)per_sm * sms));
        e = cudaMemsetAsync(C.sync, 0, 4 * sizeof(unsigned), st);
        if (e != cudaSuccess) return e;
        unsigned *bar = C.sync, *ctr = C.sync + 2;
        void *args[3] = {&Cs, &bar, &ctr};
        e = cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k), dim3(blocks), dim3(kBlk), args, smem, st);
        if (e != cudaSuccess) return e;
        ++*launches;
        return cudaSuccess;
    }
    // The step kernel reads its iteration from C.ctl: every launch is the same, and the
    // arguments leave out what only the prologue and the export read.
    Cs.a.t0 = 0;
    Cs.a.nsteps = 0;
    auto k = csr_step<SMEM, C16, STAGED>;
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTwo);
    if (e != cudaSuccess) return e;
    void *args[1] = {&Cs};
    for (int set = 0; set < C.nsets; ++set) {
        if (set > 0) {
            csr_next_set<<<1, 1, 0, st>>>(C.ctl, C.a.t0, C.a.nsteps, set);
            ++*launches;
        }
        e = launch_steps(graphs, reinterpret_cast<const void *>(k), dim3(max_blocks, ny), dim3(kBlk), smem, args, &Cs,
                         sizeof Cs, C.a.nsteps, st, true);
        if (e != cudaSuccess) return e;
        *launches += (int)C.a.nsteps;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t launch_csr(const CsrArgs &Cin, const int32_t *max_len, StepGraphCache *graphs, cudaStream_t st, int *launches) {
    CsrArgs C = Cin;
    int n = 0, dev = 0, sms = 0;
    cudaError_t e = cudaMemsetAsync(C.Esum, 0, 2 * (size_t)C.total_reps * sizeof(int64_t), st);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    if (C.a.field_mode) {
        const int64_t work = C.total_slices * 32 * C.R;
        csr_field_only<<<(unsigned)((work + 255) / 256), 256, 0, st>>>(C);
        csr_field_energy<<<(unsigned)((C.total_reps + 255) / 256), 256, 0, st>>>(C);
        if (launches) *launches += 2;
        return cudaGetLastError();
    }
    const int groups = C.R / 32;
    const unsigned conv = (unsigned)(C.total_slices * groups);
    // Groups per block: up to 8 share one reading of the couplings (through L1), as many as leave
    // two blocks an SM their shared memory (the figures here before copy_best took its present form),
    // with x and v staged in it (48 instances of 100 .. 3000
    // spins x 256 replicas 122 us an iteration against 140 from registers, one of 10000 19.5 against
    // 21.8).  A single group's spins that leave no room for both keep the two blocks and load x and
    // v into registers (20000 spins x 256 36 us against 43 with one block, x 1024 117 against 153
    // with the spins gathered from global memory).  Larger ones are gathered from global memory, by
    // position (30000 x 256 48 against 62 from one block's shared memory).
    constexpr size_t kStage = (size_t)kWarps * 16 * 32 * sizeof(float4);      // x and v of a slice per warp
    int G = 1;
    while (G < 8 && G < groups) G *= 2;
    while (G > 1 && (size_t)G * C.max_np * 4 + kStage > kTwo) G /= 2;
    size_t bytes = (size_t)G * C.max_np * 4;
    const bool in_smem = bytes <= kTwo, staged = bytes + kStage <= kTwo;
    if (!in_smem) {
        for (G = 1; G < 8 && G < groups;) G *= 2;
        bytes = 0;
    }
    C.by_pos = in_smem ? 0 : 1;
    C.stage_off = (int32_t)bytes;
    if (staged) bytes += kStage;
    C.gblock = G;
    const int spar = kWarps / G, ny = (groups + G - 1) / G;
    // Slices per block: 4, or as many as it has lanes for, fewer while the units do not fill the GPU
    // twice over (a set's time is that of its heaviest blocks).
    int li = spar >= 8 ? 3 : 2;                 // block lists of 1, 2, 4, 8 slices
    while ((1 << li) > spar && (int64_t)max_len[li] * ny < 4 * (int64_t)sms) --li;
    C.slices = 1 << li;
    C.list = li;
    csr_prologue<<<conv, kBlk, 0, st>>>(C);
    ++n;
    auto go = [&](auto smem, auto c16, auto stg) {
        return launch_iterations<smem.value, c16.value, stg.value>(C, bytes, graphs, st, sms, max_len[li], &n);
    };
    constexpr std::true_type yes{};
    constexpr std::false_type no{};
    if (!in_smem) e = go(no, no, no);                  // more than 16384 positions
    else if (staged) e = go(yes, yes, yes);            // at most 12544
    else e = C.col16 ? go(yes, yes, no) : go(yes, no, no);
    if (e != cudaSuccess) return e;
    const int64_t t_last = C.a.t0 + C.a.nsteps - 1;
    csr_settle_all<<<C.count, 256, 0, st>>>(C, t_last);
    const dim3 cg((unsigned)(((int64_t)groups * C.max_words + kWarps - 1) / kWarps), C.count);
    csr_copy_all<<<cg, kBlk, 0, st>>>(C, t_last - 1 >= C.a.t0 ? t_last - 1 : t_last, t_last);
    csr_count<<<1, 32, 0, st>>>(C);
    n += 3;
    if (C.x_out) {
        csr_export<<<conv, kBlk, 0, st>>>(C);
        ++n;
    }
    if (launches) *launches += n;
    return cudaGetLastError();
}

}  // namespace phia
