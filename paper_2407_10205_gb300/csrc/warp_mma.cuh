#pragma once
// warp_mma.cuh -- what the warp-level resident kernels share (k_warp.cu, k_cluster.cu): the
// warp-level tensor-core MMA and its fragments, the update of a thread's elements, and the
// best state that a thread holds for them.
//
// A warp owns 16 spins and 8 replicas; lane (g, q) = (lane / 4, lane % 4) holds the elements of
// the spins i[u] = 16 w + g + 8 u and the replicas 2 q + j at [u][j].
#include <climits>

#include <cuda_bf16.h>
#include <cuda_fp8.h>

#include "device_common.cuh"
#include "phia_internal.h"

namespace phia {

constexpr uint32_t kMagicBits = 0x4B400000u;   // 1.5 x 2^23: x + this holds x in its low bits

template <int OP>
__device__ __forceinline__ void mma_step(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
    if constexpr (OP == kOpE4M3) {
        asm volatile(
            "mma.sync.aligned.m16n8k32.row.col.f32.e4m3.e4m3.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
    } else {
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
            : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
    }
}

// One K-step's B fragment.  Volatile, so that the loads stay with their MMAs: hoisted together
// they cost more registers than the kernels have.
__device__ __forceinline__ uint2 lds_fragment(const uint2 *p) {
    uint2 b;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(b.x), "=r"(b.y) : "r"(smem_u32(p)) : "memory");
    return b;
}

// The 8 x 8 matrix of 16-bit values whose row lane / 4 holds this lane's pair, transposed.
__device__ __forceinline__ uint32_t transpose_8x8(uint32_t v) {
    asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %0;" : "+r"(v));
    return v;
}

// A fragments of the warp's 16 rows of J: element e holds row i[e % 2] and the K slots 4 q ..
// (e4m3) or 2 q .. (bf16) of the K-step's half e / 2, a half being a block of 16 spins (e4m3) or
// of 8 (bf16).  The slots 4 q + {0, 1, 2, 3} of an e4m3 block are its spins 2q, 2q + 8, 2q + 1,
// 2q + 9, the order in which the transposed signs come out of spin_fragment_e4m3.
template <int OP, int KS>
__device__ __forceinline__ void load_fragments(uint32_t (&af)[KS][4], const int8_t *Jk, int N, const int (&i)[2], int q) {
    auto enc = [&](int row, int col) -> uint32_t {
        const float k = (row < N && col < N) ? (float)Jk[(size_t)row * N + col] : 0.0f;
        if constexpr (OP == kOpE4M3) return (uint32_t)__nv_fp8_e4m3(k).__x;
        else return __bfloat16_as_ushort(__float2bfloat16_rn(k));
    };
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int row = i[e & 1];
            if constexpr (OP == kOpE4M3) {
                const int col = 32 * ks + 16 * (e >> 1) + 2 * q;
                af[ks][e] = enc(row, col) | (enc(row, col + 8) << 8) | (enc(row, col + 1) << 16) | (enc(row, col + 9) << 24);
            } else {
                const int col = 16 * ks + 8 * (e >> 1) + 2 * q;
                af[ks][e] = enc(row, col) | (enc(row, col + 1) << 16);
            }
        }
}

// The warp's signs (minus masks [u][j]) as B fragments: rows of the 8 x 8
// transpose are spins, columns replicas.  e4m3: an element is the two bytes of spins g and
// g + 8, and the transposed pair is the warp's half of K-step w / 2; bf16: one transpose per 8
// spins, both halves of K-step w.
__device__ __forceinline__ uint32_t spin_fragment_e4m3(const uint32_t (&m)[2][2]) {
    const uint32_t w = __byte_perm(__byte_perm(m[0][0], m[1][0], 0x0040), __byte_perm(m[0][1], m[1][1], 0x0040), 0x5410);
    return transpose_8x8(0x38383838u ^ (w & 0x80808080u));
}
__device__ __forceinline__ uint2 spin_fragment_bf16(const uint32_t (&m)[2][2]) {
    return make_uint2(transpose_8x8(spins2_bf16(m[0][0], m[0][1])), transpose_8x8(spins2_bf16(m[1][0], m[1][1])));
}

// Sum of the warp's 16 spins' terms (es[j]: this lane's two spins, replica 2 q + j): replica c of
// the tile in lane c < 8, stored as q + 4 j.
__device__ __forceinline__ int32_t sum_rows(const int32_t (&es)[2], int lane) {
    const bool hi = lane & 4;
    int32_t s = (hi ? es[1] : es[0]) + __shfl_xor_sync(0xffffffffu, hi ? es[0] : es[1], 4);
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    return s;
}

// The elements of a thread: position, momentum, minus mask of the spin.
struct Elems {
    float x[2][2], v[2][2];
    uint32_t m[2][2];
};

// Derivative factors of the elements' positions.
__device__ __forceinline__ void factors(const Elems &s, float (&f)[2][2], int deriv, float bgq, float gamma) {
    if (deriv == 1) {
#pragma unroll
        for (int e = 0; e < 4; ++e) f[e >> 1][e & 1] = factor_quad(s.x[e >> 1][e & 1], bgq, gamma);
    } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) f[e >> 1][e & 1] = factor_exact(s.x[e >> 1][e & 1], 4.0f * bgq, gamma);
    }
}

// Energy terms s (J s + 2 h) of an iteration (d = J s; m its spins) per replica, exact: the sum
// of d with the rounding constant holds d in its bits.  Rows past N have d = h = 0.
__device__ __forceinline__ void energy_terms(const float (&d)[2][2], const uint32_t (&m)[2][2], const int32_t (&h2c)[2],
                                             int32_t (&es)[2]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        es[j] = 0;
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int32_t e = __float_as_int(__fadd_rn(d[u][j], 12582912.0f)) + h2c[u], k = (int32_t)m[u][j];
            es[j] += (e ^ k) - k;
        }
    }
}

// Field I = d + h (Eq. 6; FP32 sum of two exact integers), momentum (Eqs. 5, 8, A7).
__device__ __forceinline__ void momentum_step(Elems &s, const float (&d)[2][2], const float (&f)[2][2], const float (&hf)[2],
                                              float eps) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int u = e >> 1, j = e & 1;
        s.v[u][j] = momentum_of(s.v[u][j], s.x[u][j], __fadd_rn(d[u][j], hf[u]), f[u][j], eps);
    }
}
__device__ __forceinline__ void position_step(Elems &s, float eps) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int u = e >> 1, j = e & 1;
        s.x[u][j] = __fmaf_rn(eps, s.v[u][j], s.x[u][j]);
        s.m[u][j] = minus_mask(s.x[u][j]);
    }
}
// Momentum draw d = t1 for replicas r, r + 1 and spins i.
__device__ __forceinline__ void refresh_step(Elems &s, uint64_t seed, uint32_t inst, uint32_t r, const int (&i)[2], uint32_t t1) {
#pragma unroll
    for (int e = 0; e < 4; ++e)
        s.v[e >> 1][e & 1] = draw_v(seed, inst, r + (e & 1), (uint32_t)i[e >> 1], t1);
}

// The state before the first iteration: the Philox draw d = 0 or the caller's, the refresh at
// t0, the position half of Eq. A7.  Elements past N or R are 0.
__device__ __forceinline__ void initial_state(Elems &s, const RunArgs &a, const SmallCta &ic, int r0, const int (&i)[2]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int u = e >> 1, j = e & 1, r = r0 + j;
        float x = 0.0f, v = 0.0f;
        if (i[u] < ic.N) {
            if (a.x_in) {
                if (r < a.R) {
                    x = a.x_in[(size_t)r * ic.N + i[u]];
                    v = a.v_in[(size_t)r * ic.N + i[u]];
                }
            } else {
                const U4 o = draw_raw(a.seed, ic.inst, (uint32_t)r, (uint32_t)i[u], 0u);
                x = box_muller(o.x, o.y);
                v = box_muller(o.z, o.w);
            }
            if (refresh_at(a.t0, a.refresh)) v = draw_v(a.seed, ic.inst, (uint32_t)r, (uint32_t)i[u], (uint32_t)a.t0);
            x = __fmaf_rn(a.eps, v, x);
        }
        s.x[u][j] = x;
        s.v[u][j] = v;
        s.m[u][j] = minus_mask(x);
    }
}
__device__ __forceinline__ void export_state(const Elems &s, const RunArgs &a, int N, int r0, const int (&i)[2]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int u = e >> 1, j = e & 1, r = r0 + j;
        if (i[u] < N && r < a.R) {
            a.x_out[(size_t)r * N + i[u]] = s.x[u][j];
            a.v_out[(size_t)r * N + i[u]] = s.v[u][j];
        }
    }
}

// The signs of a thread's elements: bit 2 j + u, set for plus.
__device__ __forceinline__ uint32_t sign_bits(const Elems &s) {
    uint32_t m = 0;
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int u = 0; u < 2; ++u) m |= ~s.m[u][j] & (1u << (2 * j + u));
    return m;
}

// The best state of a thread's elements (bits as above) and whether its two replicas ever
// improved (bits 0 and 1).
struct BestBits {
    uint32_t bits = 0, ever = 0;
    // `was` where the replicas 2 q, 2 q + 1 improved: the bytes of imp2.
    __device__ __forceinline__ void take(uint32_t imp2, uint32_t was) {
        if (!imp2) return;
        const uint32_t sel = (imp2 & 1u) * 3u | (imp2 & 0x100u ? 12u : 0u);
        bits = (bits & ~sel) | (was & sel);
        ever |= (imp2 & 1u) | ((imp2 >> 7) & 2u);
    }
    // Into the packed best states of replicas rbase .. rbase + 7: the 16 spins of warp gw are
    // half a word.
    __device__ __forceinline__ void store(uint32_t *best_bits, int rbase, int R, int W, int gw, int N, int lane) const {
        uint32_t bal[2][2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int u = 0; u < 2; ++u) bal[j][u] = __ballot_sync(0xffffffffu, (bits >> (2 * j + u)) & 1u);
        const int qq = (lane & 7) >> 1, jj = lane & 1, r = rbase + (lane & 7);
        const uint32_t ev = __shfl_sync(0xffffffffu, ever, qq);
        if (lane < 8 && r < R && ((ev >> jj) & 1u) && 16 * gw < N) {
            const uint32_t lo = (jj ? bal[1][0] : bal[0][0]) >> qq, hi = (jj ? bal[1][1] : bal[0][1]) >> qq;
            uint32_t w = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) w |= ((lo >> (4 * k)) & 1u) << k | ((hi >> (4 * k)) & 1u) << (k + 8);
            if (N - 16 * gw < 16) w &= (1u << (N - 16 * gw)) - 1u;
            reinterpret_cast<uint16_t *>(best_bits + (size_t)r * W)[gw] = (uint16_t)w;
        }
    }
};

// Record of one replica (Table 3, state 5), held alike by the lanes that settle it.
struct Record {
    long long best_e, best_step, hit;
    uint64_t hit_ns;
    bool live;
    __device__ __forceinline__ void load(const RunArgs &a, int64_t off, int r) {
        live = r < a.R;
        best_e = live ? (long long)a.best_e[off + r] : LLONG_MAX;
        best_step = live ? (long long)a.best_step[off + r] : -1;
        hit = live ? (long long)a.hit_step[off + r] : -1;
        hit_ns = live && a.hit_ns ? a.hit_ns[off + r] : 0ull;
    }
    __device__ __forceinline__ void store(const RunArgs &a, int64_t off, int r) const {
        if (!live) return;
        a.best_e[off + r] = best_e;
        a.best_step[off + r] = best_step;
        a.hit_step[off + r] = hit;
        if (a.hit_ns) a.hit_ns[off + r] = hit_ns;
    }
    // Iteration t with twice = sum s (I + h) = -2 E; true when it improved.  first_hit: set when
    // the replica reached its target in it.
    __device__ __forceinline__ bool settle(const RunArgs &a, int64_t target, int64_t t, long long twice, bool &first_hit) {
        const long long E = -twice / 2;                          // Eq. 2 via the field
        const bool imp = live && !(a.stop_at_target && hit >= 0) && E < best_e;
        if (imp) {
            best_e = E;
            best_step = t;
        }
        first_hit = live && a.has_target && hit < 0 && E <= target;
        if (first_hit) {
            hit = t;
            hit_ns = globaltimer_ns();
        }
        return imp;
    }
};

}  // namespace phia
