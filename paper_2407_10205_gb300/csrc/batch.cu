// batch.cu -- batched multi-instance runs (phia_batch_* of the C ABI): instance validation
// and packing, per-replica state of every instance.  Small dense instances (N <= 384 with
// every |k| <= 16, N <= 256 otherwise) run on resident kernels over a table of CTAs, all their
// iterations in one launch per size class; the rest run on the sparse path (dense ones
// converted): slices of 32 rows in sets of instances (k_csr.cu), or for large instances of few
// couplings a row the form with a row to a warp (k_csr_rows.cu), with one launch per iteration
// or one persistent launch over all iterations.  Batches of small sparse instances alone run on
// the resident kernels too.
#include <algorithm>
#include <atomic>
#include <climits>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <functional>
#include <new>
#include <string>
#include <system_error>
#include <thread>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/phia.h"
#include "device_common.cuh"
#include "grow.h"
#include "phia_internal.h"

using namespace phia;

namespace {

// What the choice between the two sparse forms goes by, over all CSR members.
struct SparseShape {
    int max_np = 0;                     // most positions (spins rounded up to 32)
    int64_t rows = 0;
    double degree = 0.0;                // couplings a row, with those that pad the slices
    int longest = 0;                    // couplings of the longest row
};

// Picoseconds per update (spin, replica as run, iteration) of the two sparse forms once an instance
// fills the GPU, fitted to 20000 .. 60000 spins x 256 .. 1024 replicas of degree 6 .. 60: k_csr.cu
// with its spins in shared memory (up to 28928 positions) or by position, and k_csr_rows.cu.
double lanes_ps(const SparseShape &s) {
    return s.max_np <= 28928 ? 4.55 + 0.023 * s.degree : 4.1 + 0.105 * s.degree;
}
double rows_ps(const SparseShape &s) { return 3.5 + 0.052 * s.degree; }

// A row of thousands of couplings among short ones: one warp's way along it, 0.036 us a coupling, can
// be the whole iteration.
bool has_hub(const SparseShape &s) { return s.longest >= 2048 && s.longest >= 8.0 * s.degree; }

// Whether a replica count exists for which k_csr_rows.cu is the faster form.  Up to 12544 positions
// k_csr.cu has x and v in shared memory too and is never slower (10000 x 1024, degree 6: 40 us
// against 42).
bool rows_form_possible(const SparseShape &s) {
    return has_hub(s) || (s.max_np > 12544 && rows_ps(s) < lanes_ps(s));
}

// Whether a run of `replicas` takes it.  It pads them to 256 instead of 32, and below 5e6 updates an
// iteration latencies set the time (13000 x 256 of degree 6: 18.3 us against 17.7).  Where a hub sets
// it (stars: a ring and one row coupled to all), k_csr.cu keeps up with 16-bit offsets and few
// replicas (10000 x 256 366 us against 368) and not past them (10000 x 1024 657 us against 400, 20000 x
// 64 878 against 724, 30000 x 64 1870 against 1094).
bool rows_form(const SparseShape &s, int replicas) {
    if (!rows_form_possible(s)) return false;
    const double updates = (double)s.rows * round_up(replicas, 256);
    const double lanes_us = 1e-6 * (double)s.rows * round_up(replicas, 32) * lanes_ps(s);
    if (has_hub(s) && 0.036 * s.longest > lanes_us) return s.max_np > 16384 || replicas > 256;
    return updates >= 5e6 && 1e-6 * updates * rows_ps(s) < lanes_us;
}

}  // namespace

struct phia_batch_s {
    int device = 0;
    cudaStream_t stream = nullptr;
    int count = 0;                      // instances (public indices 0 .. count-1)
    std::vector<CsrInst> inst;          // CSR members only (offsets for replicas set per run)
    std::vector<int> csr_pub;           // CSR member -> public index
    std::vector<int> N, frac;           // per public instance
    std::vector<uint32_t> inst_id;
    std::vector<int64_t> h_off;         // into d_hk
    // small dense members: a resident kernel over a table of CTAs
    std::vector<int> dense_pub;         // public indices
    std::vector<int64_t> dense_joff;    // offset of each member's J in d_dJ
    std::vector<int> dense_op;          // kOpE4M3 / kOpBF16
    // sparse members that are small enough for a resident kernel as well (all of the batch's, else
    // none): offset of each one's dense J in d_dJ
    std::vector<int64_t> cand_joff;
    int8_t *d_dJ = nullptr;
    SmallCta *d_small = nullptr;
    size_t small_cap = 0;
    std::vector<SmallCta> small_host;
    std::vector<int64_t> bits_pub;      // per public instance: offset of its best states
    std::vector<long long> targets;     // per instance, LLONG_MIN = none
    std::vector<CsrBlock> blocks;       // the block lists for 1, 2, 4 and 8 slices a block, in instance order
    std::vector<int32_t> first_block[4];   // per CSR member (and one past): its first block in each list
    std::vector<CsrSet> sets;           // instances whose state fits in L2 together, for sets_R replicas
    int sets_R = 0;
    int32_t set_max[4] = {0, 0, 0, 0};
    CsrSet *d_sets = nullptr;
    int64_t total_slices = 0;
    int max_words = 0;
    CsrInst *d_inst = nullptr;
    CsrBlock *d_blocks = nullptr;
    void *d_col = nullptr;              // uint16 offsets (col16) or uint32
    bool col16 = false;
    int32_t *d_slice = nullptr, *d_hk2 = nullptr, *d_rowof = nullptr, *d_posof = nullptr;
    uint32_t *d_val = nullptr;
    int32_t *d_hk = nullptr;            // fields of the small dense members
    // the CSR members once more with a row to a warp (k_csr_rows.cu), where some replica count may take it
    std::vector<CsrRowsInst> rows_inst;
    int32_t rows_blocks = 0;
    SparseShape shape;
    CsrRowsInst *d_rows_inst = nullptr;
    CsrRowsBlock *d_rows_blocks = nullptr;
    int32_t *d_rows_ptr = nullptr, *d_rows_col = nullptr, *d_rows_h = nullptr;
    int8_t *d_rows_val = nullptr;
    long long *d_targets = nullptr;
    bool any_target = false;
    // replica state (R padded to a multiple of 32)
    int Rcap = 0, R = 0, R_real = 0;
    float *d_X = nullptr, *d_V = nullptr;
    uint32_t *d_S = nullptr;
    int64_t *d_Esum = nullptr;
    int8_t *d_flags = nullptr;
    int64_t *d_best_e = nullptr, *d_best_step = nullptr, *d_hit = nullptr;
    uint32_t *d_bits = nullptr;
    unsigned long long *d_min_hit = nullptr, *d_iters = nullptr;
    uint64_t *d_hit_ns = nullptr;       // %globaltimer of each replica's first hit
    uint64_t *d_start_ns = nullptr;     // %globaltimer when the run's records were reset
    int32_t *d_err = nullptr;
    IterCtl *d_ctl = nullptr;               // iteration control of the step kernel
    unsigned *d_sync = nullptr;             // barrier and work counters of the persistent launch
    int csr_mode = 2;                       // 1 persistent CSR launch, 2 one launch per iteration
    StepGraphCache *graphs = nullptr;       // its step launches as replayable graphs
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    bool ran = false;
    bool waits_checked = false;         // the last run's error flag has been read (and is clear)
    int64_t last_steps = 0;
    int last_launches = 0;
    int last_stop = 0;
};

namespace {

int bfail(int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    return set_last_error(code, buf);
}

#define BCU(call)                                                                                   \
    do {                                                                                            \
        cudaError_t e_ = (call);                                                                    \
        if (e_ != cudaSuccess) return bfail(PHIA_ECUDA, "%s: %s", #call, cudaGetErrorString(e_));   \
    } while (0)

__global__ void batch_reset_records(int64_t n, int64_t nbits, int64_t *best_e, int64_t *best_step, int64_t *hit,
                                    uint32_t *bits, uint64_t *hit_ns, uint64_t *start_ns) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx < n) {
        best_e[idx] = LLONG_MAX;
        best_step[idx] = -1;
        hit[idx] = -1;
        hit_ns[idx] = 0;
    }
    if (idx < nbits) bits[idx] = 0u;
    if (idx == 0) *start_ns = globaltimer_ns();   // the run's start on the device clock
}

void free_state(phia_batch_s *b) {
    for (void *p : {(void *)b->d_X, (void *)b->d_V, (void *)b->d_S, (void *)b->d_Esum, (void *)b->d_flags,
                    (void *)b->d_best_e, (void *)b->d_bits, (void *)b->d_hit_ns})
        pool_free(p, b->stream);
    b->d_X = b->d_V = nullptr; b->d_S = nullptr; b->d_Esum = nullptr; b->d_flags = nullptr;
    b->d_best_e = b->d_best_step = b->d_hit = nullptr; b->d_bits = nullptr; b->d_hit_ns = nullptr;
    b->Rcap = 0;
}

int64_t words_of(int n) { return (n + 31) / 32; }

// Per-replica offsets for R replicas per instance: records and best states by public
// index (instance k's records start at k R), CSR state over the CSR members only.
void layout(phia_batch_s *b, int R) {
    b->bits_pub.assign((size_t)b->count, 0);
    int64_t bits = 0;
    for (int k = 0; k < b->count; ++k) {
        b->bits_pub[(size_t)k] = bits;
        bits += (int64_t)R * words_of(b->N[(size_t)k]);
    }
    int64_t x = 0, xin = 0, s = 0;
    for (size_t c = 0; c < b->inst.size(); ++c) {
        CsrInst &in = b->inst[c];
        const int k = b->csr_pub[c];
        in.x_off = x; in.xin_off = xin; in.s_off = s;
        in.rec_off = (int64_t)k * R;
        in.bits_off = b->bits_pub[(size_t)k];
        x += (int64_t)in.Np * R;
        xin += (int64_t)in.N * b->R_real;
        s += (int64_t)in.Np * (R / 32);
        if (c < b->rows_inst.size()) {
            CsrRowsInst &ri = b->rows_inst[c];
            ri.x_off = ri.row_base * R;
            ri.xin_off = in.xin_off;
            ri.s_off = ri.row_base * (R / 32);
            ri.rec_off = in.rec_off;
            ri.bits_off = in.bits_off;
        }
    }
}

// Sets of consecutive CSR members for R replicas: as few as keep a set's x and v within 0.4 of L2,
// of about equal size.  The device gets a copy of the block lists with each set's blocks sorted: the
// host's stay in instance order, which first_block counts on when another replica count cuts the
// members into other sets.
int make_sets(phia_batch_s *b, int R) {
    int l2 = 0;
    BCU(cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, b->device));
    const int n = (int)b->inst.size();
    int64_t total = 0;
    for (const CsrInst &in : b->inst) total += (int64_t)in.Np * R * 8;
    const int64_t budget = std::max<int64_t>(1, (int64_t)(0.4 * l2));
    const int64_t share = total / std::max<int64_t>(1, (total + budget - 1) / budget) + 1;
    b->sets_R = 0;
    b->sets.clear();
    std::fill(b->set_max, b->set_max + 4, 0);
    std::vector<CsrBlock> blocks = b->blocks;
    int64_t seen = 0;
    for (int c0 = 0, c = 0; c < n; ++c) {
        seen += (int64_t)b->inst[(size_t)c].Np * R * 8;
        if (c + 1 < n && seen < share * (int64_t)(b->sets.size() + 1)) continue;
        CsrSet s;
        for (int l = 0; l < 4; ++l) {
            s.off[l] = b->first_block[l][(size_t)c0];
            s.len[l] = b->first_block[l][(size_t)c + 1] - s.off[l];
            b->set_max[l] = std::max(b->set_max[l], s.len[l]);
        }
        // the heaviest blocks first
        for (int l = 0; l < 4; ++l)
            std::stable_sort(blocks.begin() + s.off[l], blocks.begin() + s.off[l] + s.len[l],
                             [&](const CsrBlock &x, const CsrBlock &y) { return x.work > y.work; });
        b->sets.push_back(s);
        c0 = c + 1;
    }
    BCU(cudaMemcpyAsync(b->d_blocks, blocks.data(), blocks.size() * sizeof(CsrBlock), cudaMemcpyHostToDevice, b->stream));
    BCU(cudaMemcpyAsync(b->d_sets, b->sets.data(), b->sets.size() * sizeof(CsrSet), cudaMemcpyHostToDevice, b->stream));
    BCU(cudaStreamSynchronize(b->stream));
    b->sets_R = R;
    return PHIA_OK;
}

int ensure_state(phia_batch_s *b, int R) {
    if (R <= b->Rcap) return PHIA_OK;
    BCU(cudaStreamSynchronize(b->stream));
    free_state(b);
    const int64_t rows = b->total_slices * 32;
    int64_t bits = 0;
    for (int k = 0; k < b->count; ++k) bits += (int64_t)R * words_of(b->N[k]);
    const int64_t reps = (int64_t)R * b->count;
    bool ok = true;
    auto al = [&](void **p, size_t n) {
        if (ok && pool_alloc(p, n, b->device, b->stream) != cudaSuccess) ok = false;
    };
    al((void **)&b->d_X, (size_t)rows * R * 4);
    al((void **)&b->d_V, (size_t)rows * R * 4);
    al((void **)&b->d_S, (size_t)4 * rows * (R / 32) * 4);
    al((void **)&b->d_Esum, (size_t)2 * reps * 8);
    al((void **)&b->d_flags, (size_t)2 * reps);
    al((void **)&b->d_best_e, (size_t)3 * reps * 8);   // best energy, its iteration, first hit
    b->d_best_step = b->d_best_e + reps;
    b->d_hit = b->d_best_step + reps;
    al((void **)&b->d_hit_ns, (size_t)reps * 8);
    al((void **)&b->d_bits, (size_t)bits * 4);
    if (!ok) {
        cudaGetLastError();
        free_state(b);
        return bfail(PHIA_ENOMEM, "device allocation for %d replicas per instance failed", R);
    }
    BCU(cudaMemsetAsync(b->d_flags, 0, (size_t)2 * reps, b->stream));
    b->Rcap = R;
    return PHIA_OK;
}

}  // namespace

namespace phia {

// Starts fn on a thread of `workers` (which has room for it); false where the system has none left.
template <typename F>
bool start_thread(std::vector<std::thread> &workers, F fn) {
    try {
        workers.emplace_back(fn);
        return true;
    } catch (const std::system_error &) {
        return false;
    }
}

// One instance of a batch, checked and converted to slices of 32 rows (relative to the
// instance), before concatenation; code/msg hold its first error.
struct PackedInst {
    int code = PHIA_OK;
    std::string msg;
    std::vector<int32_t> slice, col, hk2, row_of, pos_of;
    std::vector<uint32_t> val;
    int wide = 0;
    int small_op = 0;       // small dense member: its tensor-core operand (no slices built)
    std::vector<int8_t> dense;   // J of a member with slices that a resident kernel could run too
};

void pack_error(PackedInst &out, int code, const char *fmt, ...) {
    char buf[512];
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(buf, sizeof buf, fmt, ap);
    va_end(ap);
    out.code = code;
    out.msg = buf;
}

// The slices of a checked instance: rows sorted by their number of couplings (descending,
// ties in row order), 32 to a slice, every row padded to the slice's longest with k = 0.
void pack_slices(int n, const int32_t *rp, const int32_t *col, const int8_t *val, const int32_t *h, int threads,
                 PackedInst &out) {
    const int np = round_up(n, 32), ns = np / 32;
    std::vector<int32_t> order((size_t)n);
    for (int i = 0; i < n; ++i) order[(size_t)i] = i;
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return rp[a + 1] - rp[a] > rp[b + 1] - rp[b]; });
    out.row_of.assign((size_t)np, -1);
    out.pos_of.resize((size_t)n);
    for (int p = 0; p < n; ++p) {
        out.row_of[(size_t)p] = order[(size_t)p];
        out.pos_of[(size_t)order[(size_t)p]] = p;
    }
    out.slice.assign((size_t)ns + 1, 0);
    for (int s = 0; s < ns; ++s) {
        const int first = order[(size_t)s * 32];       // the slice's longest row
        out.slice[(size_t)s + 1] = out.slice[(size_t)s] + (rp[first + 1] - rp[first] + 3) / 4;
    }
    out.col.assign((size_t)out.slice[(size_t)ns] * 128, 0);
    out.val.assign((size_t)out.slice[(size_t)ns] * 32, 0u);
    out.hk2.assign((size_t)np * 2, 0);
    // Whole slices to a host thread: an instance of 1e6 couplings takes several ms on one.
    std::atomic<int64_t> bound{0};
    auto fill = [&](int s0, int s1) {
        int64_t most = 0;
        for (int p = s0 * 32; p < std::min(n, s1 * 32); ++p) {
            const int i = order[(size_t)p], lane = p & 31;
            const size_t e0 = (size_t)out.slice[(size_t)p / 32];
            int64_t mag = 2 * std::abs((int64_t)h[i]);
            int32_t ksum = 0;
            for (int32_t c = rp[i]; c < rp[i + 1]; ++c) {
                const size_t m = (size_t)(c - rp[i]), e = e0 + m / 4;
                out.col[(e * 32 + (size_t)lane) * 4 + m % 4] = out.pos_of[(size_t)col[c]] * 4;
                out.val[e * 32 + (size_t)lane] |= (uint32_t)(uint8_t)val[c] << (8 * (m % 4));
                ksum += val[c];
                mag += std::abs((int)val[c]);
            }
            out.hk2[(size_t)p * 2] = h[i];
            out.hk2[(size_t)p * 2 + 1] = h[i] - ksum;
            most = std::max(most, mag);
        }
        for (int64_t b = bound.load(); b < most && !bound.compare_exchange_weak(b, most);) {}
    };
    const int nt = std::min<int>({threads, ns, rp[n] / 65536 + 1});
    std::vector<std::thread> workers;
    workers.reserve((size_t)nt);
    int done = 0;                                  // slices given out, by entries
    for (int k = 1; k <= nt; ++k) {
        int next = done;
        while (next < ns && (k == nt || (int64_t)out.slice[(size_t)next] * nt < (int64_t)out.slice[(size_t)ns] * k)) ++next;
        if (k == nt || !start_thread(workers, [&fill, done, next] { fill(done, next); })) fill(done, next);
        done = next;
    }
    for (std::thread &w : workers) w.join();
    // |I + h| <= bound: 128 rows' terms and a sum scaled by 2^7 stay in 32 bits up to 2^23.
    out.wide = bound.load() > ((int64_t)1 << 23);
    if (n > cluster_batch_max_n()) return;
    out.dense.assign((size_t)n * n, 0);
    for (int i = 0; i < n; ++i)
        for (int32_t c = rp[i]; c < rp[i + 1]; ++c) {
            int8_t &k = out.dense[(size_t)i * n + col[c]];
            const int sum = (int)k + val[c];                // entries of one coupling add up
            if (std::abs(sum) > 127) {
                out.dense.clear();
                return;
            }
            k = (int8_t)sum;
        }
}

// The rows of a checked instance in their own order, every one padded to a multiple of 8 entries with
// k = 0, after those of the instances before.
void append_rows(const phia_instance_desc &x, std::vector<int32_t> &ptr, std::vector<int32_t> &col, std::vector<int8_t> &val) {
    const size_t base = col.size();
    ptr.push_back(0);
    for (int i = 0; i < x.N; ++i) {
        if (x.J_k) {
            const int8_t *row = x.J_k + (size_t)i * x.N;
            for (int j = 0; j < x.N; ++j)
                if (row[j] != 0) {
                    col.push_back(j);
                    val.push_back(row[j]);
                }
        } else {
            col.insert(col.end(), x.col + x.row_ptr[i], x.col + x.row_ptr[i + 1]);
            val.insert(val.end(), x.val_k + x.row_ptr[i], x.val_k + x.row_ptr[i + 1]);
        }
        col.resize(base + (col.size() - base + 7) / 8 * 8, 0);
        val.resize(col.size(), 0);
        ptr.push_back((int32_t)(col.size() - base));
    }
}

void pack_instance(const phia_instance_desc &x, int k, int threads, PackedInst &out) {
    const int n = x.N;
    if (n < 1) return pack_error(out, PHIA_EINVAL, "instance %d: N must be >= 1", k);
    if (x.frac_bits < 0 || x.frac_bits > 30) return pack_error(out, PHIA_EINVAL, "instance %d: bad frac_bits", k);
    if (!x.h_k) return pack_error(out, PHIA_EINVAL, "instance %d: h_k is NULL", k);
    for (int i = 0; i < n; ++i)
        if (x.h_k[i] >= (1 << 24) || x.h_k[i] <= -(1 << 24))
            return pack_error(out, PHIA_ERANGE, "instance %d: |h_k[%d]| >= 2^24", k, i);
    // Rows as lists of (column, coupling), in CSR order.
    std::vector<int32_t> rp((size_t)n + 1, 0), col;
    std::vector<int8_t> val;
    if (x.J_k) {
        // Small enough for the resident tensor-core kernel: checked here, kept dense.
        int maxk = 0;
        for (int i = 0; i < n; ++i) {
            if (x.J_k[(size_t)i * n + i] != 0) return pack_error(out, PHIA_EINVAL, "instance %d: nonzero diagonal", k);
            for (int j = i + 1; j < n; ++j) {
                const int a = x.J_k[(size_t)i * n + j];
                if (a != x.J_k[(size_t)j * n + i])
                    return pack_error(out, PHIA_EINVAL, "instance %d: J_k is not symmetric at (%d, %d)", k, i, j);
                maxk = std::max(maxk, std::abs(a));
            }
        }
        const int op = maxk <= 16 ? kOpE4M3 : kOpBF16;
        if (n <= tc_small_max_n(op)) {
            out.small_op = op;
            return;
        }
        for (int i = 0; i < n; ++i) {
            if (x.J_k[(size_t)i * n + i] != 0) return pack_error(out, PHIA_EINVAL, "instance %d: nonzero diagonal", k);
            for (int j = 0; j < n; ++j) {
                if (x.J_k[(size_t)i * n + j] != x.J_k[(size_t)j * n + i])
                    return pack_error(out, PHIA_EINVAL, "instance %d: J_k is not symmetric at (%d, %d)", k, i, j);
                if (x.J_k[(size_t)i * n + j] != 0) {
                    col.push_back(j);
                    val.push_back(x.J_k[(size_t)i * n + j]);
                }
            }
            rp[i + 1] = (int32_t)col.size();
        }
        return pack_slices(n, rp.data(), col.data(), val.data(), x.h_k, threads, out);
    }
    if (!x.row_ptr || !x.col || !x.val_k) return pack_error(out, PHIA_EINVAL, "instance %d: CSR arrays missing", k);
    if (x.row_ptr[0] != 0) return pack_error(out, PHIA_EINVAL, "instance %d: row_ptr[0] != 0", k);
    for (int i = 0; i < n; ++i)
        if (x.row_ptr[i + 1] < x.row_ptr[i]) return pack_error(out, PHIA_EINVAL, "instance %d: row_ptr decreases", k);
    // Rows with ascending columns are searched by bisection in the symmetry check.
    std::vector<uint8_t> row_sorted(n);
    for (int i = 0; i < n; ++i) row_sorted[i] = std::is_sorted(x.col + x.row_ptr[i], x.col + x.row_ptr[i + 1]);
    for (int i = 0; i < n; ++i) {
        for (int32_t p = x.row_ptr[i]; p < x.row_ptr[i + 1]; ++p) {
            const int j = x.col[p];
            if (j < 0 || j >= n) return pack_error(out, PHIA_EINVAL, "instance %d: col out of range", k);
            if (j == i) return pack_error(out, PHIA_EINVAL, "instance %d: self loop at %d", k, i);
            // symmetry: (j, i) must exist with the same value
            const int32_t *cb = x.col + x.row_ptr[j], *ce = x.col + x.row_ptr[j + 1];
            const int32_t *f = row_sorted[j] ? std::lower_bound(cb, ce, i) : std::find(cb, ce, i);
            if (f != ce && *f != i) f = ce;
            if (f == ce || x.val_k[x.row_ptr[j] + (f - cb)] != x.val_k[p])
                return pack_error(out, PHIA_EINVAL, "instance %d: CSR is not symmetric at (%d, %d)", k, i, j);
        }
    }
    pack_slices(n, x.row_ptr, x.col, x.val_k, x.h_k, threads, out);
}

int64_t csr_device_bytes(int n, const int32_t *row_ptr, int replicas) {
    const int np = round_up(n, 32);
    std::vector<int32_t> len((size_t)np, 0);
    int64_t padded8 = 0;
    for (int i = 0; i < n; ++i) {
        len[(size_t)i] = row_ptr[i + 1] - row_ptr[i];
        padded8 += (len[(size_t)i] + 7) / 8 * 8;
    }
    std::sort(len.begin(), len.end(), std::greater<int32_t>());
    int64_t entries = 0;
    for (int p = 0; p < np; p += 32) entries += (len[(size_t)p] + 3) / 4;
    const SparseShape s{np, n, 128.0 * (double)entries / n, len[0]};
    const int64_t R = round_up(replicas, rows_form(s, replicas) ? 256 : 32);
    int64_t b = entries * 32 * (np <= 16384 ? 12 : 20) + (int64_t)np * 20;           // slices, h, positions
    if (rows_form_possible(s)) b += padded8 * 5 + (int64_t)n * 8;
    if (n <= cluster_batch_max_n()) b += (int64_t)n * n;
    b += (int64_t)np * R * 8 + 4 * (int64_t)np * (R / 32) * 4;                       // x, v, spins
    return b + R * (16 + 2 + 24 + 8) + R * words_of(n) * 4;                          // sums, flags, records
}

// batch_create; b: the batch as far as it got, for the caller to destroy after an exception.
int create_batch(phia_batch_s *&b, phia_batch_s **out, int32_t count, const phia_instance_desc *d, const phia_opts *opts) {
    if (count < 1 || !d) return bfail(PHIA_EINVAL, "need count >= 1 and descriptors");
    phia_opts o{};
    if (opts) o = *opts;
    if (o.path != PHIA_PATH_AUTO && o.path != PHIA_PATH_CSR)
        return bfail(PHIA_ENOTSUP, "batches run on the CSR path");
    if (o.tc_kernel < 0 || o.tc_kernel > 2) return bfail(PHIA_EINVAL, "batches: tc_kernel must be 0, 1 or 2");
    b = new phia_batch_s();
    b->csr_mode = o.tc_kernel == 1 ? 1 : 2;
    auto cleanup = [&](int code) {
        phia_batch_destroy(b);
        b = nullptr;
        return code;
    };
    b->count = count;
    // Instances are checked and converted independently, on every host core (a batch of
    // 256 instances with 2.8e7 couplings took 1.3 s on one core); the first failing
    // instance in order is reported, as a sequential pass would.
    std::vector<PackedInst> packed((size_t)count);
    {
        std::atomic<int> next{0};
        const int cores = std::max(1, (int)std::thread::hardware_concurrency());
        const int nthreads = std::min<int>(count, cores);
        auto work = [&]() {
            for (int k; (k = next.fetch_add(1)) < count;) {
                try {
                    pack_instance(d[k], k, cores / nthreads, packed[(size_t)k]);
                } catch (const std::bad_alloc &) {
                    packed[(size_t)k] = PackedInst();
                    packed[(size_t)k].code = PHIA_ENOMEM;
                    packed[(size_t)k].msg = "no host memory";
                }
            }
        };
        std::vector<std::thread> workers;
        workers.reserve((size_t)nthreads);
        for (int t = 1; t < nthreads && start_thread(workers, work); ++t) {}
        work();
        for (std::thread &t : workers) t.join();
    }
    size_t tot_sl = 0, tot_ent = 0, tot_pos = 0, tot_inv = 0, tot_h = 0, tot_dj = 0;
    bool all_cand = true;
    for (int k = 0; k < count; ++k) {
        if (packed[(size_t)k].code != PHIA_OK)
            return cleanup(bfail(packed[(size_t)k].code, "%s", packed[(size_t)k].msg.c_str()));
        tot_sl += packed[(size_t)k].slice.size();
        tot_ent += packed[(size_t)k].val.size();
        tot_pos += packed[(size_t)k].row_of.size();
        tot_inv += packed[(size_t)k].pos_of.size();
        all_cand &= packed[(size_t)k].small_op || !packed[(size_t)k].dense.empty();
        if (packed[(size_t)k].small_op || !packed[(size_t)k].dense.empty()) {
            tot_h += (size_t)d[k].N;
            tot_dj += (size_t)d[k].N * d[k].N;
        }
    }
    if (tot_ent / 32 > (size_t)INT32_MAX) return cleanup(bfail(PHIA_ERANGE, "too many couplings in one batch"));
    std::vector<int32_t> slice, col, hk2, row_of, pos_of, hk;
    std::vector<uint32_t> val;
    std::vector<int8_t> dj;
    if (count > 1) {
        col.reserve(4 * tot_ent);
        val.reserve(tot_ent);
    }
    slice.reserve(tot_sl); hk2.reserve(2 * tot_pos);
    row_of.reserve(tot_pos); pos_of.reserve(tot_inv); hk.reserve(tot_h); dj.reserve(tot_dj);
    for (int k = 0; k < count; ++k) {
        const phia_instance_desc &x = d[k];
        PackedInst &pk = packed[(size_t)k];
        const int n = x.N;
        b->N.push_back(n);
        b->frac.push_back(x.frac_bits);
        b->inst_id.push_back(x.instance_id);
        b->h_off.push_back((int64_t)hk.size());
        b->targets.push_back(x.has_target ? (long long)x.target_k : LLONG_MIN);
        b->any_target |= x.has_target != 0;
        b->max_words = std::max<int>(b->max_words, (int)words_of(n));
        if (pk.small_op) {
            b->dense_pub.push_back(k);
            b->dense_joff.push_back((int64_t)dj.size());
            b->dense_op.push_back(pk.small_op);
            dj.insert(dj.end(), x.J_k, x.J_k + (size_t)n * n);
            hk.insert(hk.end(), x.h_k, x.h_k + n);
            continue;
        }
        b->csr_pub.push_back(k);
        if (all_cand) {
            b->cand_joff.push_back((int64_t)dj.size());
            dj.insert(dj.end(), pk.dense.begin(), pk.dense.end());
            hk.insert(hk.end(), x.h_k, x.h_k + n);
        }
        CsrInst in{};
        in.N = n;
        in.Np = round_up(n, 32);
        in.inst_id = x.instance_id;
        in.q = ldexpf(1.0f, -x.frac_bits);
        in.wide = pk.wide;
        in.slice_base = b->total_slices;
        in.slice_off = (int64_t)slice.size();
        in.pos_off = (int64_t)row_of.size();
        in.inv_off = (int64_t)pos_of.size();
        const int32_t ent0 = (int32_t)(val.size() / 32);
        const int longest = 4 * pk.slice[1];           // rows are sorted by length
        for (int32_t e : pk.slice) slice.push_back(ent0 + e);
        if (count == 1) {
            col = std::move(pk.col);
            val = std::move(pk.val);
        } else {
            col.insert(col.end(), pk.col.begin(), pk.col.end());
            val.insert(val.end(), pk.val.begin(), pk.val.end());
        }
        hk2.insert(hk2.end(), pk.hk2.begin(), pk.hk2.end());
        row_of.insert(row_of.end(), pk.row_of.begin(), pk.row_of.end());
        pos_of.insert(pos_of.end(), pk.pos_of.begin(), pk.pos_of.end());
        pk = PackedInst();
        b->shape.max_np = std::max(b->shape.max_np, in.Np);
        b->total_slices += in.Np / 32;
        b->shape.rows += n;
        b->shape.longest = std::max(b->shape.longest, longest);
        b->inst.push_back(in);
    }
    std::vector<int32_t> rows_ptr, rows_col, rows_h;
    std::vector<int8_t> rows_val;
    std::vector<CsrRowsBlock> rows_blocks;
    b->shape.degree = b->shape.rows ? 4.0 * (double)(slice.empty() ? 0 : slice.back()) * 32.0 / (double)b->shape.rows : 0.0;
    if (rows_form_possible(b->shape)) {
        const size_t most = (size_t)(b->shape.degree * (double)b->shape.rows) + 8 * (size_t)b->shape.rows;
        rows_col.reserve(most);
        rows_val.reserve(most);
        int64_t row_base = 0;
        for (size_t c = 0; c < b->inst.size(); ++c) {
            const phia_instance_desc &x = d[b->csr_pub[c]];
            CsrRowsInst ri{};
            ri.N = x.N;
            ri.inst_id = x.instance_id;
            ri.q = b->inst[c].q;
            ri.rp_off = (int64_t)rows_ptr.size();
            ri.nz_off = (int64_t)rows_col.size();
            ri.h_off = (int64_t)rows_h.size();
            ri.row_base = row_base;
            row_base += x.N;
            append_rows(x, rows_ptr, rows_col, rows_val);
            rows_h.insert(rows_h.end(), x.h_k, x.h_k + x.N);
            for (int i0 = 0; i0 < x.N; i0 += 64) rows_blocks.push_back(CsrRowsBlock{(int32_t)c, i0});
            b->rows_inst.push_back(ri);
        }
        b->rows_blocks = (int32_t)rows_blocks.size();
    }
    for (int l = 0; l < 4; ++l)
        for (size_t c = 0; c <= b->inst.size(); ++c) {
            b->first_block[l].push_back((int32_t)b->blocks.size());
            if (c < b->inst.size())
                for (int ns = b->inst[c].Np / 32, s0 = 0; s0 < ns; s0 += 1 << l) {
                    const int32_t *e = slice.data() + b->inst[c].slice_off;
                    b->blocks.push_back(CsrBlock{(int32_t)c, s0, e[std::min(ns, s0 + (1 << l))] - e[s0]});
                }
        }
    int dev_count = 0;
    if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count == 0)
        return cleanup(bfail(PHIA_ECUDA, "no CUDA device available"));
    if (o.device < 0 || o.device >= dev_count) return cleanup(bfail(PHIA_EINVAL, "device %d out of range", o.device));
    if (cudaSetDevice(o.device) != cudaSuccess) return cleanup(bfail(PHIA_ECUDA, "cudaSetDevice failed"));
    b->device = o.device;
    b->stream = (cudaStream_t)o.stream;
    bool ok = true;
    auto al = [&](void **dst, size_t bytes) {
        if (ok && pool_alloc(dst, bytes, b->device, b->stream) != cudaSuccess) ok = false;
    };
    auto up = [&](void **dst, const void *src, size_t bytes) {
        al(dst, bytes);
        if (ok && bytes && cudaMemcpyAsync(*dst, src, bytes, cudaMemcpyHostToDevice, b->stream) != cudaSuccess) ok = false;
    };
    up((void **)&b->d_slice, slice.data(), slice.size() * 4);
    b->col16 = b->shape.max_np <= 16384;
    std::vector<uint16_t> col16;
    if (b->col16) col16.assign(col.begin(), col.end());
    if (b->col16) up(&b->d_col, col16.data(), col16.size() * 2);
    else up(&b->d_col, col.data(), col.size() * 4);
    up((void **)&b->d_val, val.data(), val.size() * 4);
    up((void **)&b->d_hk2, hk2.data(), hk2.size() * 4);
    up((void **)&b->d_rowof, row_of.data(), row_of.size() * 4);
    up((void **)&b->d_posof, pos_of.data(), pos_of.size() * 4);
    up((void **)&b->d_hk, hk.data(), hk.size() * 4);
    up((void **)&b->d_blocks, b->blocks.data(), b->blocks.size() * sizeof(CsrBlock));
    up((void **)&b->d_targets, b->targets.data(), b->targets.size() * sizeof(long long));
    up((void **)&b->d_dJ, dj.data(), dj.size());
    if (!b->rows_inst.empty()) {
        up((void **)&b->d_rows_ptr, rows_ptr.data(), rows_ptr.size() * 4);
        up((void **)&b->d_rows_col, rows_col.data(), rows_col.size() * 4);
        up((void **)&b->d_rows_val, rows_val.data(), rows_val.size());
        up((void **)&b->d_rows_h, rows_h.data(), rows_h.size() * 4);
        up((void **)&b->d_rows_blocks, rows_blocks.data(), rows_blocks.size() * sizeof(CsrRowsBlock));
        al((void **)&b->d_rows_inst, sizeof(CsrRowsInst) * b->rows_inst.size());
    }
    al((void **)&b->d_inst, sizeof(CsrInst) * b->inst.size());
    al((void **)&b->d_sets, sizeof(CsrSet) * b->inst.size());
    al((void **)&b->d_min_hit, 8);
    al((void **)&b->d_start_ns, 8);
    al((void **)&b->d_iters, 8);
    al((void **)&b->d_err, 4);
    al((void **)&b->d_ctl, sizeof(IterCtl));
    al((void **)&b->d_sync, 4 * sizeof(unsigned));
    if (ok && cudaMemsetAsync(b->d_start_ns, 0, 8, b->stream) != cudaSuccess) ok = false;
    if (ok && cudaStreamSynchronize(b->stream) != cudaSuccess) ok = false;    // the host arrays end here
    if (ok) b->graphs = step_graphs_new();
    if (ok && (cudaEventCreate(&b->ev0) != cudaSuccess || cudaEventCreate(&b->ev1) != cudaSuccess)) ok = false;
    if (!ok) {
        cudaGetLastError();
        return cleanup(bfail(PHIA_ENOMEM, "device allocation or upload failed"));
    }
    *out = b;
    return PHIA_OK;
}

int batch_create(phia_batch_s **out, int32_t count, const phia_instance_desc *d, const phia_opts *opts) {
    if (!out) return bfail(PHIA_EINVAL, "out is NULL");
    *out = nullptr;
    phia_batch_s *b = nullptr;
    try {
        return create_batch(b, out, count, d, opts);
    } catch (const std::bad_alloc &) {
        phia_batch_destroy(b);
        return bfail(PHIA_ENOMEM, "no host memory for the batch");
    }
}

int batch_run(phia_batch_s *b, const phia_schedule *sched, int32_t R_real, int64_t t0, int64_t steps, int64_t total,
              uint64_t seed, const float *x_in, float *x_out, const float *v_in, float *v_out, int reset,
              const int8_t *spins_in, int32_t *field_out, int64_t *energy_out) try {
    if (!b) return bfail(PHIA_EINVAL, "batch is NULL");
    const bool field_mode = spins_in != nullptr;
    if (!field_mode) {
        if (!sched) return bfail(PHIA_EINVAL, "schedule is NULL");
        if (!(sched->eps > 0.0f) || !(sched->gamma > 0.0f) || sched->refresh < 0 || (sched->deriv != 0 && sched->deriv != 1) ||
            sched->reserved != 0)
            return bfail(PHIA_EINVAL, "invalid schedule");
        if (sched->accept_test != 0)
            return bfail(PHIA_ENOTSUP, "schedule.accept_test = 1 runs on the resident tcgen05 and FP32 paths only");
        if (steps < 1 || t0 < 0 || total < t0 + steps) return bfail(PHIA_EINVAL, "need steps >= 1, t0 + steps <= total");
        if (total > ((int64_t)1 << 31)) return bfail(PHIA_ERANGE, "total_steps must be < 2^31");
    }
    if (R_real < 1) return bfail(PHIA_EINVAL, "replicas must be >= 1");
    const bool by_rows = !field_mode && b->d_rows_inst && rows_form(b->shape, R_real);
    const int R = round_up(R_real, by_rows ? 256 : 32);
    BCU(cudaSetDevice(b->device));
    if (!field_mode && !reset && (!b->ran || b->R_real != R_real))
        return bfail(PHIA_ESTATE, "reset_best = 0 needs a previous run with the same replica count");
    int rc = ensure_state(b, R);
    if (rc) return rc;
    b->R_real = R_real;
    layout(b, R);
    const int ncsr = (int)b->inst.size();
    if (field_mode && !b->dense_pub.empty()) return bfail(PHIA_ENOTSUP, "field-only runs take CSR instances");
    if ((x_in || x_out) && !b->dense_pub.empty())
        return bfail(PHIA_ENOTSUP, "runs from a given state take CSR instances");
    if (ncsr > 0)
        BCU(cudaMemcpyAsync(b->d_inst, b->inst.data(), sizeof(CsrInst) * ncsr, cudaMemcpyHostToDevice, b->stream));
    if (by_rows)
        BCU(cudaMemcpyAsync(b->d_rows_inst, b->rows_inst.data(), sizeof(CsrRowsInst) * ncsr, cudaMemcpyHostToDevice, b->stream));
    // Whether the sparse members gather, or run on the resident kernels (below).
    bool gathers = ncsr > 0;
    if (ncsr > 0 && !b->cand_joff.empty() && !field_mode && (b->count == 1 || (!x_in && !x_out))) {
        int sms = 0;
        BCU(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device));
        double us = 0.0;
        for (const CsrInst &in : b->inst)
            us += in.N <= warp_small_auto_n() ? warp_small_estimate(in.N, R_real, sms) : cluster_small_estimate(in.N, R_real, kOpBF16, sms, 5.0);
        gathers = us > 5.0;
    }
    if (gathers && !by_rows && !field_mode && b->sets_R != R) {      // host work: before the run's time begins
        rc = make_sets(b, R);
        if (rc) return rc;
    }
    const int64_t reps = (int64_t)R * b->count;
    int64_t nbits = 0;
    for (int k = 0; k < b->count; ++k) nbits += (int64_t)R * words_of(b->N[k]);
    int launches = 0;
    if (reset && !field_mode) {
        const int64_t n = std::max(reps, nbits);
        batch_reset_records<<<(unsigned)((n + 255) / 256), 256, 0, b->stream>>>(
            reps, nbits, b->d_best_e, b->d_best_step, b->d_hit, b->d_bits, b->d_hit_ns, b->d_start_ns);
        BCU(cudaGetLastError());
        ++launches;
    }
    BCU(cudaMemsetAsync(b->d_min_hit, 0xFF, 8, b->stream));
    BCU(cudaMemsetAsync(b->d_iters, 0, 8, b->stream));
    BCU(cudaMemsetAsync(b->d_err, 0, 4, b->stream));
    b->waits_checked = false;
    CsrArgs C;
    memset(&C, 0, sizeof C);
    RunArgs &a = C.a;
    a.R = R;
    a.t0 = t0; a.nsteps = field_mode ? 1 : steps; a.T_total = field_mode ? 1 : total;
    if (!field_mode) {
        a.beta0 = sched->beta0; a.beta1 = sched->beta1; a.eps = sched->eps; a.gamma = sched->gamma;
        a.refresh = sched->refresh;
        a.deriv = sched->deriv;
        a.has_target = (sched->has_target || b->any_target) ? 1 : 0;
        a.stop_at_target = sched->stop_at_target;
        a.target = sched->target_k;
    }
    a.seed = seed;
    a.field_mode = field_mode ? 1 : 0;
    a.spins_in = spins_in; a.field_out = field_out; a.energy_out = energy_out;
    a.best_e = b->d_best_e; a.best_step = b->d_best_step; a.hit_step = b->d_hit;
    a.hit_ns = b->d_hit_ns;
    a.min_hit = b->d_min_hit; a.replica_iters = b->d_iters; a.err = b->d_err;
    C.inst = b->d_inst; C.count = ncsr;
    C.blocks = b->d_blocks;
    C.sets = b->d_sets;
    C.max_np = b->shape.max_np;
    C.slice = b->d_slice; C.col = b->d_col; C.col16 = b->col16 ? 1 : 0; C.val = b->d_val; C.hk = b->d_hk2;
    C.row_of = b->d_rowof; C.pos_of = b->d_posof;
    C.X = b->d_X; C.V = b->d_V;
    C.x_in = x_in; C.v_in = v_in; C.x_out = x_out; C.v_out = v_out;
    C.S = b->d_S;
    C.total_swords = b->total_slices * 32 * (R / 32);
    C.Esum = b->d_Esum; C.flags = b->d_flags; C.total_reps = reps;
    C.best_bits = b->d_bits;
    // per-instance targets: the instance's own, else the schedule's (CSR members, by CSR index)
    auto target_of = [&](int k) {
        return b->targets[(size_t)k] != LLONG_MIN ? b->targets[(size_t)k]
                                                  : (sched->has_target ? (long long)sched->target_k : LLONG_MIN);
    };
    if (!field_mode && (b->any_target) && ncsr > 0) {
        std::vector<long long> tg((size_t)ncsr);
        for (int c = 0; c < ncsr; ++c) tg[(size_t)c] = target_of(b->csr_pub[(size_t)c]);
        BCU(cudaMemcpyAsync(b->d_targets, tg.data(), tg.size() * sizeof(long long), cudaMemcpyHostToDevice, b->stream));
        BCU(cudaStreamSynchronize(b->stream));
        C.targets = b->d_targets;
    }
    C.R = R; C.R_real = R_real;
    C.max_words = b->max_words;
    C.total_slices = b->total_slices;
    // Members on the resident kernels: a table of CTAs or clusters (8 replicas each) per size
    // class, every instance's own couplings, field, scale, Philox id, target and records.  Up to 240
    // spins the warp-level kernel (classes, as its register use grows with the size it is built
    // for; 32 dense members of 200 spins x 512 replicas: 18.8 us an iteration on the tcgen05 one); dense members
    // above on the resident tcgen05 kernel (256 spins x 512: 20.0 us against 22.4 on the warp-level one),
    // sparse ones on the cluster kernel.  Sparse members run here where their estimated iterations
    // take less together than the gather's, which no instance takes below 7 us (launch, records, the
    // copy of the spins and a slice come one after the other).
    enum { kWarp, kTcgen05, kCluster };
    struct SmallGroup {
        size_t begin, end;       // in small_host
        int nmax, kernel, op;
    };
    std::vector<SmallGroup> groups;
    const bool resident = ncsr > 0 && !gathers;
    if (!b->dense_pub.empty() || resident) {
        b->small_host.clear();
        struct Class {
            int above, nmax, kernel, op;     // op: of the dense members that kTcgen05 takes
        };
        const Class classes[] = {{0, 64, kWarp, 0},
                                 {64, 128, kWarp, 0},
                                 {128, 240, kWarp, 0},
                                 {240, 256, kTcgen05, kOpE4M3},
                                 {240, 256, kTcgen05, kOpBF16},
                                 {256, 384, kTcgen05, kOpE4M3},
                                 {240, 384, kCluster, 0},
                                 {384, 512, kCluster, 0}};
        for (const Class &cls : classes) {
            const size_t beg = b->small_host.size();
            int nmax = 0;
            auto add = [&](int k, int64_t joff) {
                const int n = b->N[(size_t)k];
                if (n <= cls.above || n > cls.nmax) return;
                nmax = std::max(nmax, n);
                for (int r0 = 0; r0 < R_real; r0 += 8) {
                    SmallCta c{};
                    c.Jk = b->d_dJ + joff;
                    c.hk = b->d_hk + b->h_off[(size_t)k];
                    c.N = n;
                    c.W = (int32_t)words_of(n);
                    c.inst = b->inst_id[(size_t)k];
                    c.q = ldexpf(1.0f, -b->frac[(size_t)k]);
                    c.rbase = r0;
                    c.rec_off = (int64_t)k * R;
                    c.bits_off = b->bits_pub[(size_t)k];
                    c.target = target_of(k);
                    b->small_host.push_back(c);
                }
            };
            if (cls.kernel != kCluster)
                for (size_t m = 0; m < b->dense_pub.size(); ++m)
                    if (cls.kernel == kWarp || b->dense_op[m] == cls.op) add(b->dense_pub[m], b->dense_joff[m]);
            if (cls.kernel != kTcgen05 && resident)
                for (size_t m = 0; m < b->csr_pub.size(); ++m) add(b->csr_pub[m], b->cand_joff[m]);
            if (b->small_host.size() > beg) groups.push_back(SmallGroup{beg, b->small_host.size(), nmax, cls.kernel, cls.op});
        }
        auto take = [&](SmallCta **q, size_t bytes) {
            return pool_alloc((void **)q, bytes, b->device, b->stream) == cudaSuccess;
        };
        if (!grow_table(b->d_small, b->small_cap, b->small_host.size(), take, [&](SmallCta *q) { pool_free(q, b->stream); })) {
            cudaGetLastError();
            return bfail(PHIA_ENOMEM, "CTA table allocation failed");
        }
        BCU(cudaMemcpyAsync(b->d_small, b->small_host.data(), b->small_host.size() * sizeof(SmallCta),
                            cudaMemcpyHostToDevice, b->stream));
    }
    BCU(cudaEventRecord(b->ev0, b->stream));
    C.ctl = b->d_ctl;
    C.sync = b->d_sync;
    C.persistent = (b->csr_mode == 1 && !field_mode) ? 1 : 0;
    if (by_rows) {
        CsrRowsArgs W;
        memset(&W, 0, sizeof W);
        W.a = C.a;
        W.inst = b->d_rows_inst; W.count = ncsr;
        W.blocks = b->d_rows_blocks; W.nblocks = b->rows_blocks;
        W.row_ptr = b->d_rows_ptr; W.col = b->d_rows_col; W.val = b->d_rows_val; W.hk = b->d_rows_h;
        W.X = C.X; W.V = C.V;
        W.x_in = x_in; W.v_in = v_in; W.x_out = x_out; W.v_out = v_out;
        W.S = C.S; W.total_swords = b->shape.rows * (R / 32);
        W.Esum = C.Esum; W.flags = C.flags; W.total_reps = reps;
        W.best_bits = C.best_bits;
        W.targets = C.targets;
        W.R = R; W.R_real = R_real;
        W.max_words = C.max_words;
        W.total_rows = b->shape.rows;
        W.ctl = C.ctl; W.persistent = C.persistent; W.sync = C.sync;
        cudaError_t e = launch_csr_rows(W, b->graphs, b->stream, &launches);
        if (e != cudaSuccess) return bfail(PHIA_ECUDA, "kernel launch failed: %s", cudaGetErrorString(e));
    } else if (gathers) {
        C.nsets = (int32_t)b->sets.size();
        cudaError_t e = launch_csr(C, b->set_max, b->graphs, b->stream, &launches);
        if (e != cudaSuccess) return bfail(PHIA_ECUDA, "kernel launch failed: %s", cudaGetErrorString(e));
    }
    for (const SmallGroup &grp : groups) {
        RunArgs ad = a;
        ad.R = R_real;
        ad.best_bits = b->d_bits;        // the CSR path keeps its best states in C.best_bits
        if (!ad.best_e || !ad.best_step || !ad.hit_step || !ad.hit_ns || !ad.best_bits || !ad.replica_iters || !ad.err)
            return bfail(PHIA_ECUDA, "internal: a record array of the dense launch is missing");
        ad.small_cta = b->d_small + grp.begin;
        ad.small_ctas = (int32_t)(grp.end - grp.begin);
        ad.has_target = b->any_target || sched->has_target;
        ad.x_in = x_in; ad.v_in = v_in; ad.x_out = x_out; ad.v_out = v_out;
        cudaError_t e = grp.kernel == kWarp      ? launch_warp_small_batch(ad, grp.nmax, b->stream)
                        : grp.kernel == kTcgen05 ? launch_tc_small_batch(ad, grp.op, grp.nmax, b->stream)
                                                 : launch_cluster_batch(ad, grp.nmax, b->stream);
        if (e != cudaSuccess) return bfail(PHIA_ECUDA, "kernel launch failed: %s", cudaGetErrorString(e));
        ++launches;
    }
    BCU(cudaEventRecord(b->ev1, b->stream));
    if (!field_mode) {
        b->ran = true;
        b->R = R;
        b->last_steps = steps;
        b->last_launches = launches;
        b->last_stop = sched->stop_at_target;
    }
    return PHIA_OK;
} catch (const std::bad_alloc &) {
    return bfail(PHIA_ENOMEM, "no host memory for the run");
}

// Per-replica records of one instance (first R_real replicas).
int batch_records(phia_batch_s *b, int inst, std::vector<int64_t> &be, std::vector<int64_t> &bs,
                  std::vector<int64_t> &hs) {
    if (!b->ran) return bfail(PHIA_ESTATE, "no run on this batch yet");
    if (inst < 0 || inst >= b->count) return bfail(PHIA_EINVAL, "instance %d out of range", inst);
    BCU(cudaSetDevice(b->device));
    BCU(cudaStreamSynchronize(b->stream));
    if (!b->waits_checked) {        // the finished run's error flag, once
        int32_t err = 0;
        BCU(cudaMemcpy(&err, b->d_err, 4, cudaMemcpyDeviceToHost));
        if (err) return bfail(PHIA_ETIMEOUT, "a bounded device wait expired during the run");
        b->waits_checked = true;
    }
    const size_t n = (size_t)b->R_real, off = (size_t)inst * b->R;
    std::vector<int64_t> raw(3 * n);            // the three records of the instance in one copy
    BCU(cudaMemcpy2D(raw.data(), n * 8, b->d_best_e + off, (size_t)(b->d_best_step - b->d_best_e) * 8, n * 8, 3,
                     cudaMemcpyDeviceToHost));
    be.assign(raw.begin(), raw.begin() + n);
    bs.assign(raw.begin() + n, raw.begin() + 2 * n);
    hs.assign(raw.begin() + 2 * n, raw.end());
    return PHIA_OK;
}

int batch_pick(const phia_batch_s *b, const std::vector<int64_t> &be, const std::vector<int64_t> &bs,
               const std::vector<int64_t> &hs) {
    int best = -1;
    if (b->last_stop) {
        for (int r = 0; r < (int)hs.size(); ++r)
            if (hs[r] >= 0 && (best < 0 || hs[r] < hs[best])) best = r;
        if (best >= 0) return best;
    }
    for (int r = 0; r < (int)be.size(); ++r) {
        if (bs[r] < 0) continue;
        if (best < 0 || be[r] < be[best] || (be[r] == be[best] && bs[r] < bs[best])) best = r;
    }
    return best;
}

int batch_bits(phia_batch_s *b, int inst, int r, uint32_t *dst, int nreps) {
    // bits of replicas r .. r+nreps-1 of one instance
    int64_t off = 0;
    for (int k = 0; k < inst; ++k) off += (int64_t)b->R * words_of(b->N[k]);
    const int64_t W = words_of(b->N[inst]);
    BCU(cudaMemcpy(dst, b->d_bits + off + (int64_t)r * W, (size_t)nreps * W * 4, cudaMemcpyDeviceToHost));
    return PHIA_OK;
}

int batch_best(phia_batch_s *b, int inst, int64_t *energy_k, int8_t *spins) {
    std::vector<int64_t> be, bs, hs;
    int rc = batch_records(b, inst, be, bs, hs);
    if (rc) return rc;
    const int r = batch_pick(b, be, bs, hs);
    if (r < 0) return bfail(PHIA_ESTATE, "no replica recorded a state");
    if (energy_k) *energy_k = be[r];
    if (spins) {
        const int n = b->N[inst];
        std::vector<uint32_t> w(words_of(n));
        rc = batch_bits(b, inst, r, w.data(), 1);
        if (rc) return rc;
        for (int i = 0; i < n; ++i) spins[i] = ((w[i >> 5] >> (i & 31)) & 1u) ? 1 : -1;
    }
    return PHIA_OK;
}

int batch_replica_results(phia_batch_s *b, int inst, int32_t R, int64_t *be_out, int64_t *bs_out, int64_t *hs_out,
                          uint32_t *bits_out) {
    std::vector<int64_t> be, bs, hs;
    int rc = batch_records(b, inst, be, bs, hs);
    if (rc) return rc;
    if (R != b->R_real) return bfail(PHIA_EINVAL, "replicas (%d) differs from the last run (%d)", R, b->R_real);
    if (be_out) memcpy(be_out, be.data(), (size_t)R * 8);
    if (bs_out) memcpy(bs_out, bs.data(), (size_t)R * 8);
    if (hs_out) memcpy(hs_out, hs.data(), (size_t)R * 8);
    if (bits_out) return batch_bits(b, inst, 0, bits_out, R);
    return PHIA_OK;
}

int batch_stats(phia_batch_s *b, int inst, phia_stats *out) {
    if (!out) return bfail(PHIA_EINVAL, "NULL argument");
    memset(out, 0, sizeof *out);
    std::vector<int64_t> be, bs, hs;
    int rc = batch_records(b, inst < 0 ? 0 : inst, be, bs, hs);
    if (rc) return rc;
    unsigned long long iters = 0;
    BCU(cudaMemcpy(&iters, b->d_iters, 8, cudaMemcpyDeviceToHost));
    float ms = 0.f;
    BCU(cudaEventElapsedTime(&ms, b->ev0, b->ev1));
    int64_t spins_total = 0;
    for (int k = 0; k < b->count; ++k) spins_total += b->N[k];
    out->replicas = b->R_real;
    out->steps = b->last_steps;
    // padded replicas excluded: every instance runs R_real real replicas
    out->spin_updates = (int64_t)b->R_real * b->last_steps * (inst < 0 ? spins_total : b->N[inst]);
    const int r = batch_pick(b, be, bs, hs);
    out->best_replica = r;
    out->best_energy_k = r >= 0 ? be[r] : 0;
    out->best_step = r >= 0 ? bs[r] : -1;
    out->hit_step = -1;
    out->hit_replica = -1;
    for (int k = 0; k < (int)hs.size(); ++k)
        if (hs[k] >= 0 && (out->hit_step < 0 || hs[k] < out->hit_step)) { out->hit_step = hs[k]; out->hit_replica = k; }
    out->hit_ns = -1;
    if (out->hit_replica >= 0) {
        uint64_t t_hit = 0, t_start = 0;
        BCU(cudaMemcpy(&t_hit, b->d_hit_ns + (size_t)(inst < 0 ? 0 : inst) * b->R + out->hit_replica, 8,
                       cudaMemcpyDeviceToHost));
        BCU(cudaMemcpy(&t_start, b->d_start_ns, 8, cudaMemcpyDeviceToHost));
        if (t_hit >= t_start && t_start != 0) out->hit_ns = (int64_t)(t_hit - t_start);
    }
    out->device_ms = ms;
    out->path = b->inst.empty() ? PHIA_PATH_TC : PHIA_PATH_CSR;   // sparse members, whichever kernel ran them
    out->kernel_launches = b->last_launches;
    (void)iters;
    return PHIA_OK;
}

}  // namespace phia

extern "C" {

int phia_batch_create(phia_batch_t **out, int32_t count, const phia_instance_desc *descs, const phia_opts *opts) {
    return batch_create(out, count, descs, opts);
}

int phia_batch_anneal(phia_batch_t *b, const phia_schedule *sched, int32_t replicas, int64_t steps, uint64_t seed) {
    return batch_run(b, sched, replicas, 0, steps, steps, seed, nullptr, nullptr, nullptr, nullptr, 1, nullptr, nullptr,
                     nullptr);
}

int phia_batch_best(phia_batch_t *b, int32_t instance, int64_t *energy_k, int8_t *spins) {
    if (!b) return bfail(PHIA_EINVAL, "batch is NULL");
    return batch_best(b, instance, energy_k, spins);
}

int phia_batch_replica_results(phia_batch_t *b, int32_t instance, int32_t replicas, int64_t *best_energy_k,
                               int64_t *best_step, int64_t *hit_step, uint32_t *best_bits) {
    if (!b) return bfail(PHIA_EINVAL, "batch is NULL");
    return batch_replica_results(b, instance, replicas, best_energy_k, best_step, hit_step, best_bits);
}

int phia_batch_stats_get(phia_batch_t *b, phia_stats *out) {
    if (!b) return bfail(PHIA_EINVAL, "batch is NULL");
    return batch_stats(b, -1, out);
}

int phia_batch_autotune(phia_batch_t *b, const phia_schedule *sched, int32_t replicas, int32_t probe_iters,
                        phia_tune_result *out) {
    if (!b || !sched) return bfail(PHIA_EINVAL, "NULL argument");
    if (replicas < 1 || probe_iters < 1) return bfail(PHIA_EINVAL, "need replicas >= 1 and probe_iters >= 1");
    float best_ms = 1e30f, worst_ms = 0.f;
    int best_mode = b->csr_mode;
    const int saved = b->csr_mode;
    for (int mode : {1, 2}) {
        b->csr_mode = mode;
        float ms = 0.f;
        for (int rep = 0; rep < 2; ++rep) {   // the first run warms up
            int rc = batch_run(b, sched, replicas, 0, probe_iters, probe_iters, 1, nullptr, nullptr, nullptr, nullptr, 1,
                               nullptr, nullptr, nullptr);
            if (rc) { b->csr_mode = saved; return rc; }
            BCU(cudaEventSynchronize(b->ev1));
            BCU(cudaEventElapsedTime(&ms, b->ev0, b->ev1));
        }
        if (ms < best_ms) { best_ms = ms; best_mode = mode; }
        worst_ms = std::max(worst_ms, ms);
    }
    b->csr_mode = best_mode;
    if (out) {
        memset(out, 0, sizeof *out);
        out->tc_kernel = best_mode;
        out->candidates = 2;
        out->best_us_per_iter = 1000.f * best_ms / probe_iters;
        out->worst_us_per_iter = 1000.f * worst_ms / probe_iters;
    }
    return PHIA_OK;
}

int phia_batch_sync(phia_batch_t *b) {
    if (!b) return bfail(PHIA_EINVAL, "batch is NULL");
    BCU(cudaSetDevice(b->device));
    BCU(cudaStreamSynchronize(b->stream));
    return PHIA_OK;
}

void phia_batch_destroy(phia_batch_t *b) {
    if (!b) return;
    cudaSetDevice(b->device);
    cudaStreamSynchronize(b->stream);
    free_state(b);
    for (void *p : {(void *)b->d_inst, (void *)b->d_blocks, (void *)b->d_slice, b->d_col, (void *)b->d_val,
                    (void *)b->d_sets, (void *)b->d_hk2, (void *)b->d_rowof, (void *)b->d_posof, (void *)b->d_hk,
                    (void *)b->d_targets, (void *)b->d_min_hit, (void *)b->d_start_ns, (void *)b->d_iters,
                    (void *)b->d_rows_inst, (void *)b->d_rows_blocks, (void *)b->d_rows_ptr, (void *)b->d_rows_col,
                    (void *)b->d_rows_val, (void *)b->d_rows_h, (void *)b->d_err, (void *)b->d_dJ, (void *)b->d_small, (void *)b->d_sync, (void *)b->d_ctl})
        pool_free(p, b->stream);
    step_graphs_free(b->graphs);
    if (b->ev0) cudaEventDestroy(b->ev0);
    if (b->ev1) cudaEventDestroy(b->ev1);
    delete b;
}

}  // extern "C"
