// api.cpp -- host side of libfewsum.so: the C ABI declared in include/fewsum.h.
//
// Responsibilities: input validation, the planning step (mode -> harmonic slot layout,
// segment sample ranges, CTA slices of equal pass cost), device memory from a context-owned
// stream-ordered pool with an HBM budget, plan uploads through pinned staging buffers, kernel
// launches, CUDA-graph capture of batches, and the device error latch.  No arithmetic of the
// waveform itself happens here; every numerical step runs in the kernels.
#include "../../include/fewsum.h"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <set>
#include <tuple>
#include <unordered_map>
#include <vector>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "fewsum_internal.h"

using namespace fewsum;

// ------------------------------------------------------------------------------ utilities

namespace {

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

#define FEW_CUDA_TRY(expr)                                  \
    do {                                                    \
        cudaError_t e__ = (expr);                           \
        if (e__ != cudaSuccess) {                           \
            (void)cudaGetLastError();                       \
            return e__ == cudaErrorMemoryAllocation ? FEW_ERR_NOMEM : FEW_ERR_CUDA; \
        }                                                   \
    } while (0)

// Pinned host staging blocks for plan uploads, reused once their copy has completed.
struct PinnedPool {
    struct Block {
        void *p = nullptr;
        size_t bytes = 0;
        cudaEvent_t ev = nullptr;
        bool pending = false;
    };
    std::vector<Block> blocks;

    ~PinnedPool() { release(); }
    void release()
    {
        for (auto &b : blocks) {
            if (b.ev) cudaEventDestroy(b.ev);
            if (b.p) cudaFreeHost(b.p);
        }
        blocks.clear();
    }
    // A block of at least `bytes` that no queued copy still reads.
    Block *acquire(size_t bytes)
    {
        for (auto &b : blocks) {
            if (b.bytes < bytes) continue;
            if (b.pending) {
                if (cudaEventQuery(b.ev) != cudaSuccess) continue;
                b.pending = false;
            }
            return &b;
        }
        Block nb;
        nb.bytes = align_up(std::max(bytes, (size_t)1 << 16), 4096);
        if (cudaHostAlloc(&nb.p, nb.bytes, cudaHostAllocDefault) != cudaSuccess) {
            (void)cudaGetLastError();
            return nullptr;
        }
        if (cudaEventCreateWithFlags(&nb.ev, cudaEventDisableTiming) != cudaSuccess) {
            (void)cudaGetLastError();
            cudaFreeHost(nb.p);
            return nullptr;
        }
        blocks.push_back(nb);
        return &blocks.back();
    }
};

}  // namespace

struct few_traj;
struct few_batch;

// Reduced basis (Sec. 3.E): FP64 B, its transposed Gram matrix in FP64 and FP32, and the split
// fp16 operand of the tensor-core product, in one device allocation; the FP64 product's digit slices in
// another, which is given up when the context has no room for something else (give_up_slices).
struct few_basis {
    few_ctx *ctx = nullptr;
    int Nb = 0, N = 0;
    void *dmem = nullptr;
    const double *bre = nullptr, *bim = nullptr;
    const double2 *gt64 = nullptr;
    const float2 *gt32 = nullptr;
    const int *bexp = nullptr;
    const unsigned char *bpack = nullptr;
    void *slices = nullptr;  // exponents, then the slices (null: no room for them)
    const int *bexp64 = nullptr;
    const unsigned char *bpack64 = nullptr;
    mutable bool captured = false;  // a captured graph of the caller's reads the slices: they stay
};

struct few_ctx {
    int device = 0;
    int sm_count = 0;
    size_t budget = 0;  // 0: unlimited
    size_t in_use = 0;
    cudaMemPool_t pool = nullptr;
    cudaStream_t internal = nullptr;
    // second streams for work beside a call's main chain (the scalar chain's phase anchors beside its
    // harmonics and fold; the reduced-basis scale of more than 128 vectors beside its pack), each with its fork and
    // join events; taken in turn, so calls on different user streams seldom share one
    struct SideLane {
        cudaStream_t s = nullptr;
        cudaEvent_t fork = nullptr, join = nullptr;
    } lanes[4];
    unsigned lane_next = 0;
    unsigned *d_err = nullptr;
    std::recursive_mutex mu;
    std::unordered_map<void *, size_t> sizes;
    std::set<few_traj *> trajs;
    std::set<few_batch *> batches;
    std::set<few_basis *> bases;
    PinnedPool pinned;
    int tile_R[2] = {1, 8};
    int tile_T[2] = {256, 256};
    int tile_S[2] = {256, 1024};  // slots per ring stage (the mode tile)
    std::map<std::tuple<int, int, int, int>, int> occ_cache;
    bool timing = false;
    cudaEvent_t tev[8] = {};
    bool trec[4] = {false, false, false, false};
};

namespace {

// A named NVTX range over an entry point's host work (inert unless a profiler is attached), so a
// timeline shows which call queued which kernels.
struct NvtxRange {
    explicit NvtxRange(const char *name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange &) = delete;
    NvtxRange &operator=(const NvtxRange &) = delete;
};

few_status try_alloc(few_ctx *c, size_t bytes, cudaStream_t st, void **out)
{
    *out = nullptr;
    if (bytes == 0) bytes = 256;
    bytes = align_up(bytes, 256);
    if (c->budget && c->in_use + bytes > c->budget) return FEW_ERR_BUDGET;
    cudaError_t e = cudaMallocFromPoolAsync(out, bytes, c->pool, st);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        *out = nullptr;
        return e == cudaErrorMemoryAllocation ? FEW_ERR_NOMEM : FEW_ERR_CUDA;
    }
    c->in_use += bytes;
    c->sizes[*out] = bytes;
    return FEW_OK;
}

void dev_free(few_ctx *c, void *p, cudaStream_t st);

// Frees the digit slices of the context's bases (the FP64 amplitudes then take the plain chain), once all
// work that may read them has ended.  False if there are none to free, or while `st` is being captured.
bool give_up_slices(few_ctx *c, cudaStream_t st)
{
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    const bool known = cudaStreamIsCapturing(st, &capture) == cudaSuccess;
    bool any = false;
    for (const few_basis *b : c->bases) any |= b->slices && !b->captured;
    if (!known || capture != cudaStreamCaptureStatusNone || !any || cudaDeviceSynchronize() != cudaSuccess) {
        (void)cudaGetLastError();
        return false;
    }
    for (few_basis *b : c->bases) {
        if (!b->slices || b->captured) continue;
        dev_free(c, b->slices, c->internal);
        b->slices = nullptr;
        b->bexp64 = nullptr;
        b->bpack64 = nullptr;
    }
    cudaStreamSynchronize(c->internal);
    return true;
}

few_status dev_alloc(few_ctx *c, size_t bytes, cudaStream_t st, void **out)
{
    few_status e = try_alloc(c, bytes, st, out);
    if ((e == FEW_ERR_BUDGET || e == FEW_ERR_NOMEM) && give_up_slices(c, st)) e = try_alloc(c, bytes, st, out);
    return e;
}

void dev_free(few_ctx *c, void *p, cudaStream_t st)
{
    if (!p) return;
    auto it = c->sizes.find(p);
    if (it != c->sizes.end()) {
        c->in_use -= it->second;
        c->sizes.erase(it);
    }
    cudaFreeAsync(p, st);
}

// Event pair `slot` (0 build, 1 harmonics, 2 fold, 3 summation) around a kernel launch.
void tmark(few_ctx *c, int slot, bool end, cudaStream_t st)
{
    if (!c->timing) return;
    cudaEventRecord(c->tev[2 * slot + (end ? 1 : 0)], st);
    if (end) c->trec[slot] = true;
}

// Copy a host image to the device through a pinned staging block, ordered on `st`.
few_status upload(few_ctx *c, void *dst, const void *src, size_t bytes, cudaStream_t st)
{
    if (bytes == 0) return FEW_OK;
    PinnedPool::Block *b = c->pinned.acquire(bytes);
    if (!b) return FEW_ERR_NOMEM;
    std::memcpy(b->p, src, bytes);
    FEW_CUDA_TRY(cudaMemcpyAsync(dst, b->p, bytes, cudaMemcpyHostToDevice, st));
    FEW_CUDA_TRY(cudaEventRecord(b->ev, st));
    b->pending = true;
    return FEW_OK;
}

bool is_fin(double x) { return std::isfinite(x); }

few_status check_knots(const double *t, int K)
{
    if (!t || K < 4) return FEW_ERR_KNOTS;
    for (int k = 0; k < K; ++k)
        if (!is_fin(t[k])) return FEW_ERR_KNOTS;
    for (int k = 0; k + 1 < K; ++k)
        if (!(t[k + 1] > t[k])) return FEW_ERR_KNOTS;
    return FEW_OK;
}

// Harmonic slot plan of a mode list (host planning of the fold and the Horner order).
// Rows are the signed m from the largest down to m_last (-max m when any mode has m > 0, else
// 0), every m in between included; row j holds the slots n = hi_j, hi_j - 1, ..., lo_j (the
// extreme n of the signed modes with that m; zero-filled in between; an empty row has no slot
// and keeps the previous row's lo).  rows[j] = (slots of row j, lo_{j-1} - lo_j).
struct SlotPlan {
    int n_slots = 0, m_last = 0, lo_last = 0;
    std::vector<int2> pair_lm;
    std::vector<int> mode_pair;
    std::vector<int> slot_ptr;
    std::vector<int2> contrib;
    std::vector<int2> rows;
    std::vector<int4> row_slot;  // (first slot, highest n, lowest n, 0) of each row
    // tensor-core summation: pairs of rows m and -m, K steps, centre of the n range, largest m;
    // pairs 0 where the mode set exceeds its accumulators or basis
    int tc_pairs = 0, tc_ks = 0, n_mid = 0, m_top = 0;
};

// Rows of a mode list, dense by signed m (from the largest m down), and the check of the list.
// The list is looked at in a few flat passes (no trees or hash sets): it is planned on the path of
// every new trajectory and checked on that of every direct sum.
struct RowRange {
    int m_top = 0, m_last = 0, n_rows = 0;
    int l_top = 0, n_min = 0, n_max = 0;  // of the listed modes
    std::vector<int> lo, hi, first;  // [n_rows] n range (lo > hi: empty), first slot
    int slots = 0;
    int slot(int ms, int ns) const { return first[m_top - ms] + hi[m_top - ms] - ns; }
};

few_status check_modes(const int *l, const int *m, const int *n, int N, RowRange &R)
{
    if (!l || !m || !n || N < 1) return FEW_ERR_MODES;
    int m_top = 0;
    for (int i = 0; i < N; ++i) {
        if (l[i] < 2 || l[i] > kMaxL || m[i] < 0 || m[i] > l[i] || n[i] < -kMaxAbsN ||
            n[i] > kMaxAbsN)
            return FEW_ERR_MODES;
        m_top = std::max(m_top, m[i]);
        R.l_top = std::max(R.l_top, l[i]);
        R.n_min = std::min(i ? R.n_min : n[0], n[i]);
        R.n_max = std::max(i ? R.n_max : n[0], n[i]);
    }
    R.m_top = m_top;
    R.m_last = -m_top;  // 0 when every mode has m = 0
    R.n_rows = 2 * m_top + 1;
    R.lo.assign(R.n_rows, kMaxAbsN + 1);
    R.hi.assign(R.n_rows, -kMaxAbsN - 1);
    for (int i = 0; i < N; ++i) {  // the modes and, for m > 0, their (-m, -n) partners
        int j = m_top - m[i];
        R.lo[j] = std::min(R.lo[j], n[i]);
        R.hi[j] = std::max(R.hi[j], n[i]);
        if (m[i] > 0) {
            j = m_top + m[i];
            R.lo[j] = std::min(R.lo[j], -n[i]);
            R.hi[j] = std::max(R.hi[j], -n[i]);
        }
    }
    R.first.assign(R.n_rows, 0);
    for (int j = 0; j < R.n_rows; ++j) {
        R.first[j] = R.slots;
        if (R.hi[j] >= R.lo[j]) R.slots += R.hi[j] - R.lo[j] + 1;
    }
    std::vector<uint64_t> seen(R.slots, 0);  // bit l of each (m, n)
    for (int i = 0; i < N; ++i) {
        uint64_t &s = seen[R.slot(m[i], n[i])];
        if (s >> l[i] & 1) return FEW_ERR_MODES;  // duplicate (l, m, n)
        s |= (uint64_t)1 << l[i];
    }
    return FEW_OK;
}

few_status plan_slots(const int *l, const int *m, const int *n, int N, SlotPlan &P)
{
    RowRange R;
    const few_status st = check_modes(l, m, n, N, R);
    if (st) return st;
    // (l, m) pairs, numbered as they appear
    std::vector<int> pair_id((kMaxL + 1) * (kMaxL + 1), -1);
    P.mode_pair.resize(N);
    for (int i = 0; i < N; ++i) {
        int &id = pair_id[l[i] * (kMaxL + 1) + m[i]];
        if (id < 0) {
            id = (int)P.pair_lm.size();
            P.pair_lm.push_back(make_int2(l[i], m[i]));
        }
        P.mode_pair[i] = id;
    }
    // rows m = m_top..m_last, slots n = hi..lo in each
    int prev_lo = 0;
    for (int j = 0; j < R.n_rows; ++j) {
        const bool any = R.hi[j] >= R.lo[j];
        const int L = any ? R.hi[j] - R.lo[j] + 1 : 0, cur_lo = any ? R.lo[j] : prev_lo;
        P.rows.push_back(make_int2(L, j == 0 ? 0 : prev_lo - cur_lo));
        P.row_slot.push_back(make_int4(R.first[j], L ? R.hi[j] : -1, L ? R.lo[j] : 0, 0));
        prev_lo = cur_lo;
    }
    const int n_lo = *std::min_element(R.lo.begin(), R.lo.end());
    const int n_hi = *std::max_element(R.hi.begin(), R.hi.end());
    // (the fold mirrors row m into row -m about n = 0: any other centre is for m = 0 alone)
    P.n_mid = R.m_top > 0 ? 0 : n_lo + (n_hi - n_lo) / 2;
    const int half = std::max(n_hi - P.n_mid, P.n_mid - n_lo);
    P.m_top = R.m_top;
    if (R.m_top < kTcMaxPairs && half <= kTcMaxHalf) {
        P.tc_pairs = R.m_top + 1;
        P.tc_ks = half / 8 + 1;
    }
    P.n_slots = R.slots;
    P.m_last = R.m_last;
    P.lo_last = prev_lo;
    // contributions CSR, each slot's in list order
    P.slot_ptr.assign(R.slots + 1, 0);
    for (int i = 0; i < N; ++i) {
        ++P.slot_ptr[R.slot(m[i], n[i]) + 1];
        if (m[i] > 0) ++P.slot_ptr[R.slot(-m[i], -n[i]) + 1];
    }
    for (int s = 0; s < R.slots; ++s) P.slot_ptr[s + 1] += P.slot_ptr[s];
    P.contrib.resize(P.slot_ptr[R.slots]);
    std::vector<int> at(P.slot_ptr.begin(), P.slot_ptr.end() - 1);
    for (int i = 0; i < N; ++i) {
        P.contrib[at[R.slot(m[i], n[i])]++] = make_int2(2 * i, 2 * P.mode_pair[i]);
        if (m[i] > 0) P.contrib[at[R.slot(-m[i], -n[i])]++] = make_int2(2 * i + 1, 2 * P.mode_pair[i] + 1);
    }
    return FEW_OK;
}

few_status segments(const double *t, int K, double t0, double dt, int64_t ns, int64_t *seg)
{
    few_status st = check_knots(t, K);
    if (st) return st;
    if (!is_fin(t0) || !is_fin(dt) || !(dt > 0.0) || ns < 0 || ns > 2147483647LL) return FEW_ERR_RANGE;
    if (ns > 0) {
        const double last = std::fma((double)(ns - 1), dt, t0);
        if (t0 < t[0] || last > t[K - 1]) return FEW_ERR_RANGE;
    }
    seg[0] = 0;
    for (int k = 1; k < K - 1; ++k) {
        double x = std::ceil((t[k] - t0) / dt);
        int64_t v = x <= 0.0 ? 0 : (x >= (double)ns ? ns : (int64_t)x);
        seg[k] = std::max(v, seg[k - 1]);
    }
    seg[K - 1] = ns;
    return FEW_OK;
}

}  // namespace

struct few_traj {
    few_ctx *ctx = nullptr;
    int K = 0, N = 0, J = 0, S = 0;
    std::vector<double> t_host;
    SlotPlan plan;
    void *dmem = nullptr;
    double *ybuf = nullptr;  // device staging for host-provided knot data (lazy)
    TrajDev dev{};
    bool has_data = false;
    // device pointers of the current knot data (for batched rebuilds)
    const double *src_phi_phi = nullptr, *src_phi_r = nullptr, *src_re = nullptr, *src_im = nullptr;
};

// Launch shape of one plan.
struct LaunchPlan {
    int variant = kVariantFp64;
    int grid = 0, threads = 0, R = 0, smem = 0, total_pairs = 0, total_fold = 0;
    int total_anchor_segs = 0;
    int total_segs = 0, total_tiles = 0, ks = 0;  // tensor-core variants
};

struct few_batch {
    // The waves of one summation variant: a batch may need both the tensor-core and the scalar
    // one of its precision, which then run one after the other.
    struct Part {
        void *blob_dev = nullptr;
        void *scratch_dev = nullptr;
        LaunchPlan launch;
    };
    few_ctx *ctx = nullptr;
    int n = 0;
    std::vector<Part> parts;
    void *jobs_dev = nullptr;
    int n_jobs = 0, build_blocks = 0, max_knots = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
};

namespace {

// Host image of a plan (the blob) plus its scratch requirements.
struct PlanImage {
    std::vector<unsigned char> blob;
    size_t off_waves = 0, off_cta = 0, off_seg = 0, off_anc = 0;
    size_t scratch_bytes = 0;
    std::vector<size_t> fcoef_off, ylm_off, anchor_off;
    size_t recs_off = 0;  // tensor-core variants: tile records of all waves
    std::vector<std::vector<int64_t>> seg;  // per wave: segment sample ranges [K]
    bool fp64 = false;
    LaunchPlan launch;
    int buf_bytes = 0, stage_slots = 0, ring = 0;
};

int occupancy(few_ctx *c, int variant, int R, int T, int smem)
{
    auto key = std::make_tuple(variant, R, T, smem);
    auto it = c->occ_cache.find(key);
    if (it != c->occ_cache.end()) return it->second;
    const int o = sum_occupancy(variant, R, T, smem);
    c->occ_cache[key] = o;
    return o;
}

few_status validate_request(const few_request &r, bool need_device_out)
{
    if (!r.traj || !r.out) return FEW_ERR_INVALID_ARG;
    if (!r.traj->has_data) return FEW_ERR_STATE;
    if (r.prec != FEW_FP64 && r.prec != FEW_MIXED) return FEW_ERR_INVALID_ARG;
    if (r.out_where != FEW_MEM_HOST && r.out_where != FEW_MEM_DEVICE) return FEW_ERR_INVALID_ARG;
    if (need_device_out && r.out_where != FEW_MEM_DEVICE) return FEW_ERR_INVALID_ARG;
    if (!is_fin(r.theta) || !is_fin(r.phi) || !is_fin(r.scale) || !is_fin(r.dphi_phi0) ||
        !is_fin(r.dphi_r0))
        return FEW_ERR_INVALID_ARG;
    if (r.frame != FEW_FRAME_SOURCE && r.frame != FEW_FRAME_SSB) return FEW_ERR_INVALID_ARG;
    if (r.frame == FEW_FRAME_SSB) {
        if (!is_fin(r.theta_K) || !is_fin(r.phi_K)) return FEW_ERR_INVALID_ARG;
        // the source frame needs R x S != 0
        const double R[3] = {std::sin(r.theta) * std::cos(r.phi), std::sin(r.theta) * std::sin(r.phi),
                             std::cos(r.theta)};
        const double S[3] = {std::sin(r.theta_K) * std::cos(r.phi_K),
                             std::sin(r.theta_K) * std::sin(r.phi_K), std::cos(r.theta_K)};
        const double x = R[1] * S[2] - R[2] * S[1], y = R[2] * S[0] - R[0] * S[2],
                     z = R[0] * S[1] - R[1] * S[0];
        if (!(x * x + y * y + z * z > 1e-24)) return FEW_ERR_INVALID_ARG;
    }
    if (!is_fin(r.t0) || !is_fin(r.dt) || !(r.dt > 0.0) || r.n_samples < 0 ||
        r.n_samples > 2147483647LL)
        return FEW_ERR_RANGE;
    const few_traj *tr = r.traj;
    if (r.n_samples > 0) {
        const double last = std::fma((double)(r.n_samples - 1), r.dt, r.t0);
        if (r.t0 < tr->t_host[0] || last > tr->t_host[tr->K - 1]) return FEW_ERR_RANGE;
    }
    return FEW_OK;
}

// Whether a mode set fits the tensor-core summation (kTcMaxPairs, kTcMaxHalf) and it is the faster one.
// seg: the request's segment ranges [K].
bool takes_tc(bool fp64, const SlotPlan &P, const std::vector<int64_t> &seg)
{
    if (P.tc_pairs == 0) return false;
    const int K = (int)seg.size();
    const TcShape s{P.tc_pairs, P.tc_ks, P.n_slots, (int)P.rows.size(), (int)P.mode_pair.size(), K};
    TcWork w;
    if (s.slots <= kTcAlwaysSlots)
        for (int k = 0; k + 1 < K; ++k) w.add(seg[k], seg[k + 1]);
    return tc_pays(fp64, s, w);
}
std::vector<int64_t> request_segments(const few_request &r)
{
    std::vector<int64_t> seg(r.traj->K);
    segments(r.traj->t_host.data(), r.traj->K, r.t0, r.dt, r.n_samples, seg.data());
    return seg;
}

// Build the host image of a plan for `n` requests of one precision; tc: by the tensor-core
// summation (every request's mode set fits it); segs: their segment ranges.
few_status build_image(few_ctx *c, const few_request *reqs, int n, bool tc, const std::vector<int64_t> *segs,
                       PlanImage &P)
{
    P.fp64 = reqs[0].prec == FEW_FP64;
    LaunchPlan &L = P.launch;
    const int pi = P.fp64 ? 0 : 1;
    L.R = c->tile_R[pi];
    L.threads = c->tile_T[pi];
    int max_slots = 1;
    for (int q = 0; q < n; ++q) max_slots = std::max(max_slots, reqs[q].traj->plan.n_slots);
    L.variant = P.fp64 ? kVariantFp64 : kVariantScalar;
    const size_t slot_bytes = (size_t)sum_slot_bytes(L.variant);
    P.stage_slots = std::min(c->tile_S[pi], max_slots);  // no stage larger than any table
    P.ring = kDefaultRing;
    P.buf_bytes = (int)align_up((size_t)P.stage_slots * slot_bytes, 128);
    L.smem = P.ring * P.buf_bytes;
    // the tile settings are checked for every variant, also one that does not use them
    const int occ = occupancy(c, L.variant, L.R, L.threads, L.smem);
    if (occ <= 0) return FEW_ERR_LIMIT;
    L.grid = c->sm_count * occ;
    P.seg.assign(segs, segs + n);
    if (tc) {
        L.variant = P.fp64 ? kVariantTc64 : kVariantTc;
        int64_t tiles = 0;
        for (int q = 0; q < n; ++q)
            for (int k = 0; k + 1 < reqs[q].traj->K; ++k)
                tiles += tiles_in_segment((int)P.seg[q][k], (int)P.seg[q][k + 1]);
        if (tiles > 0x7fffffff) return FEW_ERR_LIMIT;
        L.total_tiles = (int)tiles;
        for (int q = 0; q < n; ++q) L.ks = std::max(L.ks, reqs[q].traj->plan.tc_ks);
        L.grid = (int)std::min<int64_t>(c->sm_count, tiles);
    }

    // layout of the blob
    size_t off = align_up(sizeof(PlanHdr), 64);
    P.off_waves = off;
    off = align_up(off + sizeof(WaveDev) * n, 64);
    P.off_cta = off;  // tensor-core variants: int first tiles instead
    off = align_up(off + sizeof(CtaStart) * (L.grid + 1), 64);
    P.off_seg = off;
    size_t seg_ints = 0;
    for (int q = 0; q < n; ++q) seg_ints += reqs[q].traj->K;
    off = align_up(off + sizeof(int) * seg_ints, 64);
    P.off_anc = off;  // per wave: first anchor (or tile) of each segment, then the wave's total
    if (!P.fp64 || tc) off += sizeof(int) * seg_ints;
    off = align_up(off, 256);
    P.blob.assign(off, 0);

    // scratch: folded coefficients (or operand tables, then their scales) and harmonic tables
    // per wave
    size_t s_off = 0;
    P.fcoef_off.resize(n);
    P.ylm_off.resize(n);
    P.anchor_off.resize(n);
    for (int q = 0; q < n; ++q) {
        const few_traj *tr = reqs[q].traj;
        P.fcoef_off[q] = s_off;
        if (tc)
            s_off = align_up(s_off + tr->S * tc_segment_bytes(P.fp64, tr->plan.tc_pairs, tr->plan.tc_ks), 256);
        else
            s_off = align_up(s_off + (size_t)tr->S * tr->plan.n_slots * slot_bytes, 256);
        P.ylm_off[q] = s_off;
        s_off = align_up(s_off + (size_t)tr->plan.pair_lm.size() * 2 * sizeof(double2), 256);
        P.anchor_off[q] = s_off;
        if (L.variant == kVariantScalar) {
            int na = 0;
            for (int k = 0; k + 1 < tr->K; ++k)
                na += anchors_in_segment((int)P.seg[q][k], (int)P.seg[q][k + 1]);
            s_off = align_up(s_off + sizeof(Anchor) * (size_t)na, 256);
        }
    }
    P.recs_off = s_off;
    if (tc) s_off += sizeof(TileRec) * (size_t)L.total_tiles;
    P.scratch_bytes = s_off;
    return FEW_OK;
}

// First tile of each CTA of a tensor-core plan: contiguous runs of tiles of equal total cost.
void partition_tiles(const std::vector<int> &tile_begin, const std::vector<double> &tile_cost,
                     int grid, int *cta)
{
    const int n = (int)tile_cost.size();
    std::vector<double> cum(n + 1, 0.0);
    for (int q = 0; q < n; ++q)
        cum[q + 1] = cum[q] + tile_cost[q] * (tile_begin[q + 1] - tile_begin[q]);
    int q = 0;
    for (int g = 0; g < grid; ++g) {
        const double x = cum[n] * g / grid;
        while (q < n - 1 && cum[q + 1] <= x) ++q;
        const int k = (int)std::ceil((x - cum[q]) / tile_cost[q]);
        cta[g] = std::min(tile_begin[q] + k, tile_begin[q + 1]);
    }
    cta[grid] = tile_begin[n];
}

// CTA slices of the concatenated (wave, sample) space of n waves (segs[q]: wave q's K[q]
// segment starts, the last its sample count), cut at pass boundaries.  A pass is `pass`
// consecutive samples of one segment, and it costs a full pass (one Horner step per slot plus the
// fixed phase work, for every thread) even when its segment ends early; so every slice gets an
// equal share of the total pass cost, to within one pass, rather than an equal share of the
// samples (which left some slices several short passes more than others).  cta[grid] = (n, 0).
void partition_ctas(int n, const int64_t *const *segs, const int *K, const int *slots, int grid,
                    long long pass, CtaStart *cta)
{
    std::vector<long double> cost(n), cum(n + 1, 0.0L);
    std::vector<long long> npass(n, 0);
    auto seg_passes = [&](int q, int k) { return (segs[q][k + 1] - segs[q][k] + pass - 1) / pass; };
    for (int q = 0; q < n; ++q) {
        for (int k = 0; k + 1 < K[q]; ++k) npass[q] += seg_passes(q, k);
        cost[q] = (long double)(slots[q] + 16);
        cum[q + 1] = cum[q] + (long double)npass[q] * cost[q];
    }
    const long double total = cum[n];
    int q = 0, sk = 0;
    long long before = 0;  // passes of wave q before its segment sk
    cta[grid] = CtaStart{n, 0};
    for (int g = 0; g < grid; ++g) {
        if (total <= 0.0L) {
            cta[g] = CtaStart{n, 0};
            continue;
        }
        const long double x = total * g / grid;
        while (q < n - 1 && cum[q + 1] <= x) {
            ++q;
            sk = 0;
            before = 0;
        }
        // first pass of wave q whose cost starts at or after x, then the segment holding it
        long long k = (long long)std::ceil((x - cum[q]) / cost[q]);
        k = std::max(0LL, std::min(k, npass[q]));
        const int S = K[q] - 1;
        while (sk < S && before + seg_passes(q, sk) <= k) {
            before += seg_passes(q, sk);
            ++sk;
        }
        const long long ns = segs[q][S];
        const long long sample = sk < S ? segs[q][sk] + (k - before) * pass : ns;
        cta[g] = CtaStart{q, (int)std::min<long long>(sample, ns)};
    }
}

// Fill the blob now that the device addresses of blob and scratch are known.
void fill_image(few_ctx *c, const few_request *reqs, int n, PlanImage &P, unsigned char *blob_dev,
                unsigned char *scratch_dev, void *const *outs)
{
    PlanHdr *hdr = reinterpret_cast<PlanHdr *>(P.blob.data());
    WaveDev *wv = reinterpret_cast<WaveDev *>(P.blob.data() + P.off_waves);
    CtaStart *cta = reinterpret_cast<CtaStart *>(P.blob.data() + P.off_cta);
    int *seg = reinterpret_cast<int *>(P.blob.data() + P.off_seg);
    int *anc = reinterpret_cast<int *>(P.blob.data() + P.off_anc);
    LaunchPlan &L = P.launch;
    const bool tc = is_tc(L.variant);
    size_t seg_pos = 0;
    int pair_begin = 0, fold_begin = 0, anchor_seg_begin = 0, seg_begin = 0;
    std::vector<int> tile_begin(1, 0);
    std::vector<double> tile_cost;
    for (int q = 0; q < n; ++q) {
        const few_request &r = reqs[q];
        const few_traj *tr = r.traj;
        WaveDev &W = wv[q];
        std::memset(&W, 0, sizeof(W));
        W.tr = tr->dev;
        set_wave_angles(r, W);
        W.scale = r.scale;
        W.dphi_phi = r.dphi_phi0;
        W.dphi_r = r.dphi_r0;
        W.t0 = r.t0;
        W.dt = r.dt;
        W.n_samples = (int)r.n_samples;
        W.out_c64 = r.out_c64 ? 1 : 0;
        W.out = outs[q];
        W.fcoef = scratch_dev + P.fcoef_off[q];
        W.ylm = reinterpret_cast<double2 *>(scratch_dev + P.ylm_off[q]);
        const std::vector<int64_t> &ss = P.seg[q];
        for (int k = 0; k < tr->K; ++k) seg[seg_pos + k] = (int)ss[k];
        W.seg_start = reinterpret_cast<const int *>(blob_dev + P.off_seg) + seg_pos;
        if (tc) {
            int a = 0;
            for (int k = 0; k + 1 < tr->K; ++k) {
                anc[seg_pos + k] = a;
                a += tiles_in_segment((int)ss[k], (int)ss[k + 1]);
            }
            anc[seg_pos + tr->K - 1] = a;
            W.tab = scratch_dev + P.fcoef_off[q];
            if (P.fp64)
                W.seg64 = reinterpret_cast<TcSeg64 *>(
                    W.tab + (size_t)tr->S * tc64_table_bytes(tr->plan.tc_pairs, tr->plan.tc_ks));
            else
                W.tab_inv = reinterpret_cast<float *>(
                    W.tab + (size_t)tr->S * tc_table_bytes(tr->plan.tc_pairs, tr->plan.tc_ks));
            W.tile_off = reinterpret_cast<const int *>(blob_dev + P.off_anc) + seg_pos;
            W.tile_begin = tile_begin[q];
            W.seg_begin = seg_begin;
            seg_begin += tr->S;
            tile_begin.push_back(tile_begin[q] + a);
            tile_cost.push_back(tc_tile_cost(P.fp64, tr->plan.tc_pairs, L.ks));
        } else if (!P.fp64) {
            int a = 0;
            for (int k = 0; k + 1 < tr->K; ++k) {
                anc[seg_pos + k] = a;
                a += anchors_in_segment((int)ss[k], (int)ss[k + 1]);
            }
            anc[seg_pos + tr->K - 1] = a;
            W.anchors = reinterpret_cast<Anchor *>(scratch_dev + P.anchor_off[q]);
            W.anchor_off = reinterpret_cast<const int *>(blob_dev + P.off_anc) + seg_pos;
            W.anchor_seg_begin = anchor_seg_begin;
            anchor_seg_begin += tr->S;
        }
        seg_pos += tr->K;
        W.pair_begin = pair_begin;
        pair_begin += (int)tr->plan.pair_lm.size();
        W.fold_blocks_per_seg = (tr->plan.n_slots + kFoldThreads - 1) / kFoldThreads;
        W.fold_begin = fold_begin;
        fold_begin += tr->S * W.fold_blocks_per_seg;
    }
    L.total_pairs = pair_begin;
    L.total_fold = fold_begin;
    L.total_anchor_segs = anchor_seg_begin;
    L.total_segs = seg_begin;
    if (tc) {
        partition_tiles(tile_begin, tile_cost, L.grid, reinterpret_cast<int *>(cta));
    } else {
        std::vector<const int64_t *> segs(n);
        std::vector<int> Ks(n), slots(n);
        for (int q = 0; q < n; ++q) {
            segs[q] = P.seg[q].data();
            Ks[q] = reqs[q].traj->K;
            slots[q] = reqs[q].traj->plan.n_slots;
        }
        partition_ctas(n, segs.data(), Ks.data(), slots.data(), L.grid,
                       (long long)L.threads * L.R, cta);
    }
    hdr->n_waves = n;
    hdr->total_pairs = L.total_pairs;
    hdr->total_fold_blocks = L.total_fold;
    hdr->total_anchor_segs = L.total_anchor_segs;
    hdr->total_segs = L.total_segs;
    hdr->total_tiles = L.total_tiles;
    hdr->tile_cta = reinterpret_cast<const int *>(blob_dev + P.off_cta);
    hdr->recs = reinterpret_cast<TileRec *>(scratch_dev + P.recs_off);
    hdr->grid_sum = L.grid;
    hdr->buf_bytes = P.buf_bytes;
    hdr->stage_slots = P.stage_slots;
    hdr->ring = P.ring;
    hdr->variant = L.variant;
    hdr->self = blob_dev;
    hdr->waves = reinterpret_cast<const WaveDev *>(blob_dev + P.off_waves);
    hdr->cta = reinterpret_cast<const CtaStart *>(blob_dev + P.off_cta);
    hdr->err = c->d_err;
}

// Queue a plan's kernels on `st`.  Errors are returned after everything queued has been joined.
// plan: a plan that travels in the first kernel's parameters instead of being at hdr_dev already (not kVariantScalar).
cudaError_t launch_kernels(few_ctx *c, const PlanHdr *hdr_dev, const PlanParam *plan, const LaunchPlan &P,
                           cudaStream_t st, bool mark)
{
    auto tm = [&](int slot, bool end) {
        if (mark) tmark(c, slot, end, st);
    };
    const bool fp64 = P.variant == kVariantFp64 || P.variant == kVariantTc64;
    cudaError_t e;
    if (is_tc(P.variant)) {
        tm(1, false);
        // the first kernel takes the plan: the harmonics, or the mixed fold, which forms its own
        if (fp64 && (e = launch_ylm(hdr_dev, plan, P.total_pairs, fp64, st)) != cudaSuccess) return e;
        tm(1, true);
        tm(2, false);
        e = fp64 ? launch_fold_tc64(hdr_dev, P.total_segs, P.total_tiles, c->sm_count, st)
                 : launch_fold_tc(hdr_dev, plan, P.total_segs, P.total_tiles, c->sm_count, st);
        if (e != cudaSuccess) return e;
        tm(2, true);
        tm(3, false);
        e = fp64 ? launch_sum_tc64(hdr_dev, P.grid, P.ks, st) : launch_sum_tc(hdr_dev, P.grid, P.ks, st);
        if (e != cudaSuccess) return e;
        tm(3, true);
        return cudaSuccess;
    }
    // the phase anchors depend on the splines only: they run on a side lane beside the
    // harmonics and the fold (FP64-pipe work next to latency-bound work), joined before the sum
    const bool fork = P.total_anchor_segs > 0;
    auto &L = c->lanes[c->lane_next++ % 4];
    if (fork) {
        // any failure after this point still leaves the side stream's work ordered before what
        // the caller queues next on `st` (the release of the call's scratch)
        if ((e = cudaEventRecord(L.fork, st)) != cudaSuccess ||
            (e = cudaStreamWaitEvent(L.s, L.fork, 0)) != cudaSuccess)
            return e;
        const cudaError_t ea = launch_anchor(hdr_dev, P.total_anchor_segs, L.s);
        if ((e = cudaEventRecord(L.join, L.s)) != cudaSuccess) {
            cudaStreamSynchronize(L.s);
            return e;
        }
        if (ea != cudaSuccess) {
            cudaStreamWaitEvent(st, L.join, 0);
            return ea;
        }
    }
    auto joined = [&](cudaError_t err) {  // a failed launch: join the side stream, then report
        if (err != cudaSuccess && fork) cudaStreamWaitEvent(st, L.join, 0);
        return err;
    };
    tm(1, false);
    if ((e = joined(launch_ylm(hdr_dev, plan, P.total_pairs, fp64, st))) != cudaSuccess) return e;
    tm(1, true);
    tm(2, false);
    if ((e = joined(launch_fold(hdr_dev, P.total_fold, fp64, st))) != cudaSuccess) return e;
    if (fork && (e = cudaStreamWaitEvent(st, L.join, 0)) != cudaSuccess) return e;
    tm(2, true);
    tm(3, false);
    if ((e = launch_sum(hdr_dev, P.grid, P.threads, P.R, P.smem, P.variant, st)) != cudaSuccess)
        return e;
    tm(3, true);
    return cudaSuccess;
}

const char *kNames[] = {"FEW_OK",           "FEW_ERR_INVALID_ARG", "FEW_ERR_KNOTS",
                        "FEW_ERR_MODES",    "FEW_ERR_RANGE",       "FEW_ERR_NOMEM",
                        "FEW_ERR_BUDGET",   "FEW_ERR_CUDA",        "FEW_ERR_TIMEOUT",
                        "FEW_ERR_LIMIT",    "FEW_ERR_STATE"};

}  // namespace

// ------------------------------------------------------------------------------ C ABI

extern "C" {

const char *few_strerror(few_status s)
{
    const int i = (int)s;
    if (i < 0 || i >= (int)(sizeof(kNames) / sizeof(kNames[0]))) return "FEW_ERR_UNKNOWN";
    return kNames[i];
}

int few_abi_version(void) { return FEW_ABI_VERSION; }

few_status few_ctx_create(few_ctx **out, int device, size_t hbm_budget_bytes)
{
    if (!out) return FEW_ERR_INVALID_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess) {
        (void)cudaGetLastError();
        return FEW_ERR_CUDA;
    }
    if (device < 0 || device >= ndev) return FEW_ERR_INVALID_ARG;
    few_ctx *c = new (std::nothrow) few_ctx();
    if (!c) return FEW_ERR_NOMEM;
    c->device = device;
    c->budget = hbm_budget_bytes;
    auto fail = [&](few_status s) {
        if (c->d_err) cudaFree(c->d_err);
        if (c->internal) cudaStreamDestroy(c->internal);
        for (auto &l : c->lanes) {
            if (l.s) cudaStreamDestroy(l.s);
            if (l.fork) cudaEventDestroy(l.fork);
            if (l.join) cudaEventDestroy(l.join);
        }
        for (auto &e : c->tev)
            if (e) cudaEventDestroy(e);
        if (c->pool) cudaMemPoolDestroy(c->pool);
        (void)cudaGetLastError();
        delete c;
        return s;
    };
    DeviceScope dev_scope(device);
    if (!dev_scope.ok) return fail(FEW_ERR_CUDA);
    if (cudaDeviceGetAttribute(&c->sm_count, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return fail(FEW_ERR_CUDA);
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    if (cudaMemPoolCreate(&c->pool, &props) != cudaSuccess) return fail(FEW_ERR_CUDA);
    uint64_t thresh = UINT64_MAX;
    cudaMemPoolSetAttribute(c->pool, cudaMemPoolAttrReleaseThreshold, &thresh);
    if (cudaStreamCreateWithFlags(&c->internal, cudaStreamNonBlocking) != cudaSuccess)
        return fail(FEW_ERR_CUDA);
    for (auto &l : c->lanes)
        if (cudaStreamCreateWithFlags(&l.s, cudaStreamNonBlocking) != cudaSuccess ||
            cudaEventCreateWithFlags(&l.fork, cudaEventDisableTiming) != cudaSuccess ||
            cudaEventCreateWithFlags(&l.join, cudaEventDisableTiming) != cudaSuccess)
            return fail(FEW_ERR_CUDA);
    if (cudaMalloc(&c->d_err, sizeof(unsigned)) != cudaSuccess) return fail(FEW_ERR_NOMEM);
    if (cudaMemset(c->d_err, 0, sizeof(unsigned)) != cudaSuccess) return fail(FEW_ERR_CUDA);
    if (sum_configure() != cudaSuccess || tc_configure() != cudaSuccess ||
        tc64_configure() != cudaSuccess || direct_configure() != cudaSuccess ||
        rb64_configure() != cudaSuccess)
        return fail(FEW_ERR_CUDA);
    for (auto &e : c->tev)
        if (cudaEventCreate(&e) != cudaSuccess) return fail(FEW_ERR_CUDA);
    *out = c;
    return FEW_OK;
}

few_status few_batch_release(few_ctx *ctx, few_batch *b);
few_status few_traj_release(few_ctx *ctx, few_traj *t);
few_status few_basis_release(few_ctx *ctx, few_basis *b);

few_status few_ctx_destroy(few_ctx *ctx)
{
    if (!ctx) return FEW_OK;
    {
        std::lock_guard<std::recursive_mutex> lk(ctx->mu);
        DeviceScope dev_scope(ctx->device);
        cudaDeviceSynchronize();
        auto bs = ctx->batches;
        for (few_batch *b : bs) few_batch_release(ctx, b);
        auto ts = ctx->trajs;
        for (few_traj *t : ts) few_traj_release(ctx, t);
        auto rbs = ctx->bases;
        for (few_basis *b : rbs) few_basis_release(ctx, b);
        cudaStreamSynchronize(ctx->internal);
        for (auto &e : ctx->tev)
            if (e) cudaEventDestroy(e);
        ctx->pinned.release();
        cudaFree(ctx->d_err);
        cudaStreamDestroy(ctx->internal);
        for (auto &l : ctx->lanes) {
            cudaStreamDestroy(l.s);
            cudaEventDestroy(l.fork);
            cudaEventDestroy(l.join);
        }
        cudaMemPoolDestroy(ctx->pool);
        (void)cudaGetLastError();
    }
    delete ctx;
    return FEW_OK;
}

few_status few_ctx_memory(few_ctx *ctx, size_t *bytes_in_use, size_t *budget_bytes)
{
    if (!ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    if (bytes_in_use) *bytes_in_use = ctx->in_use;
    if (budget_bytes) *budget_bytes = ctx->budget;
    return FEW_OK;
}

few_status few_traj_create(few_ctx *ctx, const double *t_knots, int K, const int *l, const int *m,
                           const int *n, int N, few_traj **out)
{
    NvtxRange nvtx_range("few_traj_create");
    if (!ctx || !out) return FEW_ERR_INVALID_ARG;
    *out = nullptr;
    few_status st = check_knots(t_knots, K);
    if (st) return st;
    if (K > FEW_MAX_KNOTS) return FEW_ERR_LIMIT;
    SlotPlan plan;
    if ((st = plan_slots(l, m, n, N, plan))) return st;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    few_traj *tr = new (std::nothrow) few_traj();
    if (!tr) return FEW_ERR_NOMEM;
    tr->ctx = ctx;
    tr->K = K;
    tr->N = N;
    tr->J = 2 + 2 * N;
    tr->S = K - 1;
    tr->t_host.assign(t_knots, t_knots + K);
    tr->plan = std::move(plan);
    const SlotPlan &P = tr->plan;

    // one device allocation for every trajectory array
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off = align_up(off + bytes, 256);
        return o;
    };
    const size_t o_t = take(sizeof(double) * K), o_h = take(sizeof(double) * K),
                 o_ih = take(sizeof(double) * K), o_ra = take(sizeof(double) * K),
                 o_rb = take(sizeof(double) * K), o_lo = take(sizeof(double) * K),
                 o_up = take(sizeof(double) * K),
                 o_ip = take(sizeof(double) * K), o_v = take(sizeof(double) * K),
                 o_x = take(sizeof(double) * K),
                 o_sinv = take(sizeof(double) * (kBuildParts - 1) * (kBuildParts - 1)),
                 o_parts = take(sizeof(int) * (kBuildParts + 2)),
                 o_coef = take(sizeof(double) * 4 * (size_t)tr->S * tr->J),
                 o_slopes = take(sizeof(double) * (size_t)K * tr->J),
                 o_pair = take(sizeof(int2) * P.pair_lm.size()), o_mp = take(sizeof(int) * N),
                 o_sp = take(sizeof(int) * P.slot_ptr.size()),
                 o_ct = take(sizeof(int2) * std::max<size_t>(1, P.contrib.size())),
                 o_rows = take(sizeof(int2) * P.rows.size()),
                 o_rslot = take(sizeof(int4) * P.row_slot.size());
    if ((st = dev_alloc(ctx, off, ctx->internal, &tr->dmem))) {
        delete tr;
        return st;
    }
    unsigned char *d = static_cast<unsigned char *>(tr->dmem);
    // host image of the small arrays
    std::vector<unsigned char> img(o_coef, 0);
    std::memcpy(img.data() + o_t, t_knots, sizeof(double) * K);
    std::vector<unsigned char> img2(off - o_pair, 0);
    auto put = [&](size_t o, const void *src, size_t bytes) {
        if (bytes) std::memcpy(img2.data() + (o - o_pair), src, bytes);
    };
    put(o_pair, P.pair_lm.data(), sizeof(int2) * P.pair_lm.size());
    put(o_mp, P.mode_pair.data(), sizeof(int) * N);
    put(o_sp, P.slot_ptr.data(), sizeof(int) * P.slot_ptr.size());
    put(o_ct, P.contrib.data(), sizeof(int2) * P.contrib.size());
    put(o_rows, P.rows.data(), sizeof(int2) * P.rows.size());
    put(o_rslot, P.row_slot.data(), sizeof(int4) * P.row_slot.size());

    TrajDev &D = tr->dev;
    D.K = K;
    D.N = N;
    D.J = tr->J;
    D.S = tr->S;
    D.n_pairs = (int)P.pair_lm.size();
    D.n_slots = P.n_slots;
    D.n_rows = (int)P.rows.size();
    D.m_last = P.m_last;
    D.lo_last = P.lo_last;
    D.t = reinterpret_cast<const double *>(d + o_t);
    D.h = reinterpret_cast<const double *>(d + o_h);
    D.inv_h = reinterpret_cast<const double *>(d + o_ih);
    D.fac_ra = reinterpret_cast<const double *>(d + o_ra);
    D.fac_rb = reinterpret_cast<const double *>(d + o_rb);
    D.fac_lo = reinterpret_cast<const double *>(d + o_lo);
    D.fac_up = reinterpret_cast<const double *>(d + o_up);
    D.fac_ip = reinterpret_cast<const double *>(d + o_ip);
    D.fac_v = reinterpret_cast<const double *>(d + o_v);
    D.fac_x = reinterpret_cast<const double *>(d + o_x);
    D.fac_sinv = reinterpret_cast<const double *>(d + o_sinv);
    D.parts = reinterpret_cast<const int *>(d + o_parts);
    D.coef = reinterpret_cast<double *>(d + o_coef);
    D.slopes = reinterpret_cast<double *>(d + o_slopes);
    D.pair_lm = reinterpret_cast<const int2 *>(d + o_pair);
    D.mode_pair = reinterpret_cast<const int *>(d + o_mp);
    D.slot_ptr = reinterpret_cast<const int *>(d + o_sp);
    D.contrib = reinterpret_cast<const int2 *>(d + o_ct);
    D.rows = reinterpret_cast<const int2 *>(d + o_rows);
    D.row_slot = reinterpret_cast<const int4 *>(d + o_rslot);
    D.tc_pairs = P.tc_pairs;
    D.tc_ks = P.tc_ks;
    D.n_mid = P.n_mid;
    D.m_top = P.m_top;

    cudaStream_t s = ctx->internal;
    few_status us = upload(ctx, d, img.data(), o_h, s);  // knot times
    if (!us) us = upload(ctx, d + o_pair, img2.data(), off - o_pair, s);
    cudaError_t e = cudaSuccess;
    if (!us) {
        FactorArrays fa;
        fa.h = reinterpret_cast<double *>(d + o_h);
        fa.inv_h = reinterpret_cast<double *>(d + o_ih);
        fa.ra = reinterpret_cast<double *>(d + o_ra);
        fa.rb = reinterpret_cast<double *>(d + o_rb);
        fa.lo = reinterpret_cast<double *>(d + o_lo);
        fa.up = reinterpret_cast<double *>(d + o_up);
        fa.ip = reinterpret_cast<double *>(d + o_ip);
        fa.v = reinterpret_cast<double *>(d + o_v);
        fa.x = reinterpret_cast<double *>(d + o_x);
        fa.sinv = reinterpret_cast<double *>(d + o_sinv);
        fa.parts = reinterpret_cast<int *>(d + o_parts);
        e = launch_factor(D.t, K, fa, s);
    }
    cudaError_t e2 = cudaStreamSynchronize(s);
    if (us || e != cudaSuccess || e2 != cudaSuccess) {
        (void)cudaGetLastError();
        dev_free(ctx, tr->dmem, s);
        cudaStreamSynchronize(s);
        delete tr;
        return us ? us : FEW_ERR_CUDA;
    }
    ctx->trajs.insert(tr);
    *out = tr;
    return FEW_OK;
}

few_status few_traj_set_data(few_ctx *ctx, few_traj *tr, const double *phi_phi, const double *phi_r,
                             const double *amp_re, const double *amp_im, few_mem where, void *stream)
{
    NvtxRange nvtx_range("few_traj_set_data");
    if (!ctx || !tr || tr->ctx != ctx) return FEW_ERR_INVALID_ARG;
    if (!phi_phi || !phi_r || !amp_re || !amp_im) return FEW_ERR_INVALID_ARG;
    if (where != FEW_MEM_HOST && where != FEW_MEM_DEVICE) return FEW_ERR_INVALID_ARG;
    std::unique_lock<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const size_t K = tr->K, N = tr->N;
    BuildJob job{};
    job.tr = tr->dev;
    cudaEvent_t copied = nullptr;  // host inputs: completion of their copies
    if (where == FEW_MEM_HOST) {
        if (!tr->ybuf) {
            void *p = nullptr;
            few_status s = dev_alloc(ctx, sizeof(double) * (2 * K + 2 * K * N), ctx->internal, &p);
            if (s) return s;
            if (cudaStreamSynchronize(ctx->internal) != cudaSuccess) return FEW_ERR_CUDA;
            tr->ybuf = static_cast<double *>(p);
        }
        double *y = tr->ybuf;
        FEW_CUDA_TRY(cudaMemcpyAsync(y, phi_phi, sizeof(double) * K, cudaMemcpyHostToDevice, st));
        FEW_CUDA_TRY(cudaMemcpyAsync(y + K, phi_r, sizeof(double) * K, cudaMemcpyHostToDevice, st));
        FEW_CUDA_TRY(cudaMemcpyAsync(y + 2 * K, amp_re, sizeof(double) * K * N, cudaMemcpyHostToDevice, st));
        FEW_CUDA_TRY(cudaMemcpyAsync(y + 2 * K + K * N, amp_im, sizeof(double) * K * N,
                                     cudaMemcpyHostToDevice, st));
        // the caller may reuse its host arrays on return: the copies' completion is waited for
        // after the build is queued behind them, so the device does not idle on the host
        FEW_CUDA_TRY(cudaEventCreateWithFlags(&copied, cudaEventDisableTiming));
        if (cudaEventRecord(copied, st) != cudaSuccess) {
            (void)cudaGetLastError();
            cudaEventDestroy(copied);
            return FEW_ERR_CUDA;
        }
        job.phi_phi = y;
        job.phi_r = y + K;
        job.amp_re = y + 2 * K;
        job.amp_im = y + 2 * K + K * N;
    } else {
        job.phi_phi = phi_phi;
        job.phi_r = phi_r;
        job.amp_re = amp_re;
        job.amp_im = amp_im;
    }
    job.block_begin = 0;
    few_status s = FEW_OK;
    const int blocks = (tr->J + kBuildSplines - 1) / kBuildSplines;
    tmark(ctx, 0, false, st);
    if (launch_build_one(job, blocks, ctx->d_err, st) != cudaSuccess) {
        (void)cudaGetLastError();
        s = FEW_ERR_CUDA;
    }
    tmark(ctx, 0, true, st);
    if (copied) {
        lk.unlock();  // the copies' completion concerns this call only
        if (cudaEventSynchronize(copied) != cudaSuccess && !s) {
            (void)cudaGetLastError();
            s = FEW_ERR_CUDA;
        }
        cudaEventDestroy(copied);
    }
    if (s) return s;
    tr->src_phi_phi = job.phi_phi;
    tr->src_phi_r = job.phi_r;
    tr->src_re = job.amp_re;
    tr->src_im = job.amp_im;
    tr->has_data = true;
    return FEW_OK;
}

few_status few_traj_release(few_ctx *ctx, few_traj *tr)
{
    if (!ctx || !tr || tr->ctx != ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    cudaDeviceSynchronize();
    dev_free(ctx, tr->ybuf, ctx->internal);
    dev_free(ctx, tr->dmem, ctx->internal);
    cudaStreamSynchronize(ctx->internal);
    (void)cudaGetLastError();
    ctx->trajs.erase(tr);
    delete tr;
    return FEW_OK;
}

few_status few_traj_info(const few_traj *tr, int *K, int *N, int *n_slots)
{
    if (!tr) return FEW_ERR_INVALID_ARG;
    if (K) *K = tr->K;
    if (N) *N = tr->N;
    if (n_slots) *n_slots = tr->plan.n_slots;
    return FEW_OK;
}

few_status few_waveform(few_ctx *ctx, const few_request *req, void *stream)
{
    NvtxRange nvtx_range("few_waveform");
    if (!ctx || !req) return FEW_ERR_INVALID_ARG;
    few_status st = validate_request(*req, false);
    if (st) return st;
    if (req->traj->ctx != ctx) return FEW_ERR_INVALID_ARG;
    if (req->n_samples == 0) return FEW_OK;
    std::unique_lock<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    PlanImage P;
    const std::vector<int64_t> seg = request_segments(*req);
    const size_t out_bytes = (size_t)req->n_samples * (req->out_c64 ? 8 : 16);
    void *out_dev = req->out;
    bool staged = false;
    if (req->out_where == FEW_MEM_HOST) {
        // page-locked host memory is addressable from the device (over NVLink-C2C on a Grace
        // host): the summation kernel stores into it directly and the transfer overlaps the
        // compute; pageable memory is staged on the device and copied back
        cudaPointerAttributes pa{};
        if (cudaPointerGetAttributes(&pa, req->out) == cudaSuccess && pa.type == cudaMemoryTypeHost &&
            pa.devicePointer != nullptr) {
            out_dev = pa.devicePointer;
        } else {
            (void)cudaGetLastError();
            staged = true;
        }
    }
    void *blob = nullptr, *dout = nullptr;  // the plan, its scratch behind it; the staged output
    auto plan = [&](bool tc) {
        P = PlanImage();
        few_status e = build_image(ctx, req, 1, tc, &seg, P);
        if (!e) e = dev_alloc(ctx, P.blob.size() + P.scratch_bytes, s, &blob);
        if (!e && staged && (e = dev_alloc(ctx, out_bytes, s, &dout))) dev_free(ctx, blob, s);
        return e;
    };
    const bool tc = takes_tc(req->prec == FEW_FP64, req->traj->plan, seg);
    st = plan(tc);
    // the tensor-core plan may need more scratch than the scalar one (sparse mode sets)
    if (tc && (st == FEW_ERR_BUDGET || st == FEW_ERR_NOMEM)) st = plan(false);
    if (st) return st;
    if (staged) out_dev = dout;
    unsigned char *blob_dev = static_cast<unsigned char *>(blob);
    fill_image(ctx, req, 1, P, blob_dev, blob_dev + P.blob.size(), &out_dev);
    // a small plan travels in the first kernel's parameters: no copy stands between the kernels, and the call can be
    // captured (mixed scalar plans are read by two streams' first kernels: they are copied)
    std::unique_ptr<PlanParam> param;
    if (P.launch.variant != kVariantScalar && P.blob.size() <= (size_t)kPlanParamBytes) param.reset(new (std::nothrow) PlanParam);
    if (param) {
        std::memcpy(param->bytes, P.blob.data(), P.blob.size());
        param->dev = blob_dev;
        param->n = (int)P.blob.size();
    } else {
        st = upload(ctx, blob, P.blob.data(), P.blob.size(), s);
    }
    if (!st && launch_kernels(ctx, static_cast<const PlanHdr *>(blob), param.get(), P.launch, s, true) !=
                   cudaSuccess) {
        (void)cudaGetLastError();
        st = FEW_ERR_CUDA;
    }
    if (!st && dout) {
        cudaError_t e = cudaMemcpyAsync(req->out, dout, out_bytes, cudaMemcpyDeviceToHost, s);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            st = FEW_ERR_CUDA;
        }
    }
    dev_free(ctx, dout, s);
    dev_free(ctx, blob, s);
    if (!st && req->out_where == FEW_MEM_HOST) {
        // everything is queued: wait for the result without holding the context, so calls from
        // other host threads (their own streams) overlap this one's transfer and compute
        lk.unlock();
        if (cudaStreamSynchronize(s) != cudaSuccess) {
            (void)cudaGetLastError();
            st = FEW_ERR_CUDA;
        }
    }
    return st;
}

few_status few_phase_samples(few_ctx *ctx, const few_traj *tr, double t0, double dt, int64_t n,
                             double dphi_phi0, double dphi_r0, double *out_dev, void *stream)
{
    NvtxRange nvtx_range("few_phase_samples");
    if (!ctx || !tr || tr->ctx != ctx || !out_dev) return FEW_ERR_INVALID_ARG;
    if (!tr->has_data) return FEW_ERR_STATE;
    if (!is_fin(dphi_phi0) || !is_fin(dphi_r0)) return FEW_ERR_INVALID_ARG;
    std::vector<int64_t> seg(tr->K);
    few_status st = segments(tr->t_host.data(), tr->K, t0, dt, n, seg.data());
    if (st) return st;
    if (n == 0) return FEW_OK;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    std::vector<int> seg32(seg.begin(), seg.end());
    void *d = nullptr;
    if ((st = dev_alloc(ctx, sizeof(int) * seg32.size(), s, &d))) return st;
    st = upload(ctx, d, seg32.data(), sizeof(int) * seg32.size(), s);
    if (!st) {
        cudaError_t e = launch_phases(tr->dev, static_cast<const int *>(d), t0, dt, (int)n,
                                      dphi_phi0, dphi_r0, out_dev, s);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            st = FEW_ERR_CUDA;
        }
    }
    dev_free(ctx, d, s);
    return st;
}

few_status few_mode_select(few_ctx *ctx, const double *amp_re, const double *amp_im, int K, int N,
                           const int *m, double eps, unsigned char *mask, void *stream)
{
    NvtxRange nvtx_range("few_mode_select");
    if (!ctx || !amp_re || !amp_im || !m || !mask) return FEW_ERR_INVALID_ARG;
    if (K < 1 || N < 1 || !is_fin(eps) || eps < 0.0) return FEW_ERR_INVALID_ARG;
    if (N > mode_select_max_modes()) return FEW_ERR_LIMIT;
    ModeDoubling dbl{};
    for (int i = 0; i < N; ++i) {
        if (m[i] < 0) return FEW_ERR_MODES;
        if (m[i] > 0) dbl.w[i >> 5] |= 1u << (i & 31);
    }
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (launch_mode_select(amp_re, amp_im, K, N, dbl, eps, mask, s) != cudaSuccess) {
        (void)cudaGetLastError();
        return FEW_ERR_CUDA;
    }
    return FEW_OK;
}

few_status few_direct_sum(few_ctx *ctx, const double *pphi, const double *pr, const double *are,
                          const double *aim, int64_t ns, const int *l, const int *m, const int *n,
                          int N, double theta, double phi, double scale, int prec, void *out,
                          int out_c64, void *stream)
{
    NvtxRange nvtx_range("few_direct_sum");
    if (!ctx || !pphi || !pr || !are || !aim || !out) return FEW_ERR_INVALID_ARG;
    if (prec != FEW_FP64 && prec != FEW_MIXED) return FEW_ERR_INVALID_ARG;
    if (!is_fin(theta) || !is_fin(phi) || !is_fin(scale) || ns < 0) return FEW_ERR_INVALID_ARG;
    RowRange modes;
    few_status st = check_modes(l, m, n, N, modes);
    if (st) return st;
    if (ns == 0) return FEW_OK;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t mc_bytes = align_up(direct_mode_const_bytes(N), 256);
    const size_t idx_bytes = align_up(sizeof(int) * (size_t)N, 256);
    void *d = nullptr;
    if ((st = dev_alloc(ctx, mc_bytes + 3 * idx_bytes, s, &d))) return st;
    unsigned char *b = static_cast<unsigned char *>(d);
    std::vector<int> lmn(3 * (idx_bytes / sizeof(int)), 0);
    const size_t stride = idx_bytes / sizeof(int);
    std::copy(l, l + N, lmn.begin());
    std::copy(m, m + N, lmn.begin() + stride);
    std::copy(n, n + N, lmn.begin() + 2 * stride);
    st = upload(ctx, b + mc_bytes, lmn.data(), 3 * idx_bytes, s);
    if (!st) {
        const int *dl = reinterpret_cast<const int *>(b + mc_bytes);
        cudaError_t e = launch_direct(pphi, pr, are, aim, (long long)ns, dl, dl + stride,
                                      dl + 2 * stride, N, theta, phi, scale, prec == FEW_FP64, out,
                                      out_c64 ? 1 : 0, b, modes.l_top, modes.m_top, modes.n_min, modes.n_max,
                                      ctx->sm_count, ctx->d_err, s);
        if (e != cudaSuccess) {
            (void)cudaGetLastError();
            st = FEW_ERR_CUDA;
        }
    }
    dev_free(ctx, d, s);
    return st;
}

few_status few_basis_create(few_ctx *ctx, const double *b_re, const double *b_im, int Nb, int N,
                            few_mem where, void *stream, few_basis **out)
{
    NvtxRange nvtx_range("few_basis_create");
    if (!ctx || !b_re || !b_im || !out || Nb < 1 || N < 1) return FEW_ERR_INVALID_ARG;
    if (where != FEW_MEM_HOST && where != FEW_MEM_DEVICE) return FEW_ERR_INVALID_ARG;
    if (Nb > FEW_MAX_BASIS) return FEW_ERR_LIMIT;
    *out = nullptr;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const RbLayout L = rb_layout(Nb, N, 0);
    const size_t b_bytes = align_up(sizeof(double) * (size_t)Nb * N, 256);
    const size_t g64 = align_up(sizeof(double2) * (size_t)Nb * Nb, 256);
    const size_t g32 = align_up(sizeof(float2) * (size_t)Nb * Nb, 256);
    const size_t ex = align_up(sizeof(int) * (size_t)L.modes_padded, 256);
    const size_t ex64 = align_up(sizeof(int) * (size_t)rb64_modes(N), 256);
    const size_t plain = align_up(2 * b_bytes + g64 + g32 + ex + L.bpack_bytes, 256);
    void *d = nullptr, *slices = nullptr;
    few_status st = dev_alloc(ctx, plain, s, &d);
    if (st) return st;
    const bool digits = try_alloc(ctx, ex64 + rb64_basis_bytes(Nb, N), s, &slices) == FEW_OK;
    unsigned char *p = static_cast<unsigned char *>(d);
    double *bre = reinterpret_cast<double *>(p), *bim = reinterpret_cast<double *>(p + b_bytes);
    const size_t bytes = sizeof(double) * (size_t)Nb * N;
    if (where == FEW_MEM_HOST) {
        st = upload(ctx, bre, b_re, bytes, s);
        if (!st) st = upload(ctx, bim, b_im, bytes, s);
    } else if (cudaMemcpyAsync(bre, b_re, bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess ||
               cudaMemcpyAsync(bim, b_im, bytes, cudaMemcpyDeviceToDevice, s) != cudaSuccess) {
        (void)cudaGetLastError();
        st = FEW_ERR_CUDA;
    }
    auto *gt64 = reinterpret_cast<double2 *>(p + 2 * b_bytes);
    auto *gt32 = reinterpret_cast<float2 *>(p + 2 * b_bytes + g64);
    int *bexp = reinterpret_cast<int *>(p + 2 * b_bytes + g64 + g32);
    unsigned char *bpack = p + 2 * b_bytes + g64 + g32 + ex;
    int *bexp64 = static_cast<int *>(slices);
    unsigned char *bpack64 = static_cast<unsigned char *>(slices) + ex64;
    if (!st && (launch_rb_exponents(bre, bim, Nb, N, L.modes_padded, bexp, digits ? bexp64 : nullptr, s) != cudaSuccess ||
                launch_rb_basis(bre, bim, Nb, N, gt64, gt32, bexp, bpack, ctx->sm_count, s) != cudaSuccess ||
                (digits &&
                 launch_rb64_basis(bre, bim, Nb, N, bexp64, bpack64, ctx->sm_count, s) != cudaSuccess))) {
        (void)cudaGetLastError();
        st = FEW_ERR_CUDA;
    }
    if (st) {
        dev_free(ctx, slices, s);
        dev_free(ctx, d, s);
        return st;
    }
    auto *b = new few_basis;
    b->ctx = ctx;
    b->Nb = Nb;
    b->N = N;
    b->dmem = d;
    b->slices = slices;
    b->bre = bre;
    b->bim = bim;
    b->gt64 = gt64;
    b->gt32 = gt32;
    b->bexp = bexp;
    b->bpack = bpack;
    b->bexp64 = digits ? bexp64 : nullptr;
    b->bpack64 = digits ? bpack64 : nullptr;
    ctx->bases.insert(b);
    *out = b;
    return FEW_OK;
}

few_status few_basis_release(few_ctx *ctx, few_basis *b)
{
    if (!ctx || !b || b->ctx != ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    cudaDeviceSynchronize();
    dev_free(ctx, b->slices, ctx->internal);
    dev_free(ctx, b->dmem, ctx->internal);
    cudaStreamSynchronize(ctx->internal);
    (void)cudaGetLastError();
    ctx->bases.erase(b);
    delete b;
    return FEW_OK;
}

few_status few_rb_amplitudes(few_ctx *ctx, const few_basis *b, const double *are,
                             const double *aim, int M, const double *nu, int prec, double *ore,
                             double *oim, void *stream)
{
    NvtxRange nvtx_range("few_rb_amplitudes");
    if (!ctx || !b || b->ctx != ctx || M < 0) return FEW_ERR_INVALID_ARG;
    if (prec != FEW_FP64 && prec != FEW_MIXED) return FEW_ERR_INVALID_ARG;
    if (M == 0) return FEW_OK;
    if (!are || !aim || !ore || !oim) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const bool fp64 = prec == FEW_FP64;
    const RbLayout L = rb_layout(b->Nb, b->N, M);
    const size_t sc_bytes = align_up(2 * sizeof(double) * (size_t)M, 256);  // scale, then q
    bool digits = fp64 && b->bpack64;
    size_t ex_bytes = 0, pack_bytes = 0;
    if (!fp64 || digits) {
        ex_bytes = align_up(sizeof(int) * (size_t)(fp64 ? rb64_rows(M) : L.rows_padded), 256);
        pack_bytes = fp64 ? rb64_coef_bytes(b->Nb, M) : L.apack_bytes;
    }
    void *d = nullptr;
    few_status st = FEW_OK;
    if (digits && try_alloc(ctx, sc_bytes + ex_bytes + pack_bytes, s, &d)) {  // no room: the plain chain
        digits = false;
        ex_bytes = pack_bytes = 0;
    }
    if (!d) st = dev_alloc(ctx, sc_bytes + ex_bytes + pack_bytes, s, &d);
    if (st) return st;
    if (digits && !b->captured) {
        cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
        if (cudaStreamIsCapturing(s, &capture) != cudaSuccess) (void)cudaGetLastError();
        b->captured = capture != cudaStreamCaptureStatusNone;
    }
    unsigned char *p = static_cast<unsigned char *>(d);
    auto &lane = ctx->lanes[ctx->lane_next++ % 4];
    cudaError_t e = launch_rb(are, aim, M, b->Nb, b->N, nu, fp64, b->bre, b->bim, b->gt64, b->gt32,
                              b->bexp, b->bpack, reinterpret_cast<double *>(p),
                              reinterpret_cast<int *>(p + sc_bytes), p + sc_bytes + ex_bytes,
                              digits ? b->bexp64 : nullptr, digits ? b->bpack64 : nullptr, ore,
                              oim, ctx->d_err, ctx->sm_count, s, lane.s, lane.fork, lane.join);
    if (e != cudaSuccess) {
        (void)cudaGetLastError();
        st = FEW_ERR_CUDA;
    }
    dev_free(ctx, d, s);
    return st;
}

few_status few_batch_plan(few_ctx *ctx, const few_request *reqs, int n, unsigned flags, few_batch **out)
{
    NvtxRange nvtx_range("few_batch_plan");
    if (!ctx || !reqs || n < 1 || !out) return FEW_ERR_INVALID_ARG;
    *out = nullptr;
    for (int q = 0; q < n; ++q) {
        few_status st = validate_request(reqs[q], true);
        if (st) return st;
        if (reqs[q].traj->ctx != ctx || reqs[q].prec != reqs[0].prec) return FEW_ERR_INVALID_ARG;
    }
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    few_status st = FEW_OK;
    few_batch *b = new (std::nothrow) few_batch();
    if (!b) return FEW_ERR_NOMEM;
    b->ctx = ctx;
    b->n = n;
    cudaStream_t s = ctx->internal;
    auto drop_parts = [&]() {
        for (auto &p : b->parts) {
            dev_free(ctx, p.scratch_dev, s);
            dev_free(ctx, p.blob_dev, s);
        }
        b->parts.clear();
    };
    auto fail = [&](few_status e) {
        dev_free(ctx, b->jobs_dev, s);
        drop_parts();
        cudaStreamSynchronize(s);
        (void)cudaGetLastError();
        if (b->exec) cudaGraphExecDestroy(b->exec);
        if (b->graph) cudaGraphDestroy(b->graph);
        delete b;
        return e;
    };
    // the build jobs first: what is left decides which summation plan fits
    if (flags & FEW_BATCH_REBUILD_SPLINES) {
        std::vector<BuildJob> jobs;
        std::set<const few_traj *> seen;
        int blocks = 0;
        for (int q = 0; q < n; ++q) {
            const few_traj *tr = reqs[q].traj;
            if (!seen.insert(tr).second) continue;
            BuildJob j{};
            j.tr = tr->dev;
            j.phi_phi = tr->src_phi_phi;
            j.phi_r = tr->src_phi_r;
            j.amp_re = tr->src_re;
            j.amp_im = tr->src_im;
            j.block_begin = blocks;
            blocks += (tr->J + kBuildSplines - 1) / kBuildSplines;
            b->max_knots = std::max(b->max_knots, tr->K);
            jobs.push_back(j);
        }
        if ((st = dev_alloc(ctx, sizeof(BuildJob) * jobs.size(), s, &b->jobs_dev))) return fail(st);
        if ((st = upload(ctx, b->jobs_dev, jobs.data(), sizeof(BuildJob) * jobs.size(), s)))
            return fail(st);
        b->n_jobs = (int)jobs.size();
        b->build_blocks = blocks;
    }
    // one part per summation variant
    auto add_part = [&](const std::vector<few_request> &rq, const std::vector<std::vector<int64_t>> &sg,
                        bool tc) -> few_status {
        if (rq.empty()) return FEW_OK;
        const int nr = (int)rq.size();
        PlanImage P;
        few_status e = build_image(ctx, rq.data(), nr, tc, sg.data(), P);
        if (e) return e;
        b->parts.emplace_back();
        few_batch::Part &part = b->parts.back();
        if ((e = dev_alloc(ctx, P.blob.size(), s, &part.blob_dev))) return e;
        if ((e = dev_alloc(ctx, P.scratch_bytes, s, &part.scratch_dev))) return e;
        std::vector<void *> outs(nr);
        for (int q = 0; q < nr; ++q) outs[q] = rq[q].out;
        fill_image(ctx, rq.data(), nr, P, static_cast<unsigned char *>(part.blob_dev),
                   static_cast<unsigned char *>(part.scratch_dev), outs.data());
        part.launch = P.launch;
        return upload(ctx, part.blob_dev, P.blob.data(), P.blob.size(), s);
    };
    // Waves on the tensor cores where they fit.  A plan past the budget moves the waves that save most by
    // it to the scalar chain (sparse mode sets: their tables are larger than the slots), twice as many
    // each time.
    std::vector<int> order;
    std::vector<char> on_tc(n);
    std::vector<std::vector<int64_t>> seg(n);
    for (int q = 0; q < n; ++q) {
        seg[q] = request_segments(reqs[q]);
        if ((on_tc[q] = takes_tc(reqs[q].prec == FEW_FP64, reqs[q].traj->plan, seg[q]))) order.push_back(q);
    }
    auto saves = [&](int q) {
        const few_traj *tr = reqs[q].traj;
        const bool fp64 = reqs[q].prec == FEW_FP64;
        const int variant = fp64 ? kVariantFp64 : kVariantScalar;
        const double table = (double)tc_segment_bytes(fp64, tr->plan.tc_pairs, tr->plan.tc_ks);
        const double recs = (double)sizeof(TileRec) / kTcTile, anchors = (double)sizeof(Anchor) / kAnchorGroup;
        return tr->S * (table - (double)tr->plan.n_slots * sum_slot_bytes(variant)) +
               (double)reqs[q].n_samples * (recs - (fp64 ? 0.0 : anchors));
    };
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return saves(a) > saves(b); });
    for (size_t moved = 0;;) {
        std::vector<few_request> rq[2];  // by the scalar chain, on the tensor cores
        std::vector<std::vector<int64_t>> sg[2];
        for (int q = 0; q < n; ++q) {
            rq[on_tc[q]].push_back(reqs[q]);
            sg[on_tc[q]].push_back(seg[q]);
        }
        st = add_part(rq[1], sg[1], true);
        if (!st) st = add_part(rq[0], sg[0], false);
        if ((st != FEW_ERR_BUDGET && st != FEW_ERR_NOMEM) || moved == order.size()) break;
        drop_parts();
        const size_t next = std::min(order.size(), 2 * moved + 1);
        for (; moved < next; ++moved) on_tc[order[moved]] = 0;
    }
    if (st) return fail(st);
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(FEW_ERR_CUDA);
    if (!(flags & FEW_BATCH_NO_GRAPH)) {
        cudaStream_t cap = nullptr;
        if (cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking) != cudaSuccess) return fail(FEW_ERR_CUDA);
        cudaError_t e = cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal);
        if (e == cudaSuccess) {
            if (b->n_jobs)
                launch_build(static_cast<const BuildJob *>(b->jobs_dev), b->n_jobs, b->build_blocks,
                             b->max_knots, ctx->d_err, cap);
            // the same forks and joins as a direct run, recorded into the graph
            for (const auto &p : b->parts)
                launch_kernels(ctx, static_cast<const PlanHdr *>(p.blob_dev), nullptr, p.launch, cap, false);
            e = cudaStreamEndCapture(cap, &b->graph);
        }
        if (e == cudaSuccess) e = cudaGraphInstantiate(&b->exec, b->graph, 0);
        cudaStreamDestroy(cap);
        if (e != cudaSuccess) return fail(FEW_ERR_CUDA);
    }
    ctx->batches.insert(b);
    *out = b;
    return FEW_OK;
}

few_status few_batch_run(few_ctx *ctx, few_batch *b, void *stream)
{
    NvtxRange nvtx_range("few_batch_run");
    if (!ctx || !b || b->ctx != ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (b->exec) {
        FEW_CUDA_TRY(cudaGraphLaunch(b->exec, s));
        return FEW_OK;
    }
    if (b->n_jobs) {
        tmark(ctx, 0, false, s);
        FEW_CUDA_TRY(launch_build(static_cast<const BuildJob *>(b->jobs_dev), b->n_jobs,
                                  b->build_blocks, b->max_knots, ctx->d_err, s));
        tmark(ctx, 0, true, s);
    }
    for (const auto &p : b->parts)
        FEW_CUDA_TRY(launch_kernels(ctx, static_cast<const PlanHdr *>(p.blob_dev), nullptr, p.launch, s, true));
    return FEW_OK;
}

few_status few_batch_release(few_ctx *ctx, few_batch *b)
{
    if (!ctx || !b || b->ctx != ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    // The caller guarantees the batch's work has completed (an event, a stream sync); no device
    // synchronisation here, so other work in flight keeps running.
    if (b->exec) cudaGraphExecDestroy(b->exec);
    if (b->graph) cudaGraphDestroy(b->graph);
    dev_free(ctx, b->jobs_dev, ctx->internal);
    for (auto &p : b->parts) {
        dev_free(ctx, p.scratch_dev, ctx->internal);
        dev_free(ctx, p.blob_dev, ctx->internal);
    }
    cudaStreamSynchronize(ctx->internal);
    (void)cudaGetLastError();
    ctx->batches.erase(b);
    delete b;
    return FEW_OK;
}

few_status few_sync_status(few_ctx *ctx)
{
    if (!ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    if (cudaDeviceSynchronize() != cudaSuccess) {
        (void)cudaGetLastError();
        return FEW_ERR_CUDA;
    }
    unsigned bits = 0;
    if (cudaMemcpy(&bits, ctx->d_err, sizeof(bits), cudaMemcpyDeviceToHost) != cudaSuccess)
        return FEW_ERR_CUDA;
    if (bits && cudaMemset(ctx->d_err, 0, sizeof(unsigned)) != cudaSuccess) return FEW_ERR_CUDA;
    if (bits & ERRBIT_TIMEOUT) return FEW_ERR_TIMEOUT;
    if (bits & ERRBIT_NONFINITE) return FEW_ERR_INVALID_ARG;
    if (bits & ERRBIT_INTERNAL) return FEW_ERR_CUDA;
    return FEW_OK;
}

few_status few_selftest_wait_expiry(few_ctx *ctx, unsigned limit_us, void *stream)
{
    if (!ctx || limit_us < 1 || limit_us > 2000000u) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    FEW_CUDA_TRY(launch_wait_selftest(ctx->d_err, limit_us, static_cast<cudaStream_t>(stream)));
    return FEW_OK;
}

few_status few_ctx_set_timing(few_ctx *ctx, int enable)
{
    if (!ctx) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    ctx->timing = enable != 0;
    for (bool &r : ctx->trec) r = false;
    return FEW_OK;
}

few_status few_last_timing(few_ctx *ctx, float *ms)
{
    if (!ctx || !ms) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    DeviceScope dev_scope(ctx->device);
    if (!dev_scope.ok) return FEW_ERR_CUDA;
    for (int i = 0; i < 4; ++i) {
        ms[i] = -1.0f;
        if (!ctx->trec[i]) continue;
        FEW_CUDA_TRY(cudaEventSynchronize(ctx->tev[2 * i + 1]));
        FEW_CUDA_TRY(cudaEventElapsedTime(&ms[i], ctx->tev[2 * i], ctx->tev[2 * i + 1]));
    }
    return FEW_OK;
}

few_status few_set_tiles(few_ctx *ctx, int prec, int R, int threads, int stage_slots)
{
    if (!ctx) return FEW_ERR_INVALID_ARG;
    if (threads != 128 && threads != 256) return FEW_ERR_INVALID_ARG;
    if (prec == FEW_FP64) {
        if (R != 1 && R != 2) return FEW_ERR_INVALID_ARG;
    } else if (prec == FEW_MIXED) {
        if (R != 2 && R != 4 && R != 8) return FEW_ERR_INVALID_ARG;
    } else {
        return FEW_ERR_INVALID_ARG;
    }
    if (stage_slots < kMinStageSlots || stage_slots > kMaxStageSlots || stage_slots % 16)
        return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    ctx->tile_R[prec] = R;
    ctx->tile_T[prec] = threads;
    ctx->tile_S[prec] = stage_slots;
    return FEW_OK;
}

few_status few_get_tiles(few_ctx *ctx, int prec, int *R, int *threads, int *stage_slots)
{
    if (!ctx || (prec != FEW_FP64 && prec != FEW_MIXED)) return FEW_ERR_INVALID_ARG;
    std::lock_guard<std::recursive_mutex> lk(ctx->mu);
    if (R) *R = ctx->tile_R[prec];
    if (threads) *threads = ctx->tile_T[prec];
    if (stage_slots) *stage_slots = ctx->tile_S[prec];
    return FEW_OK;
}

few_status few_plan_segments(const double *t_knots, int K, double t0, double dt, int64_t n_samples,
                             int64_t *seg_start)
{
    if (!seg_start) return FEW_ERR_INVALID_ARG;
    return segments(t_knots, K, t0, dt, n_samples, seg_start);
}

few_status few_plan_chain(const double *t_knots, int K, const int *l, const int *m, const int *n, int N,
                          double t0, double dt, int64_t n_samples, int prec, int *tensor_cores,
                          size_t *scalar_bytes, size_t *tc_bytes)
{
    if (prec != FEW_FP64 && prec != FEW_MIXED) return FEW_ERR_INVALID_ARG;
    SlotPlan P;
    few_status st = plan_slots(l, m, n, N, P);
    if (st) return st;
    std::vector<int64_t> seg(K > 0 ? K : 0);
    if ((st = segments(t_knots, K, t0, dt, n_samples, seg.data()))) return st;
    const bool fp64 = prec == FEW_FP64;
    if (tensor_cores) *tensor_cores = takes_tc(fp64, P, seg) ? 1 : 0;
    // the layout of build_image; the plan itself: headers, the CTAs' starts, two ints a knot
    const size_t S = K - 1, plan = 16384 + 2 * sizeof(int) * (size_t)K;
    const size_t ylm = P.pair_lm.size() * 2 * sizeof(double2);
    size_t anchors = 0, tiles = 0;
    for (int k = 0; k + 1 < K; ++k) {
        anchors += anchors_in_segment((int)seg[k], (int)seg[k + 1]);
        tiles += tiles_in_segment((int)seg[k], (int)seg[k + 1]);
    }
    if (scalar_bytes)
        *scalar_bytes = plan + ylm + S * P.n_slots * sum_slot_bytes(fp64 ? kVariantFp64 : kVariantScalar) +
                        (fp64 ? 0 : anchors * sizeof(Anchor));
    if (tc_bytes)
        *tc_bytes = P.tc_pairs == 0 ? 0
                                    : plan + ylm + S * tc_segment_bytes(fp64, P.tc_pairs, P.tc_ks) +
                                          tiles * sizeof(TileRec);
    return FEW_OK;
}

few_status few_mode_slots(const int *l, const int *m, const int *n, int N, int *n_slots, int *n_rows)
{
    SlotPlan P;
    few_status st = plan_slots(l, m, n, N, P);
    if (st) return st;
    if (n_slots) *n_slots = P.n_slots;
    if (n_rows) *n_rows = (int)P.rows.size();
    return FEW_OK;
}

few_status few_plan_cta_slices(int n_waves, const int64_t *seg_start, const int *K,
                               const int *n_slots, int grid, int pass, int *out_wave,
                               int *out_sample)
{
    if (!seg_start || !K || !n_slots || !out_wave || !out_sample || n_waves < 1 || grid < 1 ||
        pass < 1)
        return FEW_ERR_INVALID_ARG;
    std::vector<const int64_t *> segs(n_waves);
    size_t off = 0;
    for (int q = 0; q < n_waves; ++q) {
        if (K[q] < 2 || n_slots[q] < 1) return FEW_ERR_INVALID_ARG;
        segs[q] = seg_start + off;
        for (int k = 0; k + 1 < K[q]; ++k)
            if (segs[q][k + 1] < segs[q][k] || segs[q][k] < 0) return FEW_ERR_INVALID_ARG;
        if (segs[q][K[q] - 1] > 2147483647LL) return FEW_ERR_INVALID_ARG;
        off += (size_t)K[q];
    }
    std::vector<CtaStart> cta((size_t)grid + 1);
    partition_ctas(n_waves, segs.data(), K, n_slots, grid, pass, cta.data());
    for (int g = 0; g <= grid; ++g) {
        out_wave[g] = cta[g].wave;
        out_sample[g] = cta[g].sample;
    }
    return FEW_OK;
}

}  // extern "C"

// ------------------------------------------------------------------------------ read-only views
// Used by the allocation-free entry point (noalloc.cu), which plans a request itself.

namespace fewsum {

bool ctx_traj_view(few_ctx *ctx, const few_traj *tr, CtxTrajView *v)
{
    if (!ctx || !tr || !v || tr->ctx != ctx) return false;
    v->device = ctx->device;
    v->sm_count = ctx->sm_count;
    v->d_err = ctx->d_err;
    v->tile_R[0] = ctx->tile_R[0];
    v->tile_R[1] = ctx->tile_R[1];
    v->tile_T[0] = ctx->tile_T[0];
    v->tile_T[1] = ctx->tile_T[1];
    v->tile_S[0] = ctx->tile_S[0];
    v->tile_S[1] = ctx->tile_S[1];
    v->has_data = tr->has_data;
    v->K = tr->K;
    v->n_slots = tr->plan.n_slots;
    v->n_pairs = (int)tr->plan.pair_lm.size();
    v->tc_pairs = tr->plan.tc_pairs;
    v->tc_ks = tr->plan.tc_ks;
    v->t_host = tr->t_host.data();
    v->dev = tr->dev;
    return true;
}

std::recursive_mutex &ctx_mutex(few_ctx *ctx) { return ctx->mu; }

few_status check_request(const few_request &r, bool need_device_out)
{
    return validate_request(r, need_device_out);
}

// Frame transformation (Sec. 2.A): from the sky position (tS, pS) and the spin direction
// (tK, pK) in the barycentre frame, the source-frame viewing angles of the propagation direction
// -R in the basis x = R x S/|R x S|, y = (R - (R.S) S)/|R x S|, z = S, and the polarization
// angle psi with tan psi = (cos tS sin tK cos(pS - pK) - sin tS cos tK)/(sin tK sin(pS - pK)).
// The detector-frame waveform is -e^{-2 i psi} times the source-frame one (a pi phase shift for
// the pi/2 basis rotation, then the 2 psi rotation), a constant folded into the harmonics.  All of it
// is per request: formed once here instead of by every harmonic's thread (a dozen FP64 functions).
void set_wave_angles(const few_request &r, WaveDev &W)
{
    W.theta = r.theta;
    W.phi = r.phi;
    W.rotate = 0;
    W.rot_r = 1.0;
    W.rot_i = 0.0;
    if (r.frame != FEW_FRAME_SSB) return;
    const double stS = std::sin(r.theta), ctS = std::cos(r.theta), spS = std::sin(r.phi),
                 cpS = std::cos(r.phi), stK = std::sin(r.theta_K), ctK = std::cos(r.theta_K),
                 spK = std::sin(r.phi_K), cpK = std::cos(r.phi_K);
    const double R[3] = {stS * cpS, stS * spS, ctS};
    const double S[3] = {stK * cpK, stK * spK, ctK};
    const double X[3] = {R[1] * S[2] - R[2] * S[1], R[2] * S[0] - R[0] * S[2],
                         R[0] * S[1] - R[1] * S[0]};
    const double nx = std::sqrt(X[0] * X[0] + X[1] * X[1] + X[2] * X[2]);
    const double rs = R[0] * S[0] + R[1] * S[1] + R[2] * S[2];
    // components of -R: along x (R x S is orthogonal to R), along y, along z = S
    const double vx = 0.0;
    const double vy = -((R[0] - rs * S[0]) * R[0] + (R[1] - rs * S[1]) * R[1] +
                        (R[2] - rs * S[2]) * R[2]) / nx;
    const double vz = -rs;
    W.theta = std::acos(std::max(-1.0, std::min(1.0, vz)));
    W.phi = std::atan2(vy, vx);
    const double psi = std::atan2(ctS * stK * std::cos(r.phi - r.phi_K) - stS * ctK,
                                  stK * std::sin(r.phi - r.phi_K));
    W.rotate = 1;
    W.rot_r = -std::cos(2.0 * psi);  // -e^{-2 i psi}
    W.rot_i = std::sin(2.0 * psi);
}

}  // namespace fewsum
