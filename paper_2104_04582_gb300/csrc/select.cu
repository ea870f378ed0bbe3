// select.cu -- Mode Selector on the device (arXiv:2104.04582 Sec. 3.D).
//
// At every knot of the trajectory, the power of each mode is |A(t_k)|^2, doubled for m > 0 (the
// mode also stands for its m < 0 partner of equal power).  The powers are sorted in descending
// order (ties: lower mode index first) and summed cumulatively; the knot keeps the shortest
// leading run whose cumulative power reaches (1 - eps) of the knot's total.  The selection is the
// union of the kept sets over all knots.
//
// The selection is index output, so it is decided exactly as the plain definition computes it:
// the power is fl(fl(re^2) + fl(im^2)) (no fused multiply-add), and the cumulative sums are the
// left-to-right FP64 sums over the sorted powers, c_j = fl(c_{j-1} + p_j), with the total equal
// to the last of them.  Any other summation order can round differently and move the cut.
//
// One CTA per knot, P = max(128, next power of two >= N) slots, P/4 threads.  The sums need the modes in
// order only down to p_0 2^-54 or so (what is smaller changes no sum and is never kept), and in a range
// of 54 binades a mode's place is nearly known from its leading bits: P/16 buckets a binade, a
// histogram, a prefix sum and the few modes of a bucket compared with one another sort them in five
// barriers.  The cumulative sums are exact integer prefix sums inside each binade of the running sum
// (see select_q).  The first 128 ranks, where the sum leaves a binade every few steps, are summed by
// one warp alone, the rest block-wide.  The kept modes are marked with plain byte stores of 1 into a
// mask zeroed beforehand (every writer stores the same value, so the union needs no atomics).
// What that cannot take (non-finite powers, sums that overflow, subnormal sums, more than 64 modes in
// a bucket, a sum of very many rounding ties) goes to select_general: bitonic sorts by warp, merge
// path, and a sequential chain as the last resort.
// Bound by the latency of one knot, and in it by instruction issue: 100 knots are 100 CTAs of 32 warps,
// one a multiprocessor.  100 knots of 3843 modes: 59 us a call with select_general for all (13 us warp
// sorts, 14 merges, 17 in eight block-wide rounds of sums, 5.5 the powers), 27 us with the buckets
// (powers 4, buckets 6, sums 5 to 9).
#include "fewsum_internal.h"
#include "launch.cuh"

namespace fewsum {

constexpr int kSelectMaxThreads = 1024;
constexpr int kSelectPerThread = 4;  // consecutive sort slots per thread
constexpr int kSelectWarpSlots = 32 * kSelectPerThread;
constexpr int kSelectChain = 32;     // ranks summed one by one before the scans
constexpr int kSelectMaxRounds = 64;  // scan rounds before the sequential chain takes over

// Non-negative doubles order exactly like their IEEE bit patterns read as unsigned integers, so
// the sort compares 64-bit integer keys (descending power = ascending inverted bits), with the
// mode index as the tie-break; integer compares avoid GB300's narrow FP64 pipe.
__device__ __forceinline__ unsigned long long power_key(double p)
{
    return ~static_cast<unsigned long long>(__double_as_longlong(p));
}

__device__ __forceinline__ double key_power(unsigned long long key)
{
    return __longlong_as_double(static_cast<long long>(~key));
}

__device__ __forceinline__ bool sorts_before(unsigned long long ka, int ia, unsigned long long kb,
                                             int ib)
{
    return ka < kb || (ka == kb && ia < ib);
}

// Compare-exchange of two slots held by one thread: a precedes b in the final order when up.
__device__ __forceinline__ void cx_pair(unsigned long long &ka, int &ia, unsigned long long &kb,
                                        int &ib, bool up)
{
    const bool swap = up ? sorts_before(kb, ib, ka, ia) : sorts_before(ka, ia, kb, ib);
    if (swap) {
        const unsigned long long tk = ka; ka = kb; kb = tk;
        const int ti = ia; ia = ib; ib = ti;
    }
}

// One side of a compare-exchange whose partner slot is held by another thread: keep the element
// that comes first (keep_first) or second of the two.  Both sides take the same comparison, so
// exactly one of them ends up with each element.
__device__ __forceinline__ void cx_keep(unsigned long long &k, int &i, unsigned long long ko, int io,
                                        bool keep_first)
{
    if (sorts_before(ko, io, k, i) == keep_first) { k = ko; i = io; }
}

// Power of mode i and its bits (doubled for m > 0).
__device__ __forceinline__ double mode_power(double re, double im, bool twice)
{
    const double p = __dadd_rn(__dmul_rn(re, re), __dmul_rn(im, im));
    return twice ? p * 2.0 : p;
}

__device__ __noinline__ void select_general(const double *__restrict__ amp_re, const double *__restrict__ amp_im,
                                            int N, const ModeDoubling &dbl, double eps, int P,
                                            unsigned char *__restrict__ mask, unsigned long long *sel_key)
{
    int *sel_ix = reinterpret_cast<int *>(sel_key + P);
    __shared__ double s_total;
    __shared__ unsigned long long s_cbits;  // bits of the running sum where a round starts
    __shared__ unsigned long long s_wsum[kSelectMaxThreads / 32];
    __shared__ int s_a, s_exit, s_fallback, s_cut;
    const int k = blockIdx.x, tid = threadIdx.x;
    const int lane = tid & 31, wid = tid >> 5;
    const int p0 = kSelectPerThread * tid;  // first slot of this thread

    unsigned long long key[kSelectPerThread];
    int ix[kSelectPerThread];
#pragma unroll
    for (int r = 0; r < kSelectPerThread; ++r) {
        const int i = p0 + r;
        if (i < N) {
            key[r] = power_key(mode_power(amp_re[(size_t)k * N + i], amp_im[(size_t)k * N + i],
                                          (dbl.w[i >> 5] >> (i & 31)) & 1u));  // m > 0
            ix[r] = i;
        } else {
            key[r] = ~0ull;  // padding: power +0, sorts after every real mode
            ix[r] = 0x7fffffff;
        }
    }
    if (tid == 0) s_cut = 0x7fffffff;

    // 1. each warp sorts its 128 slots (4 per lane) into ascending "sorts_before" order by a
    //    bitonic network in registers and shuffles; below the last stage slot p runs up when
    //    (p & size) == 0, the last stage runs up in every warp
    for (int size = 2; size <= kSelectWarpSlots; size <<= 1) {
        const bool last = size == kSelectWarpSlots;
        int stride = size >> 1;
        for (; stride >= kSelectPerThread; stride >>= 1) {
            const int lane_mask = stride / kSelectPerThread;
            const bool is_lo = (p0 & stride) == 0, up = last || (p0 & size) == 0;
#pragma unroll
            for (int r = 0; r < kSelectPerThread; ++r) {
                const unsigned long long ko = __shfl_xor_sync(0xffffffffu, key[r], lane_mask);
                const int io = __shfl_xor_sync(0xffffffffu, ix[r], lane_mask);
                cx_keep(key[r], ix[r], ko, io, up == is_lo);
            }
        }
        if (stride == 2) {
            const bool up = last || (p0 & size) == 0;  // size >= 4: the same for all four slots
            cx_pair(key[0], ix[0], key[2], ix[2], up);
            cx_pair(key[1], ix[1], key[3], ix[3], up);
            stride = 1;
        }
        // stride 1: slots (0,1) and (2,3); for size 2 the direction alternates inside the thread
        cx_pair(key[0], ix[0], key[1], ix[1], last || ((p0 + 0) & size) == 0);
        cx_pair(key[2], ix[2], key[3], ix[3], last || ((p0 + 2) & size) == 0);
    }
    // 2. the sorted runs merged pairwise in shared memory, log2(P / 128) levels (merge path): a
    //    thread finds by binary search how many of its 4 output ranks come from the first run,
    //    merges them in registers and stores them once the whole level has been read.  Every
    //    (key, index) pair of a real mode is distinct, so the order is the unique sorted one.
    for (int L = kSelectWarpSlots; L < P; L <<= 1) {
        ulonglong2 *kv = reinterpret_cast<ulonglong2 *>(sel_key + p0);
        kv[0] = make_ulonglong2(key[0], key[1]);
        kv[1] = make_ulonglong2(key[2], key[3]);
        *reinterpret_cast<int4 *>(sel_ix + p0) = make_int4(ix[0], ix[1], ix[2], ix[3]);
        __syncthreads();
        const int base = p0 & ~(2 * L - 1), d = p0 - base;  // this thread's first output rank
        const unsigned long long *ak = sel_key + base, *bk = ak + L;
        const int *ai = sel_ix + base, *bi = ai + L;
        int lo = d > L ? d - L : 0, hi = d < L ? d : L;
        while (lo < hi) {  // first i whose A[i] does not precede B[d - 1 - i]
            const int mid = (lo + hi) >> 1;
            if (sorts_before(ak[mid], ai[mid], bk[d - 1 - mid], bi[d - 1 - mid]))
                lo = mid + 1;
            else
                hi = mid;
        }
        int i = lo, j = d - lo;
#pragma unroll
        for (int r = 0; r < kSelectPerThread; ++r) {
            const bool take_a = j >= L || (i < L && sorts_before(ak[i], ai[i], bk[j], bi[j]));
            key[r] = take_a ? ak[i] : bk[j];
            ix[r] = take_a ? ai[i] : bi[j];
            i += take_a ? 1 : 0;
            j += take_a ? 0 : 1;
        }
        __syncthreads();  // every thread has read this level before any stores the next
    }

    // sorted powers to shared memory (slot j = rank j; padding holds +0)
    double *s_pw = reinterpret_cast<double *>(sel_key);
    double *s_cs = s_pw;  // c_j overwrites p_j: a round writes only ranks below where the next starts
    __syncthreads();  // the last shared-memory exchange stage may still be read
#pragma unroll
    for (int r = 0; r < kSelectPerThread; ++r) s_pw[p0 + r] = key_power(key[r]);
    __syncthreads();

    // the cumulative sums c_j = fl(c_{j-1} + p_j), c_{-1} = 0, into s_cs[j] for every j < N.
    // While c stays in one binade [2^E, 2^(E+1)) (ulp U = 2^(E-52), E >= -1022), c/U is an
    // integer below 2^53 and fl(c + p) adds to it the integer nearest p/U (p <= c, so p/U < 2^53
    // and is read off p's bits); those additions are prefix sums, computed block-wide at once.
    // A step whose integer sum reaches 2^53 (the sum leaves the binade) or whose p/U lies exactly
    // halfway between integers (a tie, resolved by the parity of the sum) is taken by the FP64
    // adder itself, and the block starts again from there: a few rounds (binade changes are at
    // most log2 N + 1 apart) give the same bits as the left-to-right chain.
    const unsigned long long kTop = 1ull << 53;
    unsigned long long pm[kSelectPerThread];
    int pe[kSelectPerThread];
    double pv[kSelectPerThread];
    unsigned bad = 0u;
#pragma unroll
    for (int r = 0; r < kSelectPerThread; ++r) {
        pv[r] = key_power(key[r]);
        const unsigned long long bits = static_cast<unsigned long long>(__double_as_longlong(pv[r]));
        const int ef = (int)((bits >> 52) & 0x7ffu);
        pm[r] = (bits & (kTop / 2 - 1)) | (ef ? kTop / 2 : 0ull);
        pe[r] = ef ? ef - 1023 : -1022;
        if (p0 + r < N && ef == 0x7ff) bad = 1u;  // inf or nan: the chain below handles them
    }
    if (tid == 0) {
        s_cbits = static_cast<unsigned long long>(__double_as_longlong(s_pw[0]));
        s_cs[0] = s_pw[0];
        s_a = 1;
        s_fallback = 0;
    }
    __syncthreads();
    if (bad) s_fallback = 1;
    for (int round = 0;; ++round) {
        __syncthreads();
        const int a = s_a;
        if (a >= N || s_fallback) break;
        if (round >= kSelectMaxRounds) {  // many ties: finish with the sequential chain
            if (tid == 0) s_fallback = 1;
            continue;
        }
        const unsigned long long cb = s_cbits;
        const int cef = (int)((cb >> 52) & 0x7ffu);
        const int E = cef ? cef - 1023 : -1022;
        const unsigned long long Mc = (cb & (kTop / 2 - 1)) | (cef ? kTop / 2 : 0ull);
        unsigned long long q[kSelectPerThread], run = 0ull;
        bool tie[kSelectPerThread];
#pragma unroll
        for (int r = 0; r < kSelectPerThread; ++r) {
            const int j = p0 + r;
            q[r] = 0ull;
            tie[r] = false;
            if (j >= a && j < N) {
                const int d = E - pe[r];  // >= 0: p_j <= c
                if (d == 0) {
                    q[r] = pm[r];
                } else if (d < 64) {
                    const unsigned long long rem = pm[r] & ((1ull << d) - 1ull), half = 1ull << (d - 1);
                    q[r] = (pm[r] >> d) + (rem > half ? 1ull : 0ull);
                    tie[r] = rem == half;
                }  // d >= 64: p/U < 1/2, nothing added
            }
            run += q[r];
        }
        // block-wide exclusive prefix of the threads' sums
        unsigned long long incl = run;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned long long v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_wsum[wid] = incl;
        if (tid == 0) s_exit = 0x7fffffff;
        __syncthreads();
        // every warp sums the totals of the warps before it itself (integer sums: exact in any
        // order), so no second barrier is needed
        unsigned long long wp = lane < wid ? s_wsum[lane] : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) wp += __shfl_xor_sync(0xffffffffu, wp, o);
        unsigned long long M[kSelectPerThread];
        unsigned long long m = Mc + wp + (incl - run);
        int jfirst = 0x7fffffff;  // this thread's first step that leaves the binade or ties
#pragma unroll
        for (int r = 0; r < kSelectPerThread; ++r) {
            m += q[r];
            M[r] = m;
            const int j = p0 + r;
            if (j >= a && j < N && (m >= kTop || tie[r]) && j < jfirst) jfirst = j;
        }
        jfirst = __reduce_min_sync(0xffffffffu, jfirst);
        if (lane == 0 && jfirst != 0x7fffffff) atomicMin(&s_exit, jfirst);
        __syncthreads();
        const int jx = s_exit;
        // c_j = M_j U for the steps inside the binade: exponent field E + 1022 plus M's bits
        const unsigned long long ebase = static_cast<unsigned long long>(E + 1022) << 52;
#pragma unroll
        for (int r = 0; r < kSelectPerThread; ++r) {
            const int j = p0 + r;
            if (j >= a && j < N && j < jx) s_cs[j] = __longlong_as_double((long long)(ebase + M[r]));
            if (j == jx) {  // the FP64 adder takes the step that leaves the binade or ties
                const double cprev = j == a ? __longlong_as_double((long long)cb)
                                            : __longlong_as_double((long long)(ebase + M[r] - q[r]));
                const double cnew = __dadd_rn(cprev, pv[r]);
                s_cs[j] = cnew;
                s_cbits = static_cast<unsigned long long>(__double_as_longlong(cnew));
                s_a = j + 1;
            }
        }
        if (jx == 0x7fffffff && tid == 0) s_a = N;
    }
    __syncthreads();
    // the sequential chain from where the rounds stopped (non-finite powers, many ties)
    if (s_fallback && tid == 0) {
        int j = s_a;
        double c = s_cs[j - 1];
        for (; j < N; ++j) {
            c = __dadd_rn(c, s_pw[j]);
            s_cs[j] = c;
        }
    }
    if (tid == 0) s_total = s_cs[N - 1];
    __syncthreads();
    const double total = s_total;
    if (!(total > 0.0)) return;  // uniform: nothing kept at a knot without power
    const double target = (1.0 - eps) * total;
#pragma unroll
    for (int r = 0; r < kSelectPerThread; ++r) {
        const int j = p0 + r;
        if (j >= N) break;
        const double cj = s_cs[j];
        if (cj >= target) {
            atomicMin(&s_cut, j);
            break;
        }
    }
    __syncthreads();
    const int cut = s_cut;  // no rank reaching the target keeps every mode
#pragma unroll
    for (int r = 0; r < kSelectPerThread; ++r)
        if (p0 + r < N && p0 + r <= cut) mask[ix[r]] = 1;
}

// What a step adds to the running sum c, in units of c's last place U: fl(c + p) = c + U q while c stays
// in its binade (exponent E), q the integer nearest p/U, unless p/U lies exactly halfway between two
// (tie: the parity of the sum decides).  pm, pe: significand and exponent of p, pe <= E.
__device__ __forceinline__ unsigned long long select_q(unsigned long long pm, int d, bool &tie)
{
    if (d > 53) return 0ull;  // p < U/2
    const unsigned long long one = 1ull << d, half = one >> 1;
    tie = d > 0 && (pm & (one - 1ull)) == half;
    return (pm + half) >> d;
}

__global__ void __launch_bounds__(kSelectMaxThreads)
k_mode_select(const double *__restrict__ amp_re, const double *__restrict__ amp_im, int N,
              const __grid_constant__ ModeDoubling dbl, double eps, int P, int sub,
              unsigned char *__restrict__ mask)
{
    using u64 = unsigned long long;
    constexpr int R = kSelectPerThread;
    constexpr u64 kTop = 1ull << 53, kFrac = (1ull << 52) - 1ull;
    extern __shared__ __align__(16) u64 sel[];
    u64 *s_key = sel;                                   // [P] bits of the powers in their order
    u64 *s_raw = sel + P;                               // [P] the same by bucket, in any order
    unsigned short *s_ix = reinterpret_cast<unsigned short *>(sel + 2 * P);  // [P] modes of s_key
    unsigned short *s_rix = s_ix + P;                                        // [P] modes of s_raw
    uint4 *s_cnt = reinterpret_cast<uint4 *>(s_key);    // [P/4] 4 P buckets' sizes, a byte each
    int *s_off = reinterpret_cast<int *>(s_key) + P;    // [P/4] first place of each 16 buckets
    __shared__ unsigned s_wmax[kSelectMaxThreads / 32], s_wcnt[kSelectMaxThreads / 32];
    __shared__ u64 s_wsum[kSelectMaxThreads / 32], s_c, s_total;
    __shared__ int s_a, s_exit, s_cut;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5, nw = nt >> 5;
    const int p0 = R * tid;

    // the powers (mode r nt + tid) and the largest one's exponent
    u64 pb[R];
    unsigned top = 0u;
    {
        const double *re = amp_re + (size_t)blockIdx.x * N, *im = amp_im + (size_t)blockIdx.x * N;
        double x[R], y[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = r * nt + tid;
            x[r] = i < N ? re[i] : 0.0;
            y[r] = i < N ? im[i] : 0.0;
        }
        s_cnt[tid] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int i = r * nt + tid;
            // doubled for m > 0 in the exponent (what is not a normal number then goes to select_general)
            const bool twice = i < N && ((dbl.w[i >> 5] >> (i & 31)) & 1u);
            pb[r] = (u64)__double_as_longlong(mode_power(x[r], y[r], false));
            top = max(top, (unsigned)(pb[r] >> 32));
            if (twice) pb[r] += 1ull << 52;
            top = max(top, (unsigned)(pb[r] >> 32));
        }
    }
    top = __reduce_max_sync(0xffffffffu, top);
    if (lane == 0) s_wmax[wid] = top;
    if (tid == 0) s_cut = 0x7fffffff;
    __syncthreads();
    top = __reduce_max_sync(0xffffffffu, lane < nw ? s_wmax[lane] : 0u);
    const int e0 = (int)(top >> 20);
    bool general = e0 < 60 || e0 > 2030;  // (uniform)

    // the buckets, in descending order: `sub` leading bits of the significand and the exponent; powers
    // below 2^(e0 - 53) are less than half a unit in the last place of any sum
    if (!general) {
        const int vtop = (int)(((unsigned)e0 << sub) | ((1u << sub) - 1u));
        int bucket[R], place[R];
        bool crowded = false;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int e = (int)(pb[r] >> 52);
            bucket[r] = e0 - e <= 53 ? vtop - (int)(pb[r] >> (52 - sub)) : -1;
            if (bucket[r] < 0) continue;
            const int sh = 8 * (bucket[r] & 3);
            place[r] = (int)(atomicAdd(reinterpret_cast<unsigned *>(s_cnt) + (bucket[r] >> 2), 1u << sh) >> sh & 255u);
            crowded |= place[r] >= 64;  // (seen before a byte can overflow)
        }
        __syncthreads();
        const uint4 c = s_cnt[tid];
        const unsigned own = __dp4a(c.x, 0x01010101u, __dp4a(c.y, 0x01010101u, __dp4a(c.z, 0x01010101u,
                             __dp4a(c.w, 0x01010101u, 0u))));
        unsigned incl = own;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
        }
        if (lane == 31) s_wcnt[wid] = incl;
        general = __syncthreads_or(crowded);
        if (!general) {
            const unsigned cnt = lane < nw ? s_wcnt[lane] : 0u;
            const int n = (int)__reduce_add_sync(0xffffffffu, cnt);  // modes that count
            const int first = (int)(__reduce_add_sync(0xffffffffu, lane < wid ? cnt : 0u) + incl - own);
            s_off[tid] = first;
            __syncthreads();
            int size[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (bucket[r] < 0) continue;
                // the bucket's first place: its group's and the sizes of the buckets before it
                const uint4 g = s_cnt[bucket[r] >> 4];
                const int w = (bucket[r] >> 2) & 3, sh = 8 * (bucket[r] & 3);
                const unsigned mine = w == 0 ? g.x : w == 1 ? g.y : w == 2 ? g.z : g.w;
                unsigned at = __dp4a(mine & ((1u << sh) - 1u), 0x01010101u, (unsigned)s_off[bucket[r] >> 4]);
                at = __dp4a(w > 0 ? g.x : 0u, 0x01010101u, at);
                at = __dp4a(w > 1 ? g.y : 0u, 0x01010101u, at);
                at = __dp4a(w > 2 ? g.z : 0u, 0x01010101u, at);
                size[r] = (int)(mine >> sh & 255u);
                place[r] += (int)at;
                size[r] |= (int)at << 8;
                s_raw[place[r]] = pb[r];
                s_rix[place[r]] = (unsigned short)(r * nt + tid);
            }
            __syncthreads();
            // a mode's place: the modes of its bucket that come before it (larger, or as large and of
            // lower index)
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (bucket[r] < 0) continue;
                const int b0 = size[r] >> 8, b1 = b0 + (size[r] & 255), self = place[r];
                if (b1 - b0 == 1) continue;
                place[r] = b0;
                for (int q = b0; q < b1; ++q) {
                    const u64 o = s_raw[q];
                    if (o > pb[r])
                        ++place[r];
                    else if (o == pb[r] && q != self && (int)s_rix[q] < r * nt + tid)
                        ++place[r];
                }
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (bucket[r] < 0) continue;
                s_key[place[r]] = pb[r];
                s_ix[place[r]] = (unsigned short)(r * nt + tid);
            }
            __syncthreads();

            // the cumulative sums c_j = fl(c_{j-1} + p_j) of the ranks p0 .. p0 + 3
            u64 pm[R], cj[R];
            int pe[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                const u64 b = p0 + r < n ? s_key[p0 + r] : 0ull;
                pb[r] = b;
                pm[r] = (b & kFrac) | (kFrac + 1ull);
                pe[r] = (int)(b >> 52);
                cj[r] = b;  // (rank 0)
            }
            // One round over the ranks a .. lim - 1 from the sum with bits c: integer prefix sums up to
            // the first step that leaves the binade (the integer reaches 2^53) or ties.
            u64 q[R], m[R], run;
            bool tie[R];
            auto add_up = [&](int a, int lim, int E) {  // -> the warp's inclusive prefix of the threads' sums
                run = 0ull;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int j = p0 + r;
                    tie[r] = false;
                    q[r] = j >= a && j < lim ? select_q(pm[r], E - pe[r], tie[r]) : 0ull;
                    run += q[r];
                }
                u64 incl = run;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const u64 v = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += v;
                }
                return incl;
            };
            auto first_exit = [&](int a, int lim, u64 base) {
                int jx = 0x7fffffff;
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    base += q[r];
                    m[r] = base;
                    const int j = p0 + r;
                    if (j >= a && j < lim && (base >= kTop || tie[r])) jx = min(jx, j);
                }
                return (int)__reduce_min_sync(0xffffffffu, (unsigned)jx);
            };
            // the sums of the ranks before the exit; the FP64 adder takes the exit's step
            auto settle = [&](int a, int lim, int jx, int E, u64 c) {
                const u64 ebase = (u64)(E - 1) << 52;  // bits of a sum: exponent field E, M - 2^52
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    const int j = p0 + r;
                    if (j >= a && j < lim && j < jx) cj[r] = ebase + m[r];
                    if (j == jx) {
                        const u64 prev = j == a ? c : ebase + (m[r] - q[r]);
                        cj[r] = (u64)__double_as_longlong(
                            __dadd_rn(__longlong_as_double((long long)prev), __longlong_as_double((long long)pb[r])));
                    }
                }
            };
            const int lim0 = min(n, 32 * R);
            if (wid == 0) {  // the first 128 ranks
                int a = 1;
                u64 c = s_key[0];
                double sum = __longlong_as_double((long long)c);
#pragma unroll
                for (int j = 1; j < kSelectChain; ++j) {  // the first few one by one
                    if (j >= lim0) break;
                    sum = __dadd_rn(sum, __longlong_as_double((long long)s_key[j]));
                    if (lane == j / R) cj[j % R] = (u64)__double_as_longlong(sum);
                    a = j + 1;
                }
                c = (u64)__double_as_longlong(sum);
                for (int round = 0; a < lim0 && round < kSelectMaxRounds; ++round) {
                    const int E = (int)(c >> 52);
                    const u64 incl = add_up(a, lim0, E);
                    const int jx = first_exit(a, lim0, ((c & kFrac) | (kFrac + 1ull)) + (incl - run));
                    settle(a, lim0, jx, E, c);
                    const int last = min(jx, lim0 - 1);
                    u64 mine = cj[0];
#pragma unroll
                    for (int r = 1; r < R; ++r)
                        if ((last & (R - 1)) == r) mine = cj[r];
                    c = __shfl_sync(0xffffffffu, mine, last / R);
                    a = last + 1;
                }
                if (lane == 0) {
                    s_c = c;
                    s_a = a;
                }
            }
            for (int round = 0;; ++round) {
                __syncthreads();
                const int a = s_a;
                if (a >= n) break;
                if (a < lim0 || round >= kSelectMaxRounds) {  // very many ties
                    general = true;
                    break;
                }
                const u64 c = s_c;
                const int E = (int)(c >> 52);
                const bool any = R * (32 * wid + 32) > a;  // a rank of this warp is summed
                u64 incl = 0ull;
                run = 0ull;
                if (any) incl = add_up(a, n, E);
                if (lane == 31) s_wsum[wid] = incl;
                if (tid == 0) s_exit = 0x7fffffff;
                __syncthreads();
                if (any) {
                    u64 before = lane < wid ? s_wsum[lane] : 0ull;
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
                    const int jx =
                        first_exit(a, n, ((c & kFrac) | (kFrac + 1ull)) + before + (incl - run));
                    if (lane == 0 && jx != 0x7fffffff) atomicMin(&s_exit, jx);
                }
                __syncthreads();
                const int jx = s_exit;
                if (any) {
                    settle(a, n, jx, E, c);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        if (p0 + r != jx) continue;
                        s_c = cj[r];
                        s_a = jx + 1;
                    }
                }
                if (jx == 0x7fffffff) break;
            }
            if (!general) {
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (p0 + r == n - 1) s_total = cj[r];
                __syncthreads();
                const double total = __longlong_as_double((long long)s_total);
                const long long target = __double_as_longlong((1.0 - eps) * total);
                // (non-negative doubles compare as integers, and any as not less than a negative one)
                unsigned cut = 0x7fffffffu;
#pragma unroll
                for (int r = R - 1; r >= 0; --r)
                    if (p0 + r < n && (long long)cj[r] >= target) cut = (unsigned)(p0 + r);
                cut = __reduce_min_sync(0xffffffffu, cut);
                if (lane == 0 && cut != 0x7fffffffu) atomicMin(&s_cut, (int)cut);
                pdl_wait();  // the mask has been zeroed
                __syncthreads();
                const int last = s_cut;  // total >= target: some rank reaches it
#pragma unroll
                for (int r = 0; r < R; ++r)
                    if (p0 + r < n && p0 + r <= last) mask[s_ix[p0 + r]] = 1;
                return;
            }
        }
    }
    pdl_wait();
    __syncthreads();
    select_general(amp_re, amp_im, N, dbl, eps, P, mask, sel);
}

// Zeroes the mask, while the selection's blocks sort.
__global__ void k_mask_zero(unsigned char *__restrict__ mask, int N)
{
    pdl_launch_dependents();
    for (int i = threadIdx.x; i < N; i += blockDim.x) mask[i] = 0;
}

cudaError_t launch_mode_select(const double *amp_re, const double *amp_im, int K, int N,
                               const ModeDoubling &dbl, double eps, unsigned char *mask,
                               cudaStream_t st)
{
    int P = kSelectWarpSlots, sub = 3;  // 2^sub = P/16 buckets a binade: 54 binades fit in 4 P
    while (P < N) P <<= 1, ++sub;
    const int threads = P / kSelectPerThread;
    constexpr int kSlotBytes = 2 * sizeof(unsigned long long) + 2 * sizeof(unsigned short);
    const int smem = P * kSlotBytes;
    cudaError_t e = cudaFuncSetAttribute(k_mode_select, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kSelectMaxModes * kSlotBytes);
    if (e != cudaSuccess) return e;
    k_mask_zero<<<1, 1024, 0, st>>>(mask, N);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    // (reads the caller's arrays beside the plain launch above: launch.cuh)
    return launch_pdl(k_mode_select, (unsigned)K, (unsigned)threads, (size_t)smem, st, amp_re, amp_im, N, dbl, eps,
                      P, sub, mask);
}

int mode_select_max_modes() { return kSelectMaxModes; }

}  // namespace fewsum
