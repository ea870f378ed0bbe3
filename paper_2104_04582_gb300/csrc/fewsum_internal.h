// fewsum_internal.h -- device-side descriptors shared by the host API (api.cpp) and the
// kernels (spline.cu, fold.cu, sum.cu).  Plain structs: the host fills them, uploads them in
// one plan blob per call or batch, and the kernels read them.
#pragma once

#include <cstdint>
#include <mutex>
#include <cuda_runtime.h>

#include "fewsum.h"

namespace fewsum {

// Device error latch bits (few_ctx::d_err); decoded by few_sync_status.
enum : unsigned {
    ERRBIT_NONFINITE = 1u,  // non-finite value in device-resident inputs
    ERRBIT_TIMEOUT = 2u,    // a bounded mbarrier wait expired
    ERRBIT_INTERNAL = 4u    // a decoded index fell outside its table (should not happen)
};

constexpr int kMaxL = 32;
constexpr int kMaxAbsN = 1024;
// Summation kernel: up to kSumMaxThreads threads per CTA; the per-segment slot table streams
// through a ring of shared-memory stages of stage_slots slots each.
constexpr int kSumMaxThreads = 256;
constexpr int kMaxRing = 4;
constexpr int kDefaultRing = 3;
constexpr int kMinStageSlots = 16, kMaxStageSlots = 4096;

// Summation kernel variants (and the folded-coefficient layout each reads).
enum : int {
    kVariantFp64 = 0,   // FP64 throughout; slot = 8 doubles
    kVariantScalar = 1,  // mixed: FP64 phases at anchors, FP32 everything else; slot = 8 floats
    kVariantTc = 2,      // mixed: the sum over n on the tensor cores (tcsum.cu)
    kVariantTc64 = 3     // FP64: the same in exact integer slices (tcsum64.cu)
};
inline bool is_tc(int variant) { return variant == kVariantTc || variant == kVariantTc64; }

// Tensor-core summation (tcsum.cu): tiles of kTcTile consecutive samples of one segment, starting
// at multiples of kTcTile (so a sample's arithmetic does not depend on the request's slicing).
constexpr int kTcTile = 128;    // the MMA's M: one sample per tensor-memory lane
constexpr int kTcMaxPairs = 11;  // rows m and -m, max m <= 10: two accumulators of 16 columns per
                                 //   pair, beside the operands, in the 512 tensor-memory columns
constexpr int kTcMaxHalf = 31;  // half-width of the n range: 64 basis values (K)
constexpr int kTcFoldThreads = 704;
// Fold blocks that fill tile records: 128 tiles each, until there are four a multiprocessor.  FP64 (segs:
// the plan's segments, else 0): no more than 16 segments each on average, since a block forms the coefficients of
// 32 at a time, in a chain of FP64 operations, and the blocks at the dense end of the knots hold more than the
// average.  FP64 fold of 100 (1000) knots, 2 modes, 20,000 samples: 66 (208) us with 128 tiles to a block whatever
// their segments and both phases in a thread, 23 (75) so.
constexpr int kTcRecTiles = 128, kTcFillSegs = 32;
inline int tc_record_blocks(int total_tiles, int segs, int sm_count)
{
    const int t = (total_tiles + kTcRecTiles - 1) / kTcRecTiles, s = (segs + 15) / 16;
    const int n = t > s ? t : s < total_tiles ? s : total_tiles, most = 4 * sm_count;
    return n < most ? n : most;
}
// Everything the summation reads for one tile, one 128-byte line.  Phases of sample a + v, a =
// max(i0, s0): c0 + c1 v + c2 v^2 + c3 v^3 turns modulo 1, each coefficient in units of 2^-64 turn
// (64-bit wrap-around arithmetic is then the exact reduction modulo one turn).
struct alignas(128) TileRec {
    long long phi[4], r[4];
    int i0, s0, s1;       // first sample of lane 0; the segment's samples [s0, s1)
    int tile_end;         // first tile after the segment
    float u0, du;         // mixed: u of sample i is u0 + (i - s0) du; FP64: the next 32 bits (units of
                          //   2^-96 turn) of the two phases' c3, as int bits
    const void *seg;      // mixed: float, inverse of the table's power-of-two scale; FP64: TcSeg64
    const unsigned char *tab;  // the segment's operand table
    void *out;
    int pairs, ks;        // row pairs, K steps of 16 (8 powers of z_r each)
    int n_mid;            // centre of the n range
    int c64;
    // FP64: pairs also holds ks and c64 (tc64_shape), whose own words hold the next 32 bits of the phases' c2
};
static_assert(sizeof(TileRec) == 128, "one line");
__host__ __device__ inline int tc64_shape(int pairs, int ks, int c64) { return pairs | ks << 8 | c64 << 16; }
// FP64 tensor-core summation (tcsum64.cu): what a segment's tiles read beside its table.
constexpr int kTc64Slices = 7;  // 8-bit digits per operand
struct TcSeg64 {
    double inv1, inv2;        // output factors: table scale and fixed-point unit
    double tk, ih, t0, dt;    // u = (t0 + i dt - tk) ih
    int shift;                // the rows' fixed-point sums are shifted right by this
    int pad[3];
};

// Phase anchors of the mixed path: the FP64 phase splines are evaluated and reduced modulo one
// turn at every kAnchorGroup-th sample (absolute sample index a = kAnchorGroup * q), together
// with the exact Taylor coefficients of the phase cubic about that sample in sample units; the
// summation kernel adds the increment to the following samples of the group in FP32.
constexpr int kAnchorGroup = 16;
constexpr int kAnchorThreads = 128, kAnchorBlocksPerSeg = 4;  // anchor kernel grid per segment
struct Anchor {
    float4 phi;  // (f0, d1, d2, d3): reduced phase (turns) and increment coefficients (turns / sample^k)
    float4 r;
    float4 g;    // phase of the final factor z_phi^{m_last} z_r^{lo_last}, same form
};
constexpr int kFoldThreads = 128;
constexpr int kYlmThreads = 16;  // few pairs per block: spreads the FP64 work over SMs
constexpr int kBuildThreads = 64;
constexpr int kBuildParts = 8;  // blocks of a spline's partitioned solve = lanes per spline
constexpr int kBuildSplines = kBuildThreads / kBuildParts;

// Trajectory-resident data (one per few_traj).
struct TrajDev {
    int K, N, J, S;        // knots, modes, splines (2 + 2N), segments (K - 1)
    int n_pairs;           // distinct (l, m) pairs
    int n_slots;           // harmonic slots per segment
    int n_rows;            // rows of the slot table: signed m from max m down to m_last
    int m_last, lo_last;   // signed m and lowest n of the last row
    const double *t;       // [K] knot times
    const double *inv_h;   // [S] 1/(t_{k+1}-t_k)
    const double *h;       // [S] t_{k+1}-t_k
    // the partitioned factorisation of the reduced not-a-knot system (k_factor); p_k = pivot
    const double *fac_ra;  // [K] right-hand side f_k = ra_k (y_k - y_{k-1}) + rb_k (y_{k+1} - y_k):
    const double *fac_rb;  //   block rows scaled by 1/p_k, separator rows plain; rows 0 and K-1
                           //   hold the end slopes' coefficients (see k_factor)
    const double *fac_lo;  // [K] block rows: sub-diagonal / p_k (0 on a block's first row);
                           //   rows 0 and K-1: the end slopes' coupling to s_1 / s_{K-2}
    const double *fac_up;  // [K] block rows: super-diagonal / p_k
    const double *fac_ip;  // [K] inverse pivots (block rows; separator system at separator rows)
    const double *fac_v;   // [K] block responses v to the left separator (separator multipliers)
    const double *fac_x;   // [K] block responses w to the right separator (separator couplings)
    const double *fac_sinv;  // [(kBuildParts-1)^2] inverse of the separator system, row-major
    const int *parts;      // [kBuildParts + 2]: block count P, block starts, then K - 1
    double *slopes;        // [K][J] spline build scratch (parked elimination values)
    double *coef;          // [S][J][4] Hermite data of every segment: (y_k, y_{k+1}, s_k,
                           //   s_{k+1}), values and knot slopes (see hermite_to_power);
                           //   columns 0,1 = Phi_phi, Phi_r (rad),
                           //   column 2+2i / 3+2i = Re / Im A_i
    const int2 *pair_lm;   // [n_pairs] (l, m)
    const int *mode_pair;  // [N] pair index of each mode
    const int *slot_ptr;   // [n_slots + 1] CSR into contrib
    const int2 *contrib;   // [n_contrib] (mode * 2 + kind, 2 * pair + kind); kind 0: A Y+,
                           //   1: conj(A) Y-
    int tc_pairs, tc_ks;   // tensor-core summation: row pairs, K steps (tc_pairs 0: not used)
    int n_mid, m_top;      //   centre of the n range; largest m
    const int4 *row_slot;  // [n_rows] (first slot, highest n, lowest n, 0); lowest > highest: empty
    const int2 *rows;      // [n_rows] (slots of the row, lowest n of the previous row minus
                           //   this row's lowest n); a row's slots run from its highest n down
};

// Power coefficients of a segment's cubic in the local variable u = (t - t_k)/h_k, u in [0, 1],
// from its Hermite data (values y0 = y_k, y1 = y_{k+1}, slopes s0, s1, width h = h_k):
//     p(u) = y0 + a u + (3 D - 2 a - b) u^2 + (a + b - 2 D) u^3,  a = h s0, b = h s1, D = y1 - y0.
template <typename T>
__host__ __device__ __forceinline__ void hermite_to_power(T y0, T y1, T s0, T s1, T h, T (&c)[4])
{
    const T D = y1 - y0, a = h * s0, b = h * s1;
    c[0] = y0;
    c[1] = a;
    c[2] = fma((T)-2, a, fma((T)3, D, -b));
    c[3] = fma((T)-2, D, a + b);
}

// One spline-build job: a trajectory and the knot data to fit.
struct BuildJob {
    TrajDev tr;
    const double *phi_phi;  // [K] rad
    const double *phi_r;    // [K] rad
    const double *amp_re;   // [K][N]
    const double *amp_im;   // [K][N]
    int block_begin;        // first block of this job in the flattened build grid
    int pad;
};

// One waveform of a plan (a request).
struct WaveDev {
    TrajDev tr;
    double theta, phi, scale;   // source-frame viewing angles
    double dphi_phi, dphi_r;    // phase offsets (rad)
    double t0, dt;
    int n_samples;
    int out_c64;
    void *out;
    void *fcoef;          // [S][n_slots][8] folded coefficients (float or double)
    Anchor *anchors;      // mixed plans: [n_anchors] phase anchors (segment by segment)
    const int *anchor_off;  // mixed plans: [K] first anchor of each segment, then the total
    int anchor_seg_begin; // first global segment index of this wave (anchor kernel grid)
    unsigned char *tab;   // tensor-core plans: [S] operand tables of tc_table_bytes
    float *tab_inv;       //   [S] inverse table scales (mixed)
    TcSeg64 *seg64;       //   [S] segment constants (FP64)
    const int *tile_off;  //   [K] first tile of each segment, then the total
    int tile_begin;       //   first tile of this wave in the plan
    int seg_begin;        //   first segment of this wave in the plan
    double2 *ylm;         // [n_pairs][2]: Y+ = -2Y_{l,m}, Y- = (-1)^l -2Y_{l,-m} (0 if m = 0)
    const int *seg_start; // [K] sample range of each segment
    int pair_begin;       // first global pair index of this wave (ylm kernel)
    int fold_begin;       // first fold block of this wave
    int fold_blocks_per_seg;
    int rotate;           // detector frame: the harmonics are multiplied by (rot_r, rot_i)
    double rot_r, rot_i;
};

// Start of one CTA's slice of the summation work: (wave, sample).
struct CtaStart {
    int wave;
    int sample;
};

// Header of a plan blob.  The blob is [PlanHdr][WaveDev x n][CtaStart x (grid+1)][ints...].
struct PlanHdr {
    int n_waves;
    int total_pairs;
    int total_fold_blocks;
    int grid_sum;
    int total_anchor_segs;  // segments over all waves of a mixed plan (0 for FP64 plans)
    int buf_bytes;   // bytes of one ring stage (stage_slots x slot bytes, rounded up)
    int stage_slots; // slots per ring stage (the mode tile)
    int ring;        // ring stages
    int variant;     // kVariant* of the summation kernel and the folded layout
    int total_segs, total_tiles;  // tensor-core plans
    const int *tile_cta;  //   [grid + 1] first tile of each CTA
    TileRec *recs;        //   [total_tiles]
    const unsigned char *self;    // the plan's device address
    const WaveDev *waves;
    const CtaStart *cta;
    unsigned *err;
};

// A plan small enough to travel as a kernel parameter (no upload): its bytes, to be read at
// `bytes` and copied to device address `dev`, for which its pointers into itself are made.
constexpr int kPlanParamBytes = 6144;
struct alignas(16) PlanParam {
    unsigned char bytes[kPlanParamBytes];
    unsigned char *dev;
    int n;
};
// Kernel launchers (defined in the .cu files; every launcher returns the launch error).
// Output arrays of k_factor (the trajectory's TrajDev fields of the same names).
struct FactorArrays {
    double *h, *inv_h, *ra, *rb, *lo, *up, *ip, *v, *x, *sinv;
    int *parts;
};
cudaError_t launch_factor(const double *t, int K, const FactorArrays &f, cudaStream_t st);
cudaError_t launch_build(const BuildJob *jobs_dev, int n_jobs, int total_blocks,
                         int max_knots, unsigned *err, cudaStream_t st);
// One trajectory's build, the job as a kernel parameter.
cudaError_t launch_build_one(const BuildJob &job, int blocks, unsigned *err, cudaStream_t st);
cudaError_t launch_ylm(const PlanHdr *hdr_dev, const PlanParam *plan, int total_pairs, bool fp64,
                       cudaStream_t st);
cudaError_t launch_fold(const PlanHdr *hdr_dev, int total_fold_blocks, bool fp64, cudaStream_t st);
cudaError_t launch_anchor(const PlanHdr *hdr_dev, int total_anchor_segs, cudaStream_t st);
// Anchors of one segment's samples [s_begin, s_end): groups floor(s_begin / G) ..
// floor((s_end - 1) / G); none for an empty segment.
inline int anchors_in_segment(int s_begin, int s_end)
{
    return s_end > s_begin ? (s_end - 1) / kAnchorGroup - s_begin / kAnchorGroup + 1 : 0;
}
cudaError_t launch_wait_selftest(unsigned *err, unsigned limit_us, cudaStream_t st);
cudaError_t launch_sum(const PlanHdr *hdr_dev, int grid, int threads, int samples_per_thread,
                       int smem_bytes, int variant, cudaStream_t st);
// Bytes of one segment's tensor-core operand table: fp16 high and low parts, N = 16 pairs rows of
// 16 ks columns each.
__host__ __device__ inline int tc_table_bytes(int pairs, int ks) { return 1024 * pairs * ks; }
// FP64: 7 digit slices, each row pair's 16 rows of 16 ks fp16 columns together.
__host__ __device__ inline int tc64_table_bytes(int pairs, int ks) { return 512 * kTc64Slices * pairs * ks; }
// Bytes of a segment's table and constants.
inline size_t tc_segment_bytes(bool fp64, int pairs, int ks)
{
    return fp64 ? tc64_table_bytes(pairs, ks) + sizeof(TcSeg64) : tc_table_bytes(pairs, ks) + sizeof(float);
}
// Relative cost of one tile, as measured (mixed: ns; its per-sample work around the MMAs is
// nearly the same for every mode set): pairs of the wave, K steps of the plan's widest.
inline double tc_tile_cost(bool fp64, int pairs, int ks)
{
    return fp64 ? 1900.0 + 690.0 * pairs + 650.0 * ks : 390.0 + 9.0 * pairs + 43.0 * ks;
}
inline int tiles_in_segment(int s_begin, int s_end)
{
    return s_end > s_begin ? (s_end - 1) / kTcTile - s_begin / kTcTile + 1 : 0;
}
// What the choice between the two summations looks at: a mode set and a request's segments.
struct TcShape {
    int pairs, ks, slots, rows, modes, K;
};
struct TcWork {
    double samples = 0.0, segs = 0.0, passes = 0.0, tiles = 0.0;  // segments with samples; passes of 256
    void add(long long s0, long long s1)
    {
        if (s1 <= s0) return;
        samples += (double)(s1 - s0);
        segs += 1.0;
        passes += (double)((s1 - s0 + 255) / 256);
        tiles += tiles_in_segment((int)s0, (int)s1);
    }
};
// Sets of more frequencies are always faster on the tensor cores.
constexpr int kTcAlwaysSlots = 128;
// Whether the tensor-core summation is the faster one (not past kTcMaxPairs, kTcMaxHalf).  A tile, a
// segment's table and an FP64 record cost about the same for one mode as for a hundred, a slot of the scalar
// chain next to nothing, so sets of a few frequencies stay with the scalar chain where there is enough of the
// one or the other.  Both sides in us, as measured (tensor cores against scalar):
//   mixed, long waveforms:  40 M samples, one frequency pair (m, n) = (2, 0): 884, 740; 18 slots: 885, 979;
//                           3.2 M samples, one pair: 82, 90
//   FP64, short segments:   one pair: 4096 knots, 20,000 samples 371, 229; 1000 knots, 1,000 samples
//                           110, 77; 100 knots, 20,000 samples 38, 61; m = 10: 4096 knots, a million samples
//                           1159, 886; m = 10, n = 0 and 30: 300 knots, 20,000 samples 135, 110;
//                           99 slots: 4096 knots, 20,000 samples 534, 784
// The estimates are fits to such times, good to 20 %; where they are near one another the tensor cores, the more
// exact of the two, are taken (FP64).
// A batch's waveforms share the launches, and what they add to it decides: 48 FP64 waveforms of 50 knots and 300
// samples, two modes of m = 10: 402, 176; one pair, 300 knots, 3,000 samples: 1179, 685.  A request takes the same
// chain alone and in a batch (its results do not depend on the others), so the tensor cores must also add at most a
// tenth more there (fits to 10 %).
inline bool tc_pays(bool fp64, const TcShape &s, const TcWork &w)
{
    if (s.slots > kTcAlwaysSlots) return true;
    if (!fp64) {
        const double scalar = 34.0 + 0.037 * w.segs + 1e-6 * w.samples * (16.1 + 0.3 * s.slots + 0.315 * s.rows);
        const double tc = 13.0 + 0.012 * w.segs + w.tiles * 0.93e-3 * tc_tile_cost(false, s.pairs, s.ks) / 152.0;
        return tc < scalar;
    }
    const double scalar = 36.0 + 0.005 * s.K + w.segs * (0.003 + 0.00015 * s.modes) +
                          w.passes * (0.03 + 0.0012 * s.slots + 0.00075 * s.rows) +
                          0.7e-3 * w.samples * (0.27 + 0.018 * s.slots + 0.012 * s.rows);
    const double tc = (8 * s.K + 2048 <= kPlanParamBytes ? 28.0 : 47.0) +
                      w.segs * (0.045 + s.pairs * (0.006 + 0.0045 * (s.ks - 1)) + 0.0001 * s.modes) +
                      w.tiles * (0.6 + 0.85 * s.pairs + 0.7 * (s.ks - 1)) / 152.0;
    if (0.9 * tc >= scalar || w.passes == 0.0) return false;
    const double fill = w.samples / w.passes;  // samples a pass
    const double adds_scalar = 0.033 * w.segs + w.passes / 152.0 * (1.0 + 0.188 * s.slots + 0.11 * s.rows +
                                                                    fill * (0.0356 + 0.00277 * s.slots + 0.00172 * s.rows));
    const double adds_tc = w.segs * (0.0433 + s.pairs * (0.0047 + 0.0052 * (s.ks - 1))) +
                           w.tiles * (0.0127 + 0.004 * s.pairs + (0.0046 + 0.0002 * s.pairs) * (s.ks - 1));
    return adds_tc < 1.1 * adds_scalar;
}
cudaError_t tc_configure();
cudaError_t tc64_configure();
cudaError_t launch_fold_tc64(const PlanHdr *hdr_dev, int total_segs, int total_tiles, int sm_count, cudaStream_t st);
cudaError_t launch_sum_tc64(const PlanHdr *hdr_dev, int grid, int ks, cudaStream_t st);
// plan: the plan itself (the kernel then writes it to hdr_dev for those that follow), or null when it
// is at hdr_dev already.
cudaError_t launch_fold_tc(const PlanHdr *hdr_dev, const PlanParam *plan, int total_segs, int total_tiles,
                           int sm_count, cudaStream_t st);
// ks: the most K steps of any wave of the plan.
cudaError_t launch_sum_tc(const PlanHdr *hdr_dev, int grid, int ks, cudaStream_t st);
// Bytes of one folded slot in the layout a variant reads.
int sum_slot_bytes(int variant);
cudaError_t launch_phases(const TrajDev &tr, const int *seg_start, double t0, double dt, int n,
                          double dphi_phi, double dphi_r, double *out, cudaStream_t st);
// Mode Selector: at most kSelectMaxModes modes; which of them stand for an m < 0 partner too
// (m > 0, power doubled) travels as one bit per mode (bit i % 32 of word i / 32) in the launch
// parameters, so a call needs no device allocation or copy.
constexpr int kSelectMaxModes = 4096;
struct ModeDoubling {
    unsigned w[kSelectMaxModes / 32];
};
cudaError_t launch_mode_select(const double *amp_re, const double *amp_im, int K, int N,
                               const ModeDoubling &dbl, double eps, unsigned char *mask,
                               cudaStream_t st);
int mode_select_max_modes();
cudaError_t launch_direct(const double *pphi, const double *pr, const double *are,
                          const double *aim, long long ns, const int *l, const int *m, const int *n,
                          int N, double theta, double phi, double scale, bool fp64, void *out,
                          int out_c64, void *mode_consts, int l_top, int m_top, int n_lo, int n_hi, int sm_count,
                          unsigned *err, cudaStream_t st);
size_t direct_mode_const_bytes(int N);
cudaError_t direct_configure();
// Reduced-basis amplitudes (rb.cu): tile counts of the packed tensor-core operands.
struct RbLayout {
    int n_kb = 0, n_tiles = 0, m_tiles = 0, modes_padded = 0, rows_padded = 0;
    int groups = 0, step = 0;  // groups of 32 modes, and modes between their first ones
    size_t bpack_bytes = 0, apack_bytes = 0;
};
RbLayout rb_layout(int Nb, int N, int M);
// FP64 amplitudes from digit slices (rb64.cu).
struct Rb64Args {
    const unsigned char *bpack, *apack;
    const int *bexp, *aexp;
    const double *are, *aim, *bre, *bim;  // for the outputs left to the plain chain
    const double *scale;                  // [M] or null
    double *out_re, *out_im;
    int M, N, Nb, steps, tiles, per;
    unsigned *err;
};
size_t rb64_basis_bytes(int Nb, int N);
size_t rb64_coef_bytes(int Nb, int M);
int rb64_rows(int M);    // padded counts
int rb64_modes(int N);
cudaError_t rb64_configure();
// The basis columns' scaling exponents of both products (bexp64 null: of the mixed one).
cudaError_t launch_rb_exponents(const double *bre, const double *bim, int Nb, int N, int n_exp, int *bexp, int *bexp64,
                                cudaStream_t st);
cudaError_t launch_rb64_basis(const double *bre, const double *bim, int Nb, int N, const int *bexp, unsigned char *pack,
                              int sm_count, cudaStream_t st);
// after_scale: the kernel launched before it on `st` forms the scale.
cudaError_t launch_rb64(Rb64Args a, unsigned char *apack, int *aexp, bool after_scale, cudaStream_t st);
cudaError_t launch_rb_basis(const double *bre, const double *bim, int Nb, int N, double2 *gt64,
                            float2 *gt32, const int *bexp, unsigned char *bpack, int sm_count, cudaStream_t st);
cudaError_t launch_rb(const double *are, const double *aim, int M, int Nb, int N, const double *nu,
                      bool fp64, const double *bre, const double *bim, const double2 *gt64,
                      const float2 *gt32, const int *bexp, const unsigned char *bpack, double *scale,
                      int *aexp, unsigned char *apack, const int *bexp64, const unsigned char *bpack64,
                      double *ore, double *oim, unsigned *err,
                      int sm_count, cudaStream_t st, cudaStream_t side, cudaEvent_t fork_ev,
                      cudaEvent_t join_ev);
// Maximum resident CTAs per SM of the summation kernel for a configuration (0 if invalid).
int sum_occupancy(int variant, int samples_per_thread, int threads, int smem_bytes);
// One-time kernel attribute setup (dynamic shared memory opt-in).
cudaError_t sum_configure();

// Makes `device` current for the lifetime of the object and then restores the caller's current
// device, so a library call never leaves a different device current behind.
struct DeviceScope {
    int prev = -1;
    bool ok = false;
    explicit DeviceScope(int device)
    {
        if (cudaGetDevice(&prev) != cudaSuccess) {
            prev = -1;
            (void)cudaGetLastError();
        }
        ok = cudaSetDevice(device) == cudaSuccess;
        if (!ok) (void)cudaGetLastError();
    }
    ~DeviceScope()
    {
        if (prev >= 0) cudaSetDevice(prev);
    }
    DeviceScope(const DeviceScope &) = delete;
    DeviceScope &operator=(const DeviceScope &) = delete;
};

// Host validation of one request (few_waveform's checks; need_device_out additionally requires
// out_where == FEW_MEM_DEVICE).
few_status check_request(const few_request &r, bool need_device_out);
// Viewing direction and frame constant of a request.
void set_wave_angles(const few_request &r, WaveDev &W);

// Read-only snapshot of a context and one of its trajectories (filled by api.cpp).
struct CtxTrajView {
    int device, sm_count;
    unsigned *d_err;
    int tile_R[2], tile_T[2], tile_S[2];
    bool has_data;
    int K, n_slots, n_pairs, tc_pairs, tc_ks;
    const double *t_host;
    TrajDev dev;
};
bool ctx_traj_view(few_ctx *ctx, const few_traj *tr, CtxTrajView *v);
std::recursive_mutex &ctx_mutex(few_ctx *ctx);

}  // namespace fewsum
