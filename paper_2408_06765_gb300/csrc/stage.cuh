// stage.cuh -- internal interface between the stage dispatcher (stage.cu) and
// the FP32C / FP64 source x target kernels (steps a3, a5, a6).
//
// Sources are staged as TILES: a 32-byte header followed by `S` fixed-size
// records, one tile per bulk copy into shared memory.
//   FP32C header : centre of the tile's bounding box as double-floats
//                  (xh, xl, yh, yl, zh, zl), tile radius, 0
//   FP32C record : p = P_i - centre (FP32, formed by df_diff exactly as the
//                  target offsets are), |p|^2, then
//                  PISTON  (A, 0, 0, 0)            A = -v0 w / (2 pi)
//                  RSI     (B.re, B.im, C.re, C.im) B = -w sigma / (2 pi), C = i k B
//                  [+ (nx, ny, nz, n.p) for per-point normals]
//   FP64 record  : (x, y, z, B.re, B.im, nx, ny, nz)  (PISTON: B = (A, 0))
// Padding records (past the last source) have zero amplitude and sit 4 m away.
#pragma once

#include "rsi_internal.cuh"

#define RSI_TILE_HDR_BYTES 32
#define RSI_PIPE_STAGES 3

struct TgtView {
    const float *xh, *xl, *yh, *yl, *zh, *zl;
    const double *x, *y, *z;
};

// Cody & Waite (1980) split of 2 pi into three floats; the first two carry 11
// significant bits so that n * P1 and n * P2 are exact for |n| < 2^13.
struct TwoPiSplit {
    float p1, p2, p3, inv;
};
TwoPiSplit two_pi_split();

// What the device decides for one stage (written by the clustered kernel's
// preparation, stage_cluster_body.cuh)
struct StageGate {
    int L, h;                  // rows of the target set and strip height of the block order
    unsigned long long cost;   // estimated weighted instructions of the clustered kernel over the sampled pairs
    unsigned long long pairs;  // samples: a tile and a quarter block (256 targets) each
};
// Which of the two kernels runs.  `cost`: the instructions per warp that the
// clustered kernel would take, over all the stage's frequencies, weighted by how
// much slower it issues them than the direct kernel (estimate()), and those of
// the direct sums it leaves; against the direct kernel's 16.8 per 32 pairs, 256
// S pairs per sample.  `ratio`: a multi-frequency stage's instructions per
// frequency, or a ray's per pair, over a single stage's, and the share of the
// direct sum's time that is left beside the clustered kernel's own
// (cluster_plan()).  FP32 arithmetic on integers: the same in every thread of both
// kernels.
__device__ __forceinline__ bool gate_clustered(const StageGate* g, int S, float ratio) {
    return float(g->cost) * 1.05f < float(g->pairs) * (134.4f * float(S)) * ratio;
}

// *out = sum of part[0], part[stride], ... (n terms; Neumaier, FP64, in order)
__device__ __forceinline__ void sum_partials(const double2* __restrict__ part, int n, int64_t stride, double2* out,
                                             int* status) {
    double sr = 0.0, cr = 0.0, si = 0.0, ci = 0.0;
    for (int s = 0; s < n; ++s) {
        double2 v = part[size_t(s) * size_t(stride)];
        double t = sr + v.x;
        cr += (fabs(sr) >= fabs(v.x)) ? (sr - t) + v.x : (v.x - t) + sr;
        sr = t;
        t = si + v.y;
        ci += (fabs(si) >= fabs(v.y)) ? (si - t) + v.y : (v.y - t) + si;
        si = t;
    }
    double re = sr + cr, im = si + ci;
    if (!isfinite(re) || !isfinite(im)) atomicExch(status, RSI_DEV_NONFINITE);
    *out = make_double2(re, im);
}

struct StageArgs {
    int kind;      // RSI_STAGE_*
    int normals;   // RSI_NORMALS_*
    int tpt;       // targets per thread
    int variant;   // FP32C: 1 reciprocal, 2 Newton, 3 Newton on packed source pairs (f32x2)
    int S;         // sources per tile
    int n_tiles;
    int tiles_per_split;
    int splits;
    int64_t n_tgt;
    size_t tile_bytes;
    const uint8_t* tiles;
    TgtView tgt;
    double k;
    float kh, kl;
    TwoPiSplit tp;
    double2* out;  // [splits][n_tgt] partials, or the field when splits == 1
    int* status;
    // where the clustered kernel is launched as well: the device's choice
    // between them; null: this kernel runs
    const StageGate* gate;
    float gate_ratio;
};

size_t fp32_record_bytes(int kind, int normals);
double stage_amp_scale(const rsi_stage& st);  // -v0/(2 pi) (piston) or -+1/(2 pi) (RSI)
// Reversed normals (RSI_NORMALS_NEG_Z, RSI_NORMALS_POINTS_NEG): cos(theta) is
// linear in the normal, so the kernels run with the stored normals and the
// sign goes into the source amplitudes (stage_amp_scale).
inline int base_normals(int n) {
    return n == RSI_NORMALS_NEG_Z ? RSI_NORMALS_Z : n == RSI_NORMALS_POINTS_NEG ? RSI_NORMALS_POINTS : n;
}
inline double normals_sign(int n) { return (n == RSI_NORMALS_NEG_Z || n == RSI_NORMALS_POINTS_NEG) ? -1.0 : 1.0; }
size_t fp64_record_bytes();

// packed: the pair-interleaved record layout of the packed kernel (variant 3)
int launch_prep_fp32(const rsi_stage& st, const PointsView& src, int64_t n_src, const double2* sigma,
                     int S, uint8_t* tiles, size_t tile_bytes, int n_tiles, cudaStream_t s, bool packed = false);
int launch_prep_fp64(const rsi_stage& st, const PointsView& src, int64_t n_src, const double2* sigma,
                     int S, uint8_t* tiles, size_t tile_bytes, int n_tiles, cudaStream_t s);
// Clustered FP32C kernel (stage_cluster.cu), for up to 4 frequencies of a stage
// at once.  Its workspace: per frequency the packed tiles, then `extra` (the
// clusters and the rectangles of the targets, the gate last), then per
// frequency the partial sums.
constexpr int kClusterMaxNF = 4;
constexpr float kClusterWeight = 1.5f;  // issue rate of the direct kernel (0.75 and more) over the clustered one's (0.5)
struct ClusterPlan {
    int nf, n_tiles, S, splits, top;
    int segs;    // CTAs per quarter block for the leftovers
    float fill;  // share of the GPU's CTA slots that the launch fills
    float gain;  // share of the direct sum's time that the clusters' arithmetic may take
    size_t tile_bytes, tiles_bytes, extra_bytes, partial_bytes;  // tiles and partial sums: of one frequency
    size_t boxes_at, left_at, any_at;  // within extra
    size_t total() const { return size_t(nf) * (tiles_bytes + partial_bytes) + extra_bytes; }
};
struct ClusterArgs {
    int kind, normals, S, n_tiles, splits, segs, top, nf;
    int64_t n_src, n_tgt;
    size_t tile_bytes;
    PointsView src;
    TgtView tgt;
    double amp_scale;
    TwoPiSplit tp;
    const void* nodes;  // source clusters, by level
    const void* boxes;  // target rectangles
    StageGate* gate;
    float gate_ratio, weight;
    int* status;
    struct {
        double k;
        float kh, kl, kph, kpl;  // k and k / pi
        uint8_t* tiles;
        const double2* sigma;
        double2* part;   // [splits + segs][n_tgt]
        double2* field;
        uint8_t* left;   // [blocks][n_tiles] quarters left to the direct sum
        int* any;        // [blocks] whether there are some
    } f[kClusterMaxNF];
};
// whether the clustered kernel takes stages of this kind (RSI_TIMING_RAYTRACE: the
// ray-tracing sum) and size, and its plan
bool cluster_plan(int kind, int normals, int nf, int64_t n_src, int64_t n_tgt, int S, int splits, int max_auto_splits,
                  ClusterPlan& p);
// Prepares a stage in `base` (p.total() bytes, 256-byte aligned) and writes the
// gate.  One frequency: the tiles are written in any case (the direct kernel
// reads the same ones); several: only if the gate chooses the clustered kernel.
int cluster_prepare(const rsi_stage& st, const double* ks, float gate_ratio, const PointsView& src, int64_t n_src,
                    const double2* sigma, const TgtView& tgt, int64_t n_tgt, double2* field, const ClusterPlan& p,
                    uint8_t* base, int* status, ClusterArgs& a, cudaStream_t s);
// the sums and, where the sources are split, their reduction
int cluster_run(const ClusterArgs& a, cudaStream_t s);
int launch_stage_fp32(const StageArgs& a, cudaStream_t s);
int launch_stage_fp64(const StageArgs& a, cudaStream_t s);
int fp32_threads();
int fp64_threads();
// resident CTAs per SM of the kernel a launch would use (>= 1)
int stage_occupancy_fp32(const StageArgs& a);
int stage_occupancy_fp64(const StageArgs& a);

// CUDA-event timing of a source x target kernel for rsi_timing_read: a no-op
// unless timing is enabled.  `kind` is RSI_STAGE_* or RSI_TIMING_RAYTRACE.
struct TimingScope {
    cudaEvent_t a = nullptr, b = nullptr;
};
TimingScope timing_begin(cudaStream_t s);
void timing_end(TimingScope& t, int kind, double pairs, cudaStream_t s);
// out[j] = sum over splits of part[split][j] (Neumaier, split order)
int launch_reduce_partials(const double2* part, int splits, int64_t n, double2* out, int* status, cudaStream_t s);
// the same for the direct kernel beside the clustered one: nothing is done where the gate chose the other
int launch_reduce_gated(const StageArgs& a, double2* out, cudaStream_t s);

