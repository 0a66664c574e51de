// stage_cluster.cu -- the clustered FP32C source x target kernel of one stage
// (steps a3, a5): CTA (bx, split) handles the targets of block bx against the
// root clusters split, split + splits, ... (interleaved, so that every split
// sees near and far ones alike).  The arithmetic is in stage_cluster_body.cuh.
#include <math.h>

#include <algorithm>

#include "stage_cluster_body.cuh"

namespace {

using namespace rsi_cluster;

constexpr int kTpt = 4;  // a block: 1024 targets

__device__ __forceinline__ Sum stage_sum(const ClusterArgs& a, int fi) {
    const auto& f = a.f[fi];
    Sum g;
    g.tiles = f.tiles;
    g.tile_bytes = uint32_t(a.tile_bytes);
    g.S = a.S;
    g.rec_f = 8;
    g.n_tiles = a.n_tiles;
    const Node* nodes = static_cast<const Node*>(a.nodes);
    g.nodes[0] = nodes;
    g.nodes[1] = nodes + a.n_tiles;
    g.nodes[2] = g.nodes[1] + (a.n_tiles + 3) / 4;
    g.boxes = static_cast<const Box*>(a.boxes);
    g.top = a.top;
    g.tgt = a.tgt;
    g.n_tgt = a.n_tgt;
    g.kh = f.kh;
    g.kl = f.kl;
    g.kph = f.kph;
    g.kpl = f.kpl;
    g.tp = a.tp;
    g.status = a.status;
    return g;
}

// CTA (block, split, frequency)
template <int KIND, int NORM>
__global__ void __launch_bounds__(kThreads, 2) cluster_kernel(const __grid_constant__ ClusterArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    Shared& sh = *reinterpret_cast<Shared*>(smem);
    float4* acc = reinterpret_cast<float4*>(smem + sizeof(Shared));
    int* slot = reinterpret_cast<int*>(acc + kTpt * kThreads);
    if (!gate_clustered(a.gate, a.S, a.gate_ratio)) return;
    init_shared(sh);
    const Sum g = stage_sum(a, blockIdx.z);
    const auto& f = a.f[blockIdx.z];
    run_block<StageModel<KIND, NORM>, kTpt>(StageModel<KIND, NORM>{g}, g, int64_t(blockIdx.x) * kTpt * kThreads,
                                            blockIdx.y, a.splits, a.gate->L, a.gate->h,
                                            f.part + size_t(blockIdx.y) * size_t(a.n_tgt),
                                            f.left + size_t(blockIdx.x) * size_t(a.n_tiles), f.any + blockIdx.x, sh, acc,
                                            slot);
}

// CTA (quarter block, segment, frequency)
template <int KIND, int NORM>
__global__ void __launch_bounds__(kThreads, 4) leftover_kernel(const __grid_constant__ ClusterArgs a) {
    extern __shared__ __align__(128) uint8_t smem[];
    const auto& f = a.f[blockIdx.z];
    const int block = blockIdx.x / kTpt;
    if (!f.any[block]) return;  // raised by the clustered kernel alone, so the gate need not be asked as well
    const Sum g = stage_sum(a, blockIdx.z);
    leftover_block<StageModel<KIND, NORM>, kTpt>(StageModel<KIND, NORM>{g}, g, block, blockIdx.x % kTpt, blockIdx.y,
                                                 a.segs, a.gate->L, a.gate->h,
                                                 f.left + size_t(block) * size_t(a.n_tiles),
                                                 f.part + size_t(a.splits + blockIdx.y) * size_t(a.n_tgt), smem);
}

__global__ void cluster_reduce_kernel(const __grid_constant__ ClusterArgs a) {
    const auto& f = a.f[blockIdx.y];
    if (gate_clustered(a.gate, a.S, a.gate_ratio))
        sum_block_order<kTpt>(f.part, a.splits, a.segs, f.any, int64_t(blockIdx.x) * blockDim.x + threadIdx.x, a.n_tgt,
                              a.gate->L, a.gate->h, f.field, a.status);
}

// CTAs 0 .. n_tiles - 1: a tile (if `tiles`) and its cluster each; then the
// clusters of 4 and of 16 tiles; then the rectangles of each block of targets
__global__ void __launch_bounds__(kThreads) cluster_prep_kernel(const __grid_constant__ ClusterArgs a, int tiles) {
    __shared__ __align__(8) float red[192];
    int b = blockIdx.x;
    const int groups = (a.n_tiles + 3) / 4, clusters = a.n_tiles + groups + (groups + 3) / 4;
    Node* nodes = static_cast<Node*>(const_cast<void*>(a.nodes));
    if (b >= clusters) {
        b -= clusters;
        int L, h;
        find_rows(a.tgt, a.n_tgt, kTpt * kThreads, L, h);
        Box* boxes = static_cast<Box*>(const_cast<void*>(a.boxes));
        make_boxes<kTpt>(a.tgt, a.n_tgt, int64_t(b) * kTpt * kThreads, L, h, boxes + 5 * int64_t(b), red);
        if (b == 0 && threadIdx.x == 0) *a.gate = StageGate{L, h, 0, 0};
        if (int(threadIdx.x) < a.nf) a.f[threadIdx.x].any[b] = 0;
        return;
    }
    b = clusters - 1 - b;  // the large clusters, which take longest, first
    const int mode = source_mode(a.kind, a.src, a.n_src, red);
    if (b < a.n_tiles && tiles)
        rsi_fp32::prep_tile(a.kind, a.normals, a.S, a.n_src, a.src, a.f[0].sigma, a.amp_scale, a.f[0].k, a.f[0].tiles,
                            a.tile_bytes, b, red, true, mode);
    int64_t len = a.S;
    int count = a.n_tiles;
    for (int l = 0; l < kLevels; ++l) {
        if (b < count) {
            const int64_t i0 = b * len, i1 = i0 + len < a.n_src ? i0 + len : a.n_src;
            make_node(a.kind, a.src, a.n_src, mode, i0, i1, nodes + b, red);
            return;
        }
        b -= count;
        nodes += count;
        count = (count + 3) / 4;
        len *= 4;
    }
}

// the tiles of every frequency (blockIdx.y), where the gate chose the clustered kernel
__global__ void __launch_bounds__(kThreads) cluster_tiles_kernel(const __grid_constant__ ClusterArgs a) {
    __shared__ __align__(8) float red[192];
    if (!gate_clustered(a.gate, a.S, a.gate_ratio)) return;
    const auto& f = a.f[blockIdx.y];
    rsi_fp32::prep_tile(a.kind, a.normals, a.S, a.n_src, a.src, f.sigma, a.amp_scale, f.k, f.tiles, a.tile_bytes,
                        blockIdx.x, red, true, source_mode(a.kind, a.src, a.n_src, red));
}

constexpr int kEstimates = 16;  // CTAs of the cost estimate, per frequency

__global__ void cluster_estimate_kernel(const __grid_constant__ ClusterArgs a, int blocks) {
    const int b = int(int64_t(blockIdx.x) * blocks / gridDim.x);
    Sum g = {};
    g.kh = a.f[blockIdx.y].kh;
    using Model = StageModel<RSI_STAGE_PISTON, RSI_NORMALS_Z>;  // both kinds choose and cost alike
    estimate<Model, kTpt>(Model{g}, static_cast<const Node*>(a.nodes), a.n_tiles, a.S, a.top,
                          static_cast<const Box*>(a.boxes) + 5 * int64_t(b), a.weight, blockIdx.x, a.gate);
}

int64_t target_blocks(int64_t n_tgt) { return (n_tgt + kTpt * kThreads - 1) / (kTpt * kThreads); }

template <int KIND, int NORM>
int run_t(const ClusterArgs* a, cudaStream_t s, int* occ) {
    auto kern = cluster_kernel<KIND, NORM>;
    constexpr size_t smem = smem_bytes<kTpt>();
    static RsiCtxOnce attr_set;
    if (attr_set.needed()) {
        RSI_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                     "cudaFuncSetAttribute(cluster)");
        attr_set.done();
    }
    if (!a) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(occ, kern, kThreads, smem) != cudaSuccess || *occ < 1)
            *occ = 1;
        return RSI_OK;
    }
    const unsigned blocks = unsigned(target_blocks(a->n_tgt));
    kern<<<dim3(blocks, unsigned(a->splits), unsigned(a->nf)), kThreads, smem, s>>>(*a);
    RSI_CHECK_LAUNCH("cluster_kernel");
    leftover_kernel<KIND, NORM><<<dim3(blocks * kTpt, unsigned(a->segs), unsigned(a->nf)), kThreads,
                                  leftover_smem(a->tile_bytes), s>>>(*a);
    RSI_CHECK_LAUNCH("leftover_kernel");
    return RSI_OK;
}

int dispatch(int kind, const ClusterArgs* a, cudaStream_t s, int* occ) {
    // (the ray-tracing sum's kernel has the same shared memory and registers as the piston's)
    return kind != RSI_STAGE_RSI ? run_t<RSI_STAGE_PISTON, RSI_NORMALS_Z>(a, s, occ)
                                    : run_t<RSI_STAGE_RSI, RSI_NORMALS_Z>(a, s, occ);
}

size_t align256(size_t v) { return (v + 255) & ~size_t(255); }
size_t nodes_bytes(int n_tiles) {
    const int groups = (n_tiles + 3) / 4, roots = (groups + 3) / 4;
    return align256(size_t(n_tiles + groups + roots) * sizeof(Node));
}

}  // namespace

// Clusters pay where the sum is long.  Where the device's estimate decides for the
// direct sum, its launches and the preparation cost 35 us, 8% of a sum of 5e8
// pairs and 4% of one of 1e9.  Random sums, speed with clusters offered over
// without (geometric mean): piston 5e8 .. 6e8 pairs 0.94 (single ones up to 3.9),
// 6e8 .. 7.5e8 1.05, 1e9 .. 1.5e9 1.17; interface 1e9 .. 1.5e9 1.10, 1.5e9 .. 2.5e9
// 1.33.  A piston's clusters are small beside the distance and mostly taken; an
// interface's may not be, so its sums have to be longer, and those of several
// frequencies, whose direct sum is shared, two or three times as long (9e8 and
// 7.8e8 pairs at three frequencies: no faster, and 40 us lost).  A ray costs the
// direct kernel 7 times a stage's pair: 3e8 .. 3.4e8 pairs 0.84, 4e8 .. 5e8 1.07,
// 5e8 .. 6e8 1.17.  Per-point normals turn within a tile on every curved surface,
// where the direct sum would be taken anyway.
bool cluster_plan(int kind, int normals, int nf, int64_t n_src, int64_t n_tgt, int S, int splits, int max_auto_splits,
                  ClusterPlan& p) {
    const double least = kind == RSI_TIMING_RAYTRACE ? 3.4e8
                         : kind == RSI_STAGE_PISTON   ? (nf > 1 ? 1e9 : 5e8)
                                                      : (nf > 1 ? 3e9 : 1e9);
    if (n_src < 8192 || n_tgt < 4096 || double(n_src) * double(n_tgt) < least) return false;
    if (kind == RSI_STAGE_RSI && base_normals(normals) != RSI_NORMALS_Z) return false;
    const int n_tiles = int((n_src + S - 1) / S);
    if (n_tiles >= 1 << 22) return false;  // an item's tile index has 22 bits
    const int64_t blocks = target_blocks(n_tgt);
    const int64_t roots = (n_tiles + kRootTiles - 1) / kRootTiles;
    // A batch takes 8 pairs of clusters at once: with fewer than 6 roots a CTA
    // is better off starting from the 4-tile clusters (16 batches' worth of
    // pairs per 4 roots instead of one half-empty batch)
    auto top = [](int64_t r) { return r >= 6 ? 2 : 1; };
    int occ = 1;
    dispatch(kind, nullptr, nullptr, &occ);
    const int64_t slots = int64_t(rsi_num_sms()) * occ;
    if (splits == 0) {
        double best = INFINITY;
        splits = 1;
        for (int s = 1; s <= max_auto_splits && s <= roots; ++s) {
            const int64_t rps = (roots + s - 1) / s, s_act = (roots + rps - 1) / rps;
            const int64_t batches = top(rps) == 2 ? 2 * ((rps + 7) / 8) : (4 * rps + 7) / 8;
            // blocks near the sources cost more than far ones: the last CTAs
            // end about 0.7 of a CTA's time after the work is used up
            const double waves = std::max(1.0, double(blocks * s_act * nf) / double(slots)) + 0.7;
            const double cost = waves * double(3 + 10 * batches);  // 3: a CTA's own set-up
            if (cost <= best) {
                best = cost;
                splits = int(s_act);
            }
        }
    }
    if (splits > roots) splits = int(roots);
    const int64_t rps = (roots + splits - 1) / splits;
    p.nf = nf;
    p.n_tiles = n_tiles;
    p.S = S;
    p.splits = int((roots + rps - 1) / rps);
    p.top = top(rps);
    p.fill = float(std::min(1.0, double(blocks * p.splits * nf) / double(slots)));
    // With few blocks of targets a CTA's own time and the preparation decide, which
    // the estimate does not see.  Direct and clustered, ms: rays from 44069 points
    // onto 8 blocks 2.07, 3.01, from 30000 onto 16 2.31, 2.17, from 65536 onto 16 4.81,
    // 2.84; piston 65536 onto 9 0.50, 0.54, 30000 onto 24 0.60, 0.64; interface 120000
    // onto 9 0.90, 1.01, but 262144 onto 5, 64 roots for their CTAs, 1.04, 0.76, and
    // 65536 onto 16 0.87, 0.14 to 0.78 by frequency and distance
    if (blocks < (kind == RSI_STAGE_PISTON ? 32 : 16) && roots < 64) return false;
    // The share of the direct sum's time (134.4 instructions per source and 256
    // targets, 9.2e11 per warp and second) that the estimate may reach: what is left
    // beside the preparation, the launches and the last CTAs, which end up to 0.2 ms
    // after the work is used up, for rays from tiles of 128 points 0.85 ms, over how
    // far the CTAs' own times lie above the estimate.  Fitted to 1600 random sums:
    // with 0.06 ms and 1 for all of them 184 went to a kernel more than 3% slower (the
    // worst 1.55 times), now 58 (the worst 1.30 times); 12 that clusters would speed
    // up by more than 5% keep the direct sum.
    const bool ray = kind == RSI_TIMING_RAYTRACE, piston = kind == RSI_STAGE_PISTON;
    const double direct = (ray ? 976.0 : 134.4) * double(n_src) * double(blocks * kTpt) * nf;
    const double ms = ray ? (S < 256 ? 0.85 : 0.19) : piston ? 0.16 : 0.2;
    p.gain = float(std::max(0.0, 1.0 - ms * 9.2e8 / direct) / (ray ? 1.0 : piston ? 1.2 : 1.05));
    p.tile_bytes = RSI_TILE_HDR_BYTES + size_t(S) * fp32_record_bytes(kind, base_normals(normals));
    p.tiles_bytes = align256(size_t(n_tiles) * p.tile_bytes);
    p.boxes_at = nodes_bytes(n_tiles);
    p.left_at = p.boxes_at + align256(size_t(blocks) * 5 * sizeof(Box));
    p.any_at = p.left_at + align256(size_t(nf) * size_t(blocks) * size_t(n_tiles));
    p.extra_bytes = p.any_at + align256(size_t(nf) * size_t(blocks) * sizeof(int)) + 256;
    // 16 segments: a block next to the sources is left whole, and its four
    // quarters are then 64 CTAs' work; more where there are few blocks, fewer where
    // there are many (at most 2^24 partial sums)
    p.segs = int(std::max<int64_t>(1, std::min<int64_t>({std::max<int64_t>(16, 608 / blocks), n_tiles / 4,
                                                         (int64_t(1) << 24) / n_tgt})));
    p.partial_bytes = align256(size_t(p.splits + p.segs) * size_t(n_tgt) * sizeof(double2));
    // 32 GiB of tables, an eighth of the GPU's memory, are the most that is asked
    // for beside the point sets: the mask's byte per block and tile reaches it at 9e15 pairs
    return double(p.extra_bytes) + double(nf) * double(p.partial_bytes) <= 0x1p35;
}

int cluster_prepare(const rsi_stage& st, const double* ks, float gate_ratio, const PointsView& src, int64_t n_src,
                    const double2* sigma, const TgtView& tgt, int64_t n_tgt, double2* field, const ClusterPlan& p,
                    uint8_t* base, int* status, ClusterArgs& a, cudaStream_t s) {
    a = ClusterArgs{};
    a.kind = st.kind;
    a.normals = st.kind == RSI_STAGE_RSI ? base_normals(st.normals) : RSI_NORMALS_Z;
    a.S = p.S;
    a.n_tiles = p.n_tiles;
    a.splits = p.splits;
    a.segs = p.segs;
    a.top = p.top;
    a.nf = p.nf;
    a.n_src = n_src;
    a.n_tgt = n_tgt;
    a.tile_bytes = p.tile_bytes;
    a.src = src;
    a.tgt = tgt;
    a.amp_scale = stage_amp_scale(st);
    a.tp = two_pi_split();
    uint8_t* extra = base + size_t(p.nf) * p.tiles_bytes;
    a.nodes = extra;
    a.boxes = extra + p.boxes_at;
    a.gate = reinterpret_cast<StageGate*>(extra + p.extra_bytes - 256);
    a.gate_ratio = gate_ratio * p.gain;
    a.weight = kClusterWeight / p.fill;
    a.status = status;
    for (int f = 0; f < p.nf; ++f) {
        auto& q = a.f[f];
        q.k = ks[f];
        q.kh = float(ks[f]);
        q.kl = float(ks[f] - double(q.kh));
        q.kph = float(ks[f] / M_PI);
        q.kpl = float(ks[f] / M_PI - double(q.kph));
        q.tiles = base + size_t(f) * p.tiles_bytes;
        q.sigma = sigma ? sigma + size_t(f) * size_t(n_src) : nullptr;
        q.field = field + size_t(f) * size_t(n_tgt);
        q.part = reinterpret_cast<double2*>(extra + p.extra_bytes + size_t(f) * p.partial_bytes);
        q.left = extra + p.left_at + size_t(f) * size_t(target_blocks(n_tgt)) * size_t(p.n_tiles);
        q.any = reinterpret_cast<int*>(extra + p.any_at) + size_t(f) * size_t(target_blocks(n_tgt));
    }
    const int groups = (p.n_tiles + 3) / 4, roots = (groups + 3) / 4;
    const unsigned blocks = unsigned(target_blocks(n_tgt));
    cluster_prep_kernel<<<unsigned(p.n_tiles + groups + roots) + blocks, kThreads, 0, s>>>(a, p.nf == 1 ? 1 : 0);
    RSI_CHECK_LAUNCH("cluster_prep_kernel");
    cluster_estimate_kernel<<<dim3(kEstimates, unsigned(p.nf)), kThreads, 0, s>>>(a, int(blocks));
    RSI_CHECK_LAUNCH("cluster_estimate_kernel");
    if (p.nf > 1) {
        cluster_tiles_kernel<<<dim3(unsigned(p.n_tiles), unsigned(p.nf)), kThreads, 0, s>>>(a);
        RSI_CHECK_LAUNCH("cluster_tiles_kernel");
    }
    return RSI_OK;
}

int cluster_run(const ClusterArgs& a, cudaStream_t s) {
    const int rc = dispatch(a.kind, &a, s, nullptr);
    if (rc != RSI_OK) return rc;
    cluster_reduce_kernel<<<dim3(unsigned(target_blocks(a.n_tgt) * kTpt), unsigned(a.nf)), 256, 0, s>>>(a);
    RSI_CHECK_LAUNCH("cluster_reduce_kernel");
    return RSI_OK;
}
