// stage_cluster_body.cuh -- device code of the clustered FP32C source x target
// sum (steps a3, a5).
//
// A cluster of sources and a cluster of targets that are far enough apart
// interact through few numbers.  With c and b their centres, d = b - c, and p,
// q the offsets from them, the distance splits as
//   r(p, q) = |d - p| + (|d + q| - |d|) + delta(p, q),
// where delta vanishes for p = 0 or q = 0: the first two parts leave the sum
// as factors of the source and of the target, and what remains, e^{ik delta}
// times 1/r and the obliquity, is a smooth function of p and q.  It is
// interpolated on N x N Chebyshev nodes of each cluster's rectangle (N = 6, 8,
// 10 or 12, by choose_nodes()):
//   moments  M_m   = sum_i L_m(p_i) B_i e^{ik |d - p_i|}
//   nodes    F_m'  = sum_m M_m e^{ik (delta(p_m, q_m') - |d|)} g(p_m, q_m')
//   targets  phi_j += e^{ik |b - c + q_j|} sum_m' L_m'(q_j) F_m'
// N^4 pair terms and 2 N^2 (S + T) multiply-adds in place of S T pair terms.
// Sources are clustered in tiles (256), groups of 4 tiles and of 16 tiles,
// targets in blocks of 1024 and their quarters; each pair is taken at the
// coarsest level that choose_nodes() admits, and pairs of a tile and a quarter
// that it does not admit (too close or thick) take the
// direct sum (stage_fp32_body.cuh).
//
// Accuracy.  The phases of sources and targets are formed as the direct sum
// forms them: a double-float reference |b - c_tile| (or |Q_j - c|) with
// k r mod 2 pi, and an FP32 offset within the tile.  At the nodes delta comes
// from differences that cancel exactly (node_pair2), to about 2^-23 of itself.
//
// A warp takes a pair of clusters through moments and nodes on its own (no
// barrier of the block), eight pairs at a time; then every thread adds the
// eight fields at its targets.
#pragma once

#include "stage_fp32_body.cuh"

namespace rsi_cluster {

using rsi_fp32::kThreads;
using rsi_fp32::rsqrt_approx;

constexpr int kWarps = kThreads / 32;
constexpr int kMaxN = 12, kMaxNN = kMaxN * kMaxN;
constexpr int kLevels = 3;  // tiles, groups of 4 tiles, groups of 16 tiles
constexpr int kRootTiles = 16;
constexpr int kRound = 256;  // tiles whose level is decided at once, one per thread

// What is kept of a source cluster (32 floats)
struct Node {
    float c[6];            // centre of its rectangle, (hi, lo) per axis
    float e1[3], e2[3], e3[3];  // unit axes; e3 is the plane's normal
    float h1, h2, h3;      // half sizes along them
    float flat;            // 1: every coordinate is a number (the obliquity's normal is e3 everywhere)
    float pad[13];
};
static_assert(sizeof(Node) == 128, "node");

// a target cluster: the block (0) or one of its quarters (1 + q)
struct Box {
    float c[6];
    float q1, q2, q3;  // half sizes along axes ax1, ax2 and the third
    int ax1, ax2;
    float o1, o2;  // the block's centre in this box's coordinates
    float pad[3];
};

// Chebyshev tables C_N[a][k] = c_k U_k(x_a).  U_k = s_k T_k with the signs
// s = + + - - + + - - ...: U_{k+1} = (s_k s_{k+1}) 2x U_k + U_{k-1} has no
// negated term (a packed negation would be an instruction of its own), and
// s_k^2 = 1 in every product of a table entry and a basis value.
__host__ __device__ constexpr int tab_off(int n) { return n == 6 ? 0 : n == 8 ? 36 : n == 10 ? 100 : 200; }
constexpr int kTabFloats = 344;

constexpr int kRowFloats = 32 * (4 * kMaxN + 4);  // 32 source pairs: U_k(xi), U_l(eta), B e^{i..}
struct alignas(16) WarpArea {
    float rows[kRowFloats];  // later the source nodes' records
    float2 x[kMaxNN];        // partial moments (x and y); the field at the target nodes
    float2 y[kMaxNN];        // between the two passes of a transform
    float2 fh[kMaxNN];       // Chebyshev coefficients of the field on the target cluster
    Node node;
    float D1h, D1l, D2h, D2l, S0h, S0l;  // prepare_targets' D along the block's axes, and |D|^2
    int item;                // level, tile, target cluster, N (0: none)
    int pad;
};

struct Shared {
    WarpArea w[kWarps];
    float tab[kTabFloats];
    Box box[5];
    int items[kRound * 4];
    int warp_sum[kWarps];
};

// items: bits 0-3 N, 4-6 target cluster, 7-8 level, 9- first tile
__device__ __forceinline__ int make_item(int n, int box, int level, int tile) {
    return n | (box << 4) | (level << 7) | (tile << 9);
}

template <int TPT>
constexpr size_t smem_bytes() {
    return sizeof(Shared) + TPT * kThreads * (sizeof(float4) + sizeof(int));
}

// Slot of the t-th target of the block order.  A set of n targets in rows of
// L (an image grid) is cut into strips of h rows, each walked column by
// column and every other one backwards, so that consecutive targets are
// compact patches; L = 0: the slots' own order (QMC sets are in cell order).
__device__ __forceinline__ int64_t strip_slot(int64_t t, int64_t n, int L, int h) {
    if (L <= 0) return t;
    const uint32_t rows = uint32_t(n) / uint32_t(L), per = uint32_t(L) * uint32_t(h), u = uint32_t(t);
    const uint32_t s = u / per, v = u - s * per;
    const uint32_t hs = min(uint32_t(h), rows - s * uint32_t(h));
    uint32_t c = v / hs;
    const uint32_t r = v - c * hs;
    if (s & 1u) c = uint32_t(L) - 1u - c;
    return int64_t(s * uint32_t(h) + r) * L + c;
}
// Position within a block of 1024 of its i-th target.  In strips of h = 2^b
// rows a block is 2^(10-b) columns of h, and quarter i >> 8 = (upper half of
// the columns, upper half of the rows) one patch of it.
template <int TPT>
__device__ __forceinline__ int block_pos(int i, int h) {
    if (TPT != 4 || h < 2 || h > 512) return i;
    const int b = 31 - __clz(h), lo = (1 << (b - 1)) - 1;  // i = [c r | c... r...] -> column * h + row
    return (i & 512) | (((i & 255) >> (b - 1)) << b) | (((i >> 8) & 1) << (b - 1)) | (i & lo);
}

// Nodes per axis for a phase excursion phi and a relative size sep.  The lines
// phi(sep) were fitted to the largest error over random pairs of rectangles
// (tilts, shapes and directions): below about 5e-7 of the term's magnitude,
// 5e-8 root mean square, against 5e-7 to 1e-6 of FP32 rounding per pair term.
__device__ __forceinline__ int nodes_for(float phi, float sep) {
    if (sep <= 0.25f && phi <= 0.45f - 1.5f * sep) return 6;
    if (sep <= 0.28f && phi <= 1.15f - 1.8f * sep) return 8;
    if (sep <= 0.36f && phi <= 2.0f - 2.0f * sep) return 10;
    if (sep <= 0.42f && phi <= 3.0f - 2.0f * sep) return 12;
    return 0;
}

// Nodes per axis for a source cluster and a target cluster, 0 if they are not
// admitted.  phi bounds the phase k delta that one axis of either rectangle
// sees: its bilinear part (k / R) (u_a . v_b - (u_a . d/R)(v_b . d/R)) h_a q_b
// summed over the other rectangle's axes, plus the cubic terms' size; sep is
// the two rectangles' half diagonals over R.
__device__ __forceinline__ int choose_nodes(const Node& s, const Box& b, float k) {
    if (!(s.flat > 0.0f) || b.q3 != 0.0f) return 0;
    float d[3], lo;
    df_diff(b.c[0], b.c[1], s.c[0], s.c[1], d[0], lo);
    df_diff(b.c[2], b.c[3], s.c[2], s.c[3], d[1], lo);
    df_diff(b.c[4], b.c[5], s.c[4], s.c[5], d[2], lo);
    const float R = sqrtf(fmaf(d[0], d[0], fmaf(d[1], d[1], d[2] * d[2])));
    if (!(R > 0.0f)) return 0;
    const float iR = 1.0f / R;
    const float hd = sqrtf(s.h1 * s.h1 + s.h2 * s.h2), qd = sqrtf(b.q1 * b.q1 + b.q2 * b.q2);
    const float sep = (hd + qd) * iR;
    // what the rectangle leaves out: sources off its plane
    if (!((k * qd + 1.0f) * s.h3 * iR <= 5e-7f)) return 0;
    const float d1 = (d[0] * s.e1[0] + d[1] * s.e1[1] + d[2] * s.e1[2]) * iR;
    const float d2 = (d[0] * s.e2[0] + d[1] * s.e2[1] + d[2] * s.e2[2]) * iR;
    const float v1 = (b.ax1 == 0 ? d[0] : d[1]) * iR, v2 = (b.ax2 == 1 ? d[1] : d[2]) * iR;
    const float u11 = b.ax1 == 0 ? s.e1[0] : s.e1[1], u12 = b.ax2 == 1 ? s.e1[1] : s.e1[2];
    const float u21 = b.ax1 == 0 ? s.e2[0] : s.e2[1], u22 = b.ax2 == 1 ? s.e2[1] : s.e2[2];
    const float f = k * iR;
    const float m11 = f * fabsf(u11 - d1 * v1) * s.h1 * b.q1, m12 = f * fabsf(u12 - d1 * v2) * s.h1 * b.q2;
    const float m21 = f * fabsf(u21 - d2 * v1) * s.h2 * b.q1, m22 = f * fabsf(u22 - d2 * v2) * s.h2 * b.q2;
    const float phi = fmaxf(fmaxf(m11 + m12, m21 + m22), fmaxf(m11 + m21, m12 + m22)) + f * hd * qd * sep;
    return nodes_for(phi, sep);
}

// |d - p| - R for an offset p: th = (|d - p|^2 - R^2) / 2, one Newton step
__device__ __forceinline__ float path_diff(float th, float R, float R2) {
    const float r2 = fmaf(2.0f, th, R2);
    const float ir = rsqrt_approx(r2);
    const float r0 = r2 * ir;
    const float am = r0 - R;
    const float eh = fmaf(am, -0.5f * (r0 + R), th);
    return fmaf(eh, ir, am);
}

// A target node: offset (q1, q2) along the box's axes, R = |d + q|, cr = the
// relative rounding error of R with its sign turned (true R = R (1 - cr))
struct NodeRef {
    float2 q1, q2, R2, nR, nRh, cr;
};

// Instructions per warp that a pair of a source cluster of `ns` sources and a
// target cluster of `nt` targets takes with N x N nodes: `src` of them for 64
// sources' phases, `node` for two source nodes onto 32 target nodes, `tgt` for
// 32 targets beside the interpolation (counted in the code)
__device__ __forceinline__ float pair_cost(float ns, float nt, int N, float node, float tgt, float src) {
    const float n = float(N), nn = n * n;
    const float rounds = N == 6 ? 3.0f : ceilf(nn * (1.0f / 32.0f)), pairs = N == 6 ? 9.0f : 0.5f * nn;
    return 150.0f + ns * (1.0f / 64.0f) * (src + (4.0f + 2.5f * n) * (32 / (32 / N))) +
           rounds * (1.7f * node + node * pairs) + nt * (1.0f / 32.0f) * (tgt + 1.5f * nn + 4.0f * n) +
           4.0f * ceilf(nn * (1.0f / 32.0f)) * (3.0f * n + 15.0f);
}

// Two source nodes onto one target node.  Records (pair-interleaved):
// v0 = p along the target box's axes (p1, p1', p2, p2'), v1 = t, a_hi, with
// t = (|d - p|^2 - |d|^2) / 2 and a = |d - p| - |d| = a_hi + a_lo, v2 = a_lo,
// beta, v3 = m.  r^2 = R^2 + 2 (t - q.p); r - R comes from one Newton step as
// in the direct sum, its residual (r0 - R)(r0 + R)/2 - t an exact difference
// up to q.p, so that delta = r - R - a carries about 2^-23 |q.p| / R of error.
template <int KIND>
__device__ __forceinline__ void node_pair2(const NodeRef& n, const float4& v0, const float4& v1, const float4& v2,
                                           const float4& v3, float2 k, float2& a1, float2& a2, float2& b1,
                                           float2& b2) {
    const float2 nqp = __ffma2_rn(n.q1, make_float2(v0.x, v0.y), __fmul2_rn(n.q2, make_float2(v0.z, v0.w)));  // -q.p
    const float2 t = make_float2(v1.x, v1.y);
    const float2 r2 = __ffma2_rn(__fadd2_rn(t, nqp), make_float2(2.0f, 2.0f), n.R2);
    const float2 ir = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
    const float2 r0 = __fmul2_rn(r2, ir);
    const float2 am = __fadd2_rn(r0, n.nR);                                   // r0 - R, exact
    const float2 hs = __ffma2_rn(r0, make_float2(-0.5f, -0.5f), n.nRh);       // -(r0 + R)/2
    const float2 eh = __fadd2_rn(__ffma2_rn(am, hs, t), nqp);                 // (r^2 - r0^2)/2
    const float2 lo = __ffma2_rn(n.cr, am, make_float2(v2.x, v2.y));          // correction of R, -a_lo
    const float2 dl = __fadd2_rn(__fadd2_rn(am, make_float2(v1.z, v1.w)), __ffma2_rn(eh, ir, lo));
    const float2 u = __ffma2_rn(k, dl, make_float2(v2.z, v2.w));
    float2 sn, cs;
    __sincosf(u.x, &sn.x, &cs.x);
    __sincosf(u.y, &sn.y, &cs.y);
    const float2 m = make_float2(v3.x, v3.y);
    if (KIND == RSI_STAGE_PISTON) {
        const float2 amp = __fmul2_rn(m, ir);
        a1 = __ffma2_rn(amp, cs, a1);
        b1 = __ffma2_rn(amp, sn, b1);
    } else {
        const float2 g = __fmul2_rn(m, __fmul2_rn(ir, ir)), gr = __fmul2_rn(g, ir);
        a1 = __ffma2_rn(gr, cs, a1);
        a2 = __ffma2_rn(g, sn, a2);
        b1 = __ffma2_rn(gr, sn, b1);
        b2 = __ffma2_rn(g, cs, b2);
    }
}

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

struct Sum {
    const uint8_t* tiles;
    uint32_t tile_bytes;
    int S, rec_f, n_tiles;
    const Node* nodes[kLevels];
    const Box* boxes;  // 5 per block: the block and its quarters
    int top;           // coarsest level of source clusters
    TgtView tgt;
    int64_t n_tgt;
    float kh, kl, kph, kpl;  // k and k / pi
    TwoPiSplit tp;
    int* status;
};

// e^{i pi r} for r = hi + lo half turns: whole turns leave hi exactly, and lo is
// a rotation of its own.  Once per target or cluster, where the error stays
// common to a cluster's sources.
__device__ __forceinline__ void exact_phase(float hi, float lo, float& c, float& s) {
    const float x = __fmaf_rn(-2.0f, rintf(0.5f * hi), hi);
    const float r = 3.14159274f * lo;
    float sx, cx;
    sincospif(x, &sx, &cx);
    c = __fmaf_rn(-sx, r, cx);
    s = __fmaf_rn(cx, r, sx);
}

// A target by its offset from the block's centre along the block's axes
// (double-floats) and the offset's square
struct TargetPos {
    float q1h, q1l, q2h, q2l, sh, sl;
};

// e^{ik |D + q|} (kh + kl = k / pi), |D + q| formed as target_reference forms its distance
__device__ __forceinline__ void target_phase(const WarpArea& w, const TargetPos& t, float kh, float kl,
                                             float& c, float& sn) {
    // |D + q|^2 = |D|^2 + |q|^2 + 2 D.q as a double-float
    float p1, e1, p2, e2, s, se, a, ae, S, Se;
    two_prod(w.D1h, t.q1h, p1, e1);
    two_prod(w.D2h, t.q2h, p2, e2);
    e1 = __fmaf_rn(w.D1h, t.q1l, __fmaf_rn(w.D1l, t.q1h, e1));
    e2 = __fmaf_rn(w.D2h, t.q2l, __fmaf_rn(w.D2l, t.q2h, e2));
    two_sum(p1, p2, s, se);
    se = __fadd_rn(se, __fadd_rn(e1, e2));
    two_sum(w.S0h, t.sh, a, ae);
    ae = __fadd_rn(ae, __fadd_rn(w.S0l, t.sl));
    two_sum(a, 2.0f * s, S, Se);
    Se = __fadd_rn(Se, __fmaf_rn(2.0f, se, ae));
    // one Newton step from the FP32 reciprocal square root
    const float y = rsqrt_approx(S), r0 = __fmul_rn(S, y);
    float Rh, Rl;
    const float e = __fadd_rn(__fmaf_rn(-r0, r0, S), Se);
    fast_two_sum(r0, __fmul_rn(e, __fmul_rn(0.5f, y)), Rh, Rl);
    float ph, pl;
    two_prod(kh, Rh, ph, pl);
    pl = __fmaf_rn(kh, Rl, __fmaf_rn(kl, Rh, pl));
    exact_phase(ph, pl, c, sn);
}

// Groups of the target nodes' loop over the source nodes: with N = 6 the 36
// nodes would fill a warp once and an eighth
template <int N>
constexpr int node_groups() {
    return N == 6 ? 2 : 1;
}

// U_0 .. U_{N-1} of two points, pair-interleaved
template <int N>
__device__ __forceinline__ void cheb_row(float2 x, float* row) {
    const float2 p = __fadd2_rn(x, x), m = __fmul2_rn(x, dup(-2.0f));
    float2 u0 = dup(1.0f), u1 = x;
#pragma unroll
    for (int q = 0; q < N; q += 2) {
        *reinterpret_cast<float4*>(row + 2 * q) = make_float4(u0.x, u0.y, u1.x, u1.y);
        u0 = __ffma2_rn(m, u1, u0);  // U_{q+2}, q even: s_{q+1} s_{q+2} = -1
        u1 = __ffma2_rn(p, u0, u1);
    }
}

// One warp: moments of a source cluster for a target cluster, the field at the
// target nodes and its Chebyshev coefficients (w.fh), the phase of the target
// (e^{ik |Q_j - c|}, c the source cluster's centre) left out.
template <class M, int N>
__device__ __forceinline__ void warp_item(const M& model, const Sum& g, const Box& b, const Box& b0, int t0, int nt,
                                          WarpArea& w, const float* tab) {
    constexpr int NN = N * N, STR = 4 * N + 4;  // row stride: 16-byte groups without bank conflicts
    static_assert(32 * STR <= kRowFloats && NN * 8 <= kRowFloats, "warp area");
    constexpr int G = 32 / N;  // source groups of the product
    static_assert(G * N * 2 * N * 4 <= int(sizeof(float2)) * 3 * kMaxNN, "partial moments");
    const int lane = threadIdx.x & 31;
    const float* C = tab + tab_off(N);
    const Node& s = w.node;
    // references of the target cluster's centre: lanes 0 .. 15 the tiles, 16 the cluster
    typename M::Ref ref;
    float gx = 0.f, gy = 0.f, gz = 0.f;  // tile centre - cluster centre
    {
        const float* hc = lane < 16 ? reinterpret_cast<const float*>(g.tiles + size_t(t0 + min(lane, nt - 1)) * g.tile_bytes)
                                    : s.c;
        float c[6];
#pragma unroll
        for (int q = 0; q < 6; ++q) c[q] = hc[q];
        ref = model.reference(b.c, c);
        float lo;
        df_diff(c[0], c[1], s.c[0], s.c[1], gx, lo);
        df_diff(c[2], c[3], s.c[2], s.c[3], gy, lo);
        df_diff(c[4], c[5], s.c[4], s.c[5], gz, lo);
    }
    const float ih1 = s.h1 > 0.0f ? 1.0f / s.h1 : 0.0f, ih2 = s.h2 > 0.0f ? 1.0f / s.h2 : 0.0f;
    const float3 f1 = make_float3(s.e1[0] * ih1, s.e1[1] * ih1, s.e1[2] * ih1);
    const float3 f2 = make_float3(s.e2[0] * ih2, s.e2[1] * ih2, s.e2[2] * ih2);
    const int gl = lane / N, l = lane - gl * N;
    // partial moments of (group, l): [k re..., k im...], summed tile by tile so that no FP32 sum is long
    float* part_m = reinterpret_cast<float*>(w.x) + (gl * N + l) * 2 * N;
    if (gl < G)
#pragma unroll
        for (int q = 0; q < 2 * N; q += 2) *reinterpret_cast<float2*>(part_m + q) = make_float2(0.f, 0.f);
    // -- moments: a lane takes a pair of sources in packed arithmetic, then one
    // column l of the product over every G-th pair
#pragma unroll 1
    for (int t = 0; t < nt; ++t) {
        const typename M::Ref rt = model.broadcast(ref, t);
        const float tx = __shfl_sync(0xffffffffu, gx, t), ty = __shfl_sync(0xffffffffu, gy, t),
                    tz = __shfl_sync(0xffffffffu, gz, t);
        const float o1 = fmaf(tx, f1.x, fmaf(ty, f1.y, tz * f1.z)), o2 = fmaf(tx, f2.x, fmaf(ty, f2.y, tz * f2.z));
        const uint8_t* tile = g.tiles + size_t(t0 + t) * g.tile_bytes + RSI_TILE_HDR_BYTES;
        float2 re[N], im[N];  // even and odd sources
#pragma unroll
        for (int q = 0; q < N; ++q) re[q] = im[q] = make_float2(0.f, 0.f);
#pragma unroll 1
        for (int i0 = 0; i0 < g.S; i0 += 64) {
            const int pi = (i0 >> 1) + lane;
            const float4* r = reinterpret_cast<const float4*>(tile) + min(pi, (g.S >> 1) - 1) * (g.rec_f >> 1);
            const float4 v0 = __ldg(r), v1 = __ldg(r + 1), v2 = __ldg(r + 2);
            const float2 px = make_float2(v0.x, v0.y), py = make_float2(v0.z, v0.w), pzn = make_float2(v1.x, v1.y);
            float2 m = M::kPolar ? make_float2(v2.z, v2.w) : make_float2(v2.x, v2.y);
            if (pi >= (g.S >> 1)) m = make_float2(0.f, 0.f);
            float2 u = model.source_phase(rt, px, py, pzn, make_float2(v1.z, v1.w));  // half turns
            if (M::kPolar) u = __ffma2_rn(make_float2(v2.x, v2.y), dup(0.318309886f), u);
            float2 sn, cs;
            sincospif(u.x, &sn.x, &cs.x);
            sincospif(u.y, &sn.y, &cs.y);
            float2 cr = __fmul2_rn(m, cs), ci = __fmul2_rn(m, sn);
            // padding sits metres away: its phase is meaningless
            if (m.x == 0.0f) cr.x = ci.x = 0.0f;
            if (m.y == 0.0f) cr.y = ci.y = 0.0f;
            float2 xi = __ffma2_rn(px, dup(f1.x), __ffma2_rn(py, dup(f1.y), __ffma2_rn(pzn, dup(-f1.z), dup(o1))));
            float2 et = __ffma2_rn(px, dup(f2.x), __ffma2_rn(py, dup(f2.y), __ffma2_rn(pzn, dup(-f2.z), dup(o2))));
            xi = make_float2(fminf(fmaxf(xi.x, -1.0f), 1.0f), fminf(fmaxf(xi.y, -1.0f), 1.0f));
            et = make_float2(fminf(fmaxf(et.x, -1.0f), 1.0f), fminf(fmaxf(et.y, -1.0f), 1.0f));
            float* row = w.rows + lane * STR;
            cheb_row<N>(xi, row);
            cheb_row<N>(et, row + 2 * N);
            *reinterpret_cast<float4*>(row + 4 * N) = make_float4(cr.x, cr.y, ci.x, ci.y);
            __syncwarp();
            if (gl < G) {
#pragma unroll 1
                for (int i = gl; i < 32; i += G) {
                    const float* q = w.rows + i * STR;
                    const float4 c = *reinterpret_cast<const float4*>(q + 4 * N);
                    const float2 te = *reinterpret_cast<const float2*>(q + 2 * N + 2 * l);
                    const float2 er = __fmul2_rn(te, make_float2(c.x, c.y)), ei = __fmul2_rn(te, make_float2(c.z, c.w));
#pragma unroll
                    for (int j = 0; j < N; j += 2) {
                        const float4 v = *reinterpret_cast<const float4*>(q + 2 * j);
                        re[j] = __ffma2_rn(make_float2(v.x, v.y), er, re[j]);
                        im[j] = __ffma2_rn(make_float2(v.x, v.y), ei, im[j]);
                        re[j + 1] = __ffma2_rn(make_float2(v.z, v.w), er, re[j + 1]);
                        im[j + 1] = __ffma2_rn(make_float2(v.z, v.w), ei, im[j + 1]);
                    }
                }
            }
            __syncwarp();
        }
        if (gl < G)
#pragma unroll
            for (int q = 0; q < N; q += 2) {
                float2* o = reinterpret_cast<float2*>(part_m + q);
                *o = __fadd2_rn(*o, make_float2(re[q].x + re[q].y, re[q + 1].x + re[q + 1].y));
                o = reinterpret_cast<float2*>(part_m + N + q);
                *o = __fadd2_rn(*o, make_float2(im[q].x + im[q].y, im[q + 1].x + im[q + 1].y));
            }
    }
    __syncwarp();
    float2* xs = reinterpret_cast<float2*>(w.rows);
    for (int o = lane; o < NN; o += 32) {  // xs[k][l]
        const int ol = o / N, ok = o - ol * N;
        float xr = 0.0f, xi = 0.0f;
#pragma unroll
        for (int p = 0; p < G; ++p) {
            const float* q = reinterpret_cast<const float*>(w.x) + (p * N + ol) * 2 * N + ok;
            xr += q[0];
            xi += q[N];
        }
        xs[ok * N + ol] = make_float2(xr, xi);
    }
    __syncwarp();
    for (int o = lane; o < NN; o += 32) {  // y[a][l] = sum_k C[a][k] xs[k][l]
        const int a = o / N, ol = o - a * N;
        float2 y = make_float2(0.f, 0.f);
#pragma unroll
        for (int kk = 0; kk < N; ++kk) y = __ffma2_rn(dup(C[a * N + kk]), xs[kk * N + ol], y);
        w.y[o] = y;
    }
    __syncwarp();
    const typename M::Ref rc = model.broadcast(ref, 16);  // the cluster's own reference
    model.prepare_targets(w, b, b0);
    __syncwarp();
    float c0, s0;  // the phase factor from the source cluster's centre to the target cluster's
    model.centre_phase(w, b, b0, rc, c0, s0);
    for (int o = lane; o < NN; o += 32) {  // source node (a, c): moment and record
        const int a = o / N, c = o - a * N;
        float2 m2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < N; ++q) m2 = __ffma2_rn(dup(C[c * N + q]), w.y[a * N + q], m2);
        const float s1 = 0.5f * N * C[a * N + 1] * s.h1, s2 = 0.5f * N * C[c * N + 1] * s.h2;  // C[.][1] = (2/N) x_a
        const float3 p = make_float3(fmaf(s1, s.e1[0], s2 * s.e2[0]), fmaf(s1, s.e1[1], s2 * s.e2[1]),
                                     fmaf(s1, s.e1[2], s2 * s.e2[2]));
        // m e^{i beta} with beta in [-pi/2, pi/2]: a negated moment negates m alone
        // the modulus over a power of two, since the squares of amplitudes in a small or
        // a large unit leave FP32's range where the amplitudes do not
        const int e = min(max((__float_as_int(fmaxf(fabsf(m2.x), fabsf(m2.y))) >> 23), 1), 253);
        const float up = __int_as_float((254 - e) << 23), mx = up * m2.x, my = up * m2.y;
        float m = __int_as_float(e << 23) * sqrtf(fmaf(mx, mx, my * my));
        if (m2.x < 0.0f || (m2.x == 0.0f && m2.y < 0.0f)) m = -m, m2.x = -m2.x, m2.y = -m2.y;
        model.node_record(b, rc, p, m, atan2f(m2.y, m2.x), w.rows + (o >> 1) * 16 + (o & 1));
    }
    __syncwarp();
    // -- node to node
    constexpr int G2 = node_groups<N>(), P2 = NN / 2, PER = (P2 + G2 - 1) / G2;
    float2* part = G2 > 1 ? w.y : w.x;
    static_assert(G2 * NN <= kMaxNN, "partial sums of the target nodes");
#pragma unroll 1
    for (int o2 = lane; o2 < NN * G2; o2 += 32) {
        const int gq = o2 / NN, o = o2 - gq * NN, a = o / N, c = o - a * N;
        const float q1 = 0.5f * N * C[a * N + 1] * b.q1, q2 = 0.5f * N * C[c * N + 1] * b.q2;
        const float2 f = model.node_field(s, b, rc, q1, q2, reinterpret_cast<const float4*>(w.rows), gq * PER,
                                          min(P2, (gq + 1) * PER));
        // the moments and the targets' phases each carry the factor of the centres: one too many
        part[o2] = make_float2(fmaf(c0, f.x, s0 * f.y), fmaf(c0, f.y, -s0 * f.x));
    }
    __syncwarp();
    if (G2 > 1) {
        for (int o = lane; o < NN; o += 32) {
            float2 f = w.y[o];
#pragma unroll
            for (int gq = 1; gq < G2; ++gq) f.x += w.y[gq * NN + o].x, f.y += w.y[gq * NN + o].y;
            w.x[o] = f;
        }
        __syncwarp();
    }
    for (int o = lane; o < NN; o += 32) {  // y[k][c] = sum_a C[a][k] x[a][c]
        const int kk = o / N, c = o - kk * N;
        float2 y = make_float2(0.f, 0.f);
#pragma unroll
        for (int a = 0; a < N; ++a) {
            const float cc = C[a * N + kk];
            y = __ffma2_rn(make_float2(cc, cc), w.x[a * N + c], y);
        }
        w.y[o] = y;
    }
    __syncwarp();
    for (int o = lane; o < NN; o += 32) {
        const int kk = o / N, ol = o - kk * N;
        float2 f = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < N; ++c) {
            const float cc = C[c * N + ol];
            f = __ffma2_rn(make_float2(cc, cc), w.y[kk * N + c], f);
        }
        w.fh[o] = f;
    }
}

// the field of an item at T targets at (u, v) in its box, without their
// phases; the coefficients fall off with the order, so the sums run from the
// highest order down and round once at the field's own size
template <int N, int T>
__device__ __forceinline__ void eval_targets(const float2* fh, const float (&u)[T], const float (&v)[T],
                                             float2 (&f)[T]) {
    float tu[T][N], tv[T][N];
#pragma unroll
    for (int q = 0; q < T; ++q) {
        tu[q][0] = tv[q][0] = 1.0f;
        tu[q][1] = u[q];
        tv[q][1] = v[q];
#pragma unroll
        for (int l = 2; l < N; ++l) {
            tu[q][l] = fmaf(l & 1 ? 2.0f * u[q] : -2.0f * u[q], tu[q][l - 1], tu[q][l - 2]);
            tv[q][l] = fmaf(l & 1 ? 2.0f * v[q] : -2.0f * v[q], tv[q][l - 1], tv[q][l - 2]);
        }
        f[q] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int kk = N - 1; kk >= 0; --kk) {
        float2 s[T];
#pragma unroll
        for (int q = 0; q < T; ++q) s[q] = make_float2(0.f, 0.f);
#pragma unroll
        for (int l = N - 2; l >= 0; l -= 2) {
            const float4 c = *reinterpret_cast<const float4*>(fh + kk * N + l);
#pragma unroll
            for (int q = 0; q < T; ++q) {
                s[q] = __ffma2_rn(make_float2(c.z, c.w), dup(tv[q][l + 1]), s[q]);
                s[q] = __ffma2_rn(make_float2(c.x, c.y), dup(tv[q][l]), s[q]);
            }
        }
#pragma unroll
        for (int q = 0; q < T; ++q) f[q] = __ffma2_rn(s[q], dup(tu[q][kk]), f[q]);
    }
}

__device__ __forceinline__ void add_comp(float4& acc, float ar, float ai) {
    float s, e;
    two_sum(acc.x, ar, s, e);
    acc.x = s;
    acc.y = __fadd_rn(acc.y, e);
    two_sum(acc.z, ai, s, e);
    acc.z = s;
    acc.w = __fadd_rn(acc.w, e);
}

// What a sum's pair terms are: the interface that warp_item and run_block need,
// for the piston and Rayleigh-Sommerfeld stages.  (raytrace.cu has its own.)
template <int KIND, int NORM>
struct StageModel {
    static constexpr bool kPolar = KIND == RSI_STAGE_RSI;  // source amplitudes m e^{i beta}, or real
    static constexpr int kDirectCost = 134;  // instructions per warp of a tile's source onto 256 targets, direct
    using Ref = rsi_fp32::TgtRef;
    const Sum& g;

    __device__ __forceinline__ int choose(const Node& s, const Box& b) const { return choose_nodes(s, b, g.kh); }
    __device__ __forceinline__ static float cost(float ns, float nt, int N) { return pair_cost(ns, nt, N, 36.f, 85.f, 75.f); }
    __device__ __forceinline__ Ref reference(const float* t, const float* c) const {
        return rsi_fp32::target_reference(t[0], t[1], t[2], t[3], t[4], t[5], c, g.kh, g.kl, g.tp);
    }
    __device__ __forceinline__ Ref broadcast(const Ref& r, int lane) const {
        Ref o;
        o.Dx = __shfl_sync(0xffffffffu, r.Dx, lane);
        o.Dy = __shfl_sync(0xffffffffu, r.Dy, lane);
        o.Dz = __shfl_sync(0xffffffffu, r.Dz, lane);
        o.R = __shfl_sync(0xffffffffu, r.R, lane);
        o.tau = 0.318309886f * __shfl_sync(0xffffffffu, r.tau, lane);  // half turns
        o.R2 = o.R * o.R;
        return o;
    }
    // k |d - p| of two sources in half turns, less whole turns
    __device__ __forceinline__ float2 source_phase(const Ref& r, float2 px, float2 py, float2 pzn, float2 pw) const {
        const float2 magic = dup(12582912.0f), nmagic = dup(-12582912.0f);  // 1.5 2^23: rounds to an integer
        const float2 th = __ffma2_rn(dup(-r.Dx), px, __ffma2_rn(dup(-r.Dy), py, __ffma2_rn(dup(r.Dz), pzn, pw)));
        const float2 r2 = __ffma2_rn(th, dup(2.0f), dup(r.R2));
        const float2 ir = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
        const float2 r0 = __fmul2_rn(r2, ir);
        const float2 am = __fadd2_rn(r0, dup(-r.R));
        const float2 a = __ffma2_rn(__ffma2_rn(am, __ffma2_rn(r0, dup(-0.5f), dup(-0.5f * r.R)), th), ir, am);
        const float2 ph = __fmul2_rn(dup(g.kph), a);
        const float2 pl = __ffma2_rn(dup(g.kpl), a, __ffma2_rn(dup(g.kph), a, __fmul2_rn(dup(-g.kph), a)));
        const float2 x = __ffma2_rn(__fadd2_rn(__ffma2_rn(ph, dup(0.5f), magic), nmagic), dup(-2.0f), ph);
        return __fadd2_rn(x, __fadd2_rn(pl, dup(r.tau)));
    }
    // for the targets' phases (one lane): D from the cluster's centre, exactly, to
    // the block's centre along the rectangles' axes, from which run_block counts
    // the targets' offsets, and to the rectangle's own plane across them: where a
    // block spans several planes, a quarter of it may lie in one
    __device__ __forceinline__ void prepare_targets(WarpArea& w, const Box& b, const Box& b0) const {
        if (threadIdx.x & 31) return;
        const Node& s = w.node;
        float dh[3], dl[3], sh[3], sl[3];
        for (int q = 0; q < 3; ++q) {
            const Box& o = q == b.ax1 || q == b.ax2 ? b0 : b;
            df_diff(o.c[2 * q], o.c[2 * q + 1], s.c[2 * q], s.c[2 * q + 1], dh[q], dl[q]);
            df_sqr(dh[q], dl[q], sh[q], sl[q]);
        }
        df_add_pos(sh[0], sl[0], sh[1], sl[1], sh[0], sl[0]);
        df_add_pos(sh[0], sl[0], sh[2], sl[2], w.S0h, w.S0l);
        w.D1h = b.ax1 == 0 ? dh[0] : dh[1], w.D1l = b.ax1 == 0 ? dl[0] : dl[1];
        w.D2h = b.ax2 == 1 ? dh[1] : dh[2], w.D2l = b.ax2 == 1 ? dl[1] : dl[2];
    }
    __device__ __forceinline__ void centre_phase(const WarpArea& w, const Box& b, const Box& b0, const Ref&, float& c,
                                                 float& s) const {
        TargetPos t;
        df_diff(b.c[2 * b.ax1], b.c[2 * b.ax1 + 1], b0.c[2 * b.ax1], b0.c[2 * b.ax1 + 1], t.q1h, t.q1l);
        df_diff(b.c[2 * b.ax2], b.c[2 * b.ax2 + 1], b0.c[2 * b.ax2], b0.c[2 * b.ax2 + 1], t.q2h, t.q2l);
        float a1, e1, a2, e2;
        df_sqr(t.q1h, t.q1l, a1, e1);
        df_sqr(t.q2h, t.q2l, a2, e2);
        df_add_pos(a1, e1, a2, e2, t.sh, t.sl);
        target_phase(w, t, g.kph, g.kpl, c, s);
    }
    __device__ __forceinline__ void target(const WarpArea& w, const TargetPos& t, int, float& c, float& s) const {
        target_phase(w, t, g.kph, g.kpl, c, s);
    }
    // the record of a source node at p (node_pair2), pair-interleaved
    __device__ __forceinline__ void node_record(const Box& b, const Ref& r, const float3& p, float m, float beta,
                                                float* q) const {
        const float t = fmaf(-r.Dx, p.x, fmaf(-r.Dy, p.y, fmaf(-r.Dz, p.z, 0.5f * fmaf(p.x, p.x, fmaf(p.y, p.y, p.z * p.z)))));
        // a = |d - p| - |d| for this t as a sum of two floats: r0 - R is exact, the Newton correction small
        const float r2 = fmaf(2.0f, t, r.R2), ir = rsqrt_approx(r2), r0 = r2 * ir, am = r0 - r.R;
        q[0] = b.ax1 == 0 ? p.x : p.y;
        q[2] = b.ax2 == 1 ? p.y : p.z;
        q[4] = t;
        q[6] = -am;
        q[8] = -(fmaf(am, -0.5f * (r0 + r.R), t) * ir);
        q[10] = beta;
        q[12] = m;
        q[14] = 0.0f;
    }
    // the field of source nodes 2 i0 .. 2 i1 - 1 at the target node (q1, q2) of the box
    __device__ __forceinline__ float2 node_field(const Node& s, const Box& b, const Ref& r, float q1, float q2,
                                                 const float4* pr, int i0, int i1) const {
        const bool x1 = b.ax1 == 0, y2 = b.ax2 == 1;
        const float qx = x1 ? q1 : 0.0f, qy = (x1 ? 0.0f : q1) + (y2 ? q2 : 0.0f), qz = y2 ? 0.0f : q2;
        // |d + q| = R + b as a sum of two floats
        const float h = fmaf(qx, r.Dx, fmaf(qy, r.Dy, fmaf(qz, r.Dz, 0.5f * fmaf(q1, q1, q2 * q2))));
        const float bq = path_diff(h, r.R, r.R2);
        const float Rh = r.R + bq, Rl = bq - (Rh - r.R);
        NodeRef n;
        n.q1 = dup(-q1);
        n.q2 = dup(-q2);
        n.R2 = dup(Rh * Rh);
        n.nR = dup(-Rh);
        n.nRh = dup(-0.5f * Rh);
        n.cr = dup(-__fdividef(Rl, Rh));
        const float2 k2 = dup(g.kh);
        float2 a1 = make_float2(0.f, 0.f), a2 = a1, b1 = a1, b2 = a1;
#pragma unroll 2
        for (int i = i0; i < i1; ++i)
            node_pair2<KIND>(n, pr[4 * i], pr[4 * i + 1], pr[4 * i + 2], pr[4 * i + 3], k2, a1, a2, b1, b2);
        if (KIND == RSI_STAGE_PISTON) return make_float2(a1.x + a1.y, b1.x + b1.y);
        // n . (Q - P) is the same for every source of a flat cluster
        const float nd = fmaf(r.Dx + qx, s.e3[0], fmaf(r.Dy + qy, s.e3[1], (r.Dz + qz) * s.e3[2]));
        return make_float2(nd * fmaf(-g.kh, a2.x + a2.y, -(a1.x + a1.y)), nd * fmaf(g.kh, b2.x + b2.y, -(b1.x + b1.y)));
    }
    // the direct sum of a staged tile at target j
    __device__ __forceinline__ float2 direct(const float* hdr, const float4* rec, int64_t j) const {
        const rsi_fp32::TgtRef ref = rsi_fp32::target_reference(
            __ldg(g.tgt.xh + j), __ldg(g.tgt.xl + j), __ldg(g.tgt.yh + j), __ldg(g.tgt.yl + j), __ldg(g.tgt.zh + j),
            __ldg(g.tgt.zl + j), hdr, g.kh, g.kl, g.tp);
        const bool far_lane = ref.R > 2.0f * hdr[6] && ref.R > 0.0f;
        const rsi_fp32::TgtRef2 r2[1] = {rsi_fp32::packed_reference(ref)};
        float2 a1[1], a2[1], b1[1], b2[1];
        a1[0] = a2[0] = b1[0] = b2[0] = make_float2(0.f, 0.f);
        const float k = g.kh;
        if (__all_sync(0xffffffffu, far_lane))
            rsi_fp32::packed_tile<KIND, NORM, 1, false>(rec, g.S, r2, dup(k), a1, a2, b1, b2);
        else
            rsi_fp32::packed_tile<KIND, NORM, 1, true>(rec, g.S, r2, dup(k), a1, a2, b1, b2);
        if (KIND == RSI_STAGE_PISTON) return make_float2(a1[0].x + a1[0].y, b1[0].x + b1[0].y);
        const float sr = fmaf(-k, a2[0].x + a2[0].y, -(a1[0].x + a1[0].y));
        const float si = fmaf(k, b2[0].x + b2[0].y, -(b1[0].x + b1[0].y));
        float st, ct;
        __sincosf(ref.tau, &st, &ct);
        return make_float2(fmaf(ct, sr, -st * si), fmaf(st, sr, ct * si));
    }
};

__device__ __forceinline__ void init_shared(Shared& sh) {
    for (int e = threadIdx.x; e < kTabFloats; e += kThreads) {
        const int n = e < 36 ? 6 : e < 100 ? 8 : e < 200 ? 10 : 12;
        const int o = e - tab_off(n), a = o / n, kk = o - a * n;
        const float v = (kk ? 2.0f : 1.0f) / float(n) * cospif(float((2 * a + 1) * kk) / float(2 * n));
        sh.tab[e] = kk & 2 ? -v : v;
    }
    __syncthreads();
}

// exclusive position of this thread's `n` entries among the CTA's (n <= 4), and the total
__device__ __forceinline__ int block_scan(int n, Shared& sh, int& total) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int v = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    __syncthreads();
    if (lane == 31) sh.warp_sum[wid] = v;
    __syncthreads();
    int base = 0;
    total = 0;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) {
        base += q < wid ? sh.warp_sum[q] : 0;
        total += sh.warp_sum[q];
    }
    return base + v - n;
}

// One CTA: targets t0 .. t0 + 256 TPT - 1 of the block order against the root
// clusters (16 tiles) r_first, r_first + r_step, ...; acc and slot hold one
// entry per target.  left[tile]: the quarters of the block that the tile's
// direct sum is left for (leftover_block); *any is raised where there are some.
template <class M, int TPT>
__device__ __forceinline__ void run_block(const M& model, const Sum& g, int64_t t0, int r_first, int r_step, int L, int h,
                                          double2* out, uint8_t* left, int* any, Shared& sh, float4* acc, int* slot) {
    const int tid = threadIdx.x, warp = tid >> 5;
    if (tid < int(5 * sizeof(Box) / 4))
        reinterpret_cast<float*>(sh.box)[tid] = __ldg(reinterpret_cast<const float*>(g.boxes + 5 * (t0 / (TPT * kThreads))) + tid);
    __syncthreads();
    const Box& b0 = sh.box[0];
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        slot[q * kThreads + tid] =
            int(strip_slot(min(t0 + int64_t(block_pos<TPT>(q * kThreads + tid, h)), g.n_tgt - 1), g.n_tgt, L, h));
        acc[q * kThreads + tid] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const int n_roots = (g.n_tiles + kRootTiles - 1) / kRootTiles;
    for (int rr = r_first; rr < n_roots; rr += r_step * (kRound / kRootTiles)) {
        // -- the level at which each of up to 256 tiles is taken
        const int root = rr + (tid / kRootTiles) * r_step;
        const int tile = root * kRootTiles + tid % kRootTiles;
        int lev = -1, n = 0, quarters[4] = {0, 0, 0, 0}, emit = 0, mask = 0;
        if (root < n_roots && tile < g.n_tiles) {
            for (int l = g.top; l >= 0 && !n; --l) {
                n = model.choose(g.nodes[l][tile >> (2 * l)], sh.box[0]);
                lev = l;
            }
            if (n) {
                emit = (tile & ((1 << (2 * lev)) - 1)) == 0 ? 1 : 0;
            } else {
                lev = 0;
                for (int q = 0; q < TPT && TPT > 1; ++q) {
                    quarters[q] = model.choose(g.nodes[0][tile], sh.box[1 + q]);
                    if (quarters[q])
                        ++emit;
                    else
                        mask |= 1 << q;
                }
                if (TPT == 1) mask = 1;
            }
        }
        // items by level and N, the largest first, so that a batch's warps have alike work
        __syncthreads();
        int at = 0;
#pragma unroll 1
        for (int cls = 0; cls < 16; ++cls) {
            const int cl = kLevels - 1 - cls / 4, cn = 12 - 2 * (cls & 3);  // cl = -1: a tile and a quarter
            int mine = 0;
            if (cl >= 0)
                mine = emit && n == cn && lev == cl;
            else if (!n && emit)
                for (int q = 0; q < 4; ++q) mine += quarters[q] == cn;
            if (!__syncthreads_or(mine)) continue;
            int total;
            int pos = at + block_scan(mine, sh, total);
            if (cl >= 0) {
                if (mine) sh.items[pos] = make_item(n, 0, lev, tile);
            } else if (mine) {
                for (int q = 0; q < 4; ++q)
                    if (quarters[q] == cn) sh.items[pos++] = make_item(cn, 1 + q, 0, tile);
            }
            at += total;
        }
        if (root < n_roots && tile < g.n_tiles) left[tile] = uint8_t(mask);
        if (mask) *any = 1;
        const int n_items = at;
        __syncthreads();

        // -- batches of one pair of clusters per warp
        for (int i0 = 0; i0 < n_items; i0 += kWarps) {
            WarpArea& w = sh.w[warp];
            const int item = i0 + warp < n_items ? sh.items[i0 + warp] : 0;
            if ((tid & 31) == 0) w.item = item;
            if (item) {
                const int N = item & 15, lev_i = (item >> 7) & 3, t_i = item >> 9;
                const float* src = reinterpret_cast<const float*>(g.nodes[lev_i] + (t_i >> (2 * lev_i)));
                reinterpret_cast<float*>(&w.node)[tid & 31] = __ldg(src + (tid & 31));
                __syncwarp();
                const Box& b = sh.box[(item >> 4) & 7];
                const int nt = min(1 << (2 * lev_i), g.n_tiles - t_i);
                switch (N) {
                    case 6: warp_item<M, 6>(model, g, b, sh.box[0], t_i, nt, w, sh.tab); break;
                    case 8: warp_item<M, 8>(model, g, b, sh.box[0], t_i, nt, w, sh.tab); break;
                    case 10: warp_item<M, 10>(model, g, b, sh.box[0], t_i, nt, w, sh.tab); break;
                    default: warp_item<M, 12>(model, g, b, sh.box[0], t_i, nt, w, sh.tab); break;
                }
            }
            __syncthreads();
            constexpr int T = TPT > 1 ? 2 : 1;  // targets at a time
#pragma unroll 1
            for (int q0 = 0; q0 < TPT; q0 += T) {
                TargetPos tp[T];
                float4 a[T];
#pragma unroll
                for (int q = 0; q < T; ++q) {
                    const int j = slot[(q0 + q) * kThreads + tid];
                    const float *h1 = b0.ax1 == 0 ? g.tgt.xh : g.tgt.yh, *l1 = b0.ax1 == 0 ? g.tgt.xl : g.tgt.yl;
                    const float *h2 = b0.ax2 == 1 ? g.tgt.yh : g.tgt.zh, *l2 = b0.ax2 == 1 ? g.tgt.yl : g.tgt.zl;
                    TargetPos& t = tp[q];
                    df_diff(__ldg(h1 + j), __ldg(l1 + j), b0.c[2 * b0.ax1], b0.c[2 * b0.ax1 + 1], t.q1h, t.q1l);
                    df_diff(__ldg(h2 + j), __ldg(l2 + j), b0.c[2 * b0.ax2], b0.c[2 * b0.ax2 + 1], t.q2h, t.q2l);
                    float a1, e1, a2, e2;
                    df_sqr(t.q1h, t.q1l, a1, e1);
                    df_sqr(t.q2h, t.q2l, a2, e2);
                    df_add_pos(a1, e1, a2, e2, t.sh, t.sl);
                    a[q] = acc[(q0 + q) * kThreads + tid];
                }
#pragma unroll 1
                for (int i = 0; i < kWarps; ++i) {
                    const WarpArea& wi = sh.w[i];
                    const int it = wi.item, bx = (it >> 4) & 7;
                    if (!it || (bx && (bx - 1) / T != q0 / T)) continue;
                    const Box& b = sh.box[bx];
                    float u[T], v[T];
                    float2 f[T];
                    const float i1 = b.q1 > 0.0f ? 1.0f / b.q1 : 0.0f, i2 = b.q2 > 0.0f ? 1.0f / b.q2 : 0.0f;
#pragma unroll
                    for (int q = 0; q < T; ++q) u[q] = fmaf(tp[q].q1h, i1, b.o1), v[q] = fmaf(tp[q].q2h, i2, b.o2);
                    switch (it & 15) {
                        case 6: eval_targets<6, T>(wi.fh, u, v, f); break;
                        case 8: eval_targets<8, T>(wi.fh, u, v, f); break;
                        case 10: eval_targets<10, T>(wi.fh, u, v, f); break;
                        default: eval_targets<12, T>(wi.fh, u, v, f); break;
                    }
#pragma unroll
                    for (int q = 0; q < T; ++q) {
                        if (bx && bx - 1 != q0 + q) continue;
                        float st, ct;
                        model.target(wi, tp[q], slot[(q0 + q) * kThreads + tid], ct, st);
                        add_comp(a[q], fmaf(ct, f[q].x, -st * f[q].y), fmaf(st, f[q].x, ct * f[q].y));
                    }
                }
#pragma unroll
                for (int q = 0; q < T; ++q) acc[(q0 + q) * kThreads + tid] = a[q];
            }
            __syncthreads();
        }

    }
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        const int64_t t = t0 + block_pos<TPT>(q * kThreads + tid, h);
        if (t >= g.n_tgt) continue;
        const float4 a = acc[q * kThreads + tid];
        const double re = double(a.x) + double(a.y), im = double(a.z) + double(a.w);
        out[slot[q * kThreads + tid]] = make_double2(re, im);
    }
}

// ---------------------------------------------------------------------------
// What the clusters leave: a CTA takes the 256 targets of one quarter (t0 in
// the block order) and the tiles seg, seg + segs, ... whose `left` mask has the
// quarter's bit, in the direct kernel's manner (bulk copies kPipe deep, one
// target a thread, 4 CTAs per SM).  A kernel of its own: the leftovers of the
// blocks at the sources are most of the work where there are any, and spread
// over the whole GPU like this they take the direct kernel's time per pair
// (inside the clustered kernel the ray-tracing image took 27.6 ms, 16 blocks
// next to the interface holding up the rest).
// ---------------------------------------------------------------------------
constexpr int kPipe = RSI_PIPE_STAGES;
__host__ __device__ constexpr size_t leftover_smem(size_t tile_bytes) {
    return kPipe * tile_bytes + kPipe * sizeof(uint64_t);
}
template <class M, int TPT>
__device__ __forceinline__ void leftover_block(const M& model, const Sum& g, int64_t block, int quarter, int seg, int segs,
                                               int L, int h, const uint8_t* __restrict__ left, double2* out,
                                               uint8_t* smem) {
    __shared__ int list[kRound];
    __shared__ int warp_sum[kWarps];
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kPipe * g.tile_bytes);
    if (tid == 0) {
        for (int s = 0; s < kPipe; ++s) mbar_init(smem_u32(&bars[s]), 1);
        fence_mbar_init();
    }
    __syncthreads();
    const int64_t t = block * TPT * kThreads + block_pos<TPT>(quarter * kThreads + tid, h);
    const int64_t j = strip_slot(t < g.n_tgt ? t : g.n_tgt - 1, g.n_tgt, L, h);
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    uint32_t uses = 0;
    for (int r0 = 0; seg + r0 * segs < g.n_tiles; r0 += kRound) {
        const int tile = seg + (r0 + tid) * segs;
        const bool mine = tile < g.n_tiles && ((left[tile] >> quarter) & 1);
        const unsigned vote = __ballot_sync(0xffffffffu, mine);
        if (lane == 0) warp_sum[wid] = __popc(vote);
        __syncthreads();
        int at = 0, n = 0;
        for (int q = 0; q < kWarps; ++q) {
            at += q < wid ? warp_sum[q] : 0;
            n += warp_sum[q];
        }
        if (mine) list[at + __popc(vote & ((1u << lane) - 1u))] = tile;
        __syncthreads();
        auto fetch = [&](int i) {
            if (tid == 0 && i < n) {
                const uint32_t u = (uses + i) % kPipe, bar = smem_u32(&bars[u]);
                mbar_expect_tx(bar, g.tile_bytes);
                bulk_g2s(smem_u32(smem + u * g.tile_bytes), g.tiles + size_t(list[i]) * g.tile_bytes, g.tile_bytes, bar);
            }
        };
        for (int s = 0; s < kPipe; ++s) fetch(s);
        for (int i = 0; i < n; ++i) {
            const uint32_t u = uses + i;
            const bool ok = mbar_wait_bounded(smem_u32(&bars[u % kPipe]), (u / kPipe) & 1u);
            if (__syncthreads_or(!ok)) {
                if (tid == 0) {
                    atomicExch(g.status, RSI_DEV_TIMEOUT);
                    for (int e = i; e < n && e < i + kPipe; ++e)
                        mbar_wait_bounded(smem_u32(&bars[(uses + e) % kPipe]), ((uses + e) / kPipe) & 1u);
                }
                return;
            }
            const uint8_t* tl = smem + (u % kPipe) * g.tile_bytes;
            const float2 f = model.direct(reinterpret_cast<const float*>(tl),
                                          reinterpret_cast<const float4*>(tl + RSI_TILE_HDR_BYTES), j);
            add_comp(acc, f.x, f.y);
            __syncthreads();  // every thread is done with this buffer
            fetch(i + kPipe);
        }
        uses += uint32_t(n);
    }
    if (t < g.n_tgt) out[j] = make_double2(double(acc.x) + double(acc.y), double(acc.z) + double(acc.w));
}

// The partial sums of `splits` clustered CTAs and, where the block has
// leftovers, of `segs` leftover CTAs (after them) at the t-th target of the
// block order (Neumaier, in order).
template <int TPT>
__device__ __forceinline__ void sum_block_order(const double2* __restrict__ part, int splits, int segs,
                                                const int* __restrict__ any, int64_t t, int64_t n, int L, int h,
                                                double2* __restrict__ out, int* status) {
    if (t >= (n + TPT * kThreads - 1) / (TPT * kThreads) * (TPT * kThreads)) return;
    const int64_t block = t / (TPT * kThreads);
    const int64_t u = block * TPT * kThreads + block_pos<TPT>(int(t - block * TPT * kThreads), h);
    if (u >= n) return;
    const int64_t j = strip_slot(u, n, L, h);
    sum_partials(part + j, splits + (any[block] ? segs : 0), n, out + j, status);
}

// ---------------------------------------------------------------------------
// preparation
// ---------------------------------------------------------------------------
// Frame and rectangle of sources [i0, i1) (in the order of `mode`) of a set; one CTA.
__device__ __forceinline__ void make_node(int kind, const PointsView& src, int64_t n, int mode, int64_t i0, int64_t i1,
                                          Node* out, float* red) {
    const int64_t first = rsi_fp32::source_slot(i0, n, mode);
    const float xh = src.xh[first], xl = src.xl[first], yh = src.yh[first], yl = src.yl[first], zh = src.zh[first],
                zl = src.zl[first];
    // plane normal: an interface's (+z, its obliquity's own), or the first source's
    float e3x = 0.0f, e3y = 0.0f, e3z = 1.0f;
    if (kind == RSI_STAGE_PISTON) {
        const float nx = float(src.nx[first]), ny = float(src.ny[first]), nz = float(src.nz[first]);
        const float l2 = fmaf(nx, nx, fmaf(ny, ny, nz * nz));
        if (l2 > 0.25f && l2 < 4.0f) {
            const float il = 1.0f / sqrtf(l2);
            e3x = nx * il, e3y = ny * il, e3z = nz * il;
        }
    }
    // e1 = y x e3 (x for a horizontal plane), or x x e3 for a plane facing y
    float e1x, e1y, e1z;
    if (fabsf(e3y) < 0.9f)
        e1x = e3z, e1y = 0.0f, e1z = -e3x;
    else
        e1x = 0.0f, e1y = -e3z, e1z = e3y;
    const float il = 1.0f / sqrtf(fmaf(e1x, e1x, fmaf(e1y, e1y, e1z * e1z)));
    e1x *= il, e1y *= il, e1z *= il;
    const float e2x = e3y * e1z - e3z * e1y, e2y = e3z * e1x - e3x * e1z, e2z = e3x * e1y - e3y * e1x;
    // extents (min, -max) along e1 and e2 turned by 0, 22.5, 45 and 67.5 degrees, and along e3
    const float ca[4] = {1.0f, 0.923879533f, 0.707106781f, 0.382683432f};
    const float sa[4] = {0.0f, 0.382683432f, 0.707106781f, 0.923879533f};
    float ext[4][4], e3e[6] = {INFINITY, INFINITY, 0.f, 0.f, 0.f, 0.f};  // min, -max along e3; -1: not a number
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int d = 0; d < 4; ++d) ext[r][d] = INFINITY;
    for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
        const int64_t j = rsi_fp32::source_slot(i, n, mode);
        float x, y, z, lo;
        df_diff(src.xh[j], src.xl[j], xh, xl, x, lo);
        df_diff(src.yh[j], src.yl[j], yh, yl, y, lo);
        df_diff(src.zh[j], src.zl[j], zh, zl, z, lo);
        const float s1 = fmaf(x, e1x, fmaf(y, e1y, z * e1z)), s2 = fmaf(x, e2x, fmaf(y, e2y, z * e2z)),
                    s3 = fmaf(x, e3x, fmaf(y, e3y, z * e3z));
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const float a = fmaf(ca[r], s1, sa[r] * s2), b = fmaf(ca[r], s2, -sa[r] * s1);
            ext[r][0] = fminf(ext[r][0], a), ext[r][1] = fminf(ext[r][1], -a);
            ext[r][2] = fminf(ext[r][2], b), ext[r][3] = fminf(ext[r][3], -b);
        }
        e3e[0] = fminf(e3e[0], s3), e3e[1] = fminf(e3e[1], -s3);
        if (!(isfinite(x) && isfinite(y) && isfinite(z))) e3e[2] = -1.0f;  // left to the direct sum
    }
    float v[3][6];
#pragma unroll
    for (int d = 0; d < 16; ++d) v[d / 6][d % 6] = ext[d / 4][d % 4];
    v[2][4] = e3e[0], v[2][5] = e3e[1];
    for (int q = 0; q < 3; ++q) rsi_fp32::block_min6(v[q], red);
    rsi_fp32::block_min6(e3e, red);
    if (threadIdx.x == 0) {
        Node o = {};
        // the turned frame with the smallest rectangle
        int best = 0;
        float area = INFINITY, m1 = 0.f, m2 = 0.f;
        for (int r = 0; r < 4; ++r) {
            const float a0 = v[(4 * r) / 6][(4 * r) % 6], a1 = v[(4 * r + 1) / 6][(4 * r + 1) % 6];
            const float b0 = v[(4 * r + 2) / 6][(4 * r + 2) % 6], b1 = v[(4 * r + 3) / 6][(4 * r + 3) % 6];
            const float ha = 0.5f * (-a1 - a0), hb = 0.5f * (-b1 - b0);
            if (ha * hb < 0.98f * area) {
                area = ha * hb, best = r;
                o.h1 = ha, o.h2 = hb, m1 = 0.5f * (a0 - a1), m2 = 0.5f * (b0 - b1);
            }
        }
        const float m3 = 0.5f * (e3e[0] - e3e[1]);
        o.h3 = 0.5f * (-e3e[1] - e3e[0]);
        o.e1[0] = fmaf(ca[best], e1x, sa[best] * e2x), o.e1[1] = fmaf(ca[best], e1y, sa[best] * e2y),
        o.e1[2] = fmaf(ca[best], e1z, sa[best] * e2z);
        o.e2[0] = fmaf(ca[best], e2x, -sa[best] * e1x), o.e2[1] = fmaf(ca[best], e2y, -sa[best] * e1y),
        o.e2[2] = fmaf(ca[best], e2z, -sa[best] * e1z);
        o.e3[0] = e3x, o.e3[1] = e3y, o.e3[2] = e3z;
        const float c[3] = {fmaf(m1, o.e1[0], fmaf(m2, o.e2[0], m3 * e3x)),
                            fmaf(m1, o.e1[1], fmaf(m2, o.e2[1], m3 * e3y)),
                            fmaf(m1, o.e1[2], fmaf(m2, o.e2[2], m3 * e3z))};
        df_diff(xh, xl, -c[0], 0.0f, o.c[0], o.c[1]);
        df_diff(yh, yl, -c[1], 0.0f, o.c[2], o.c[3]);
        df_diff(zh, zl, -c[2], 0.0f, o.c[4], o.c[5]);
        o.flat = e3e[2] == 0.0f ? 1.0f : 0.0f;
        *out = o;
    }
}

// The order in which a piston's sources are cut into tiles (source_slot): that
// in which four runs of 256 spread over the set have the smaller boxes.  Every
// CTA measures it for itself, which costs less than a launch that does it once.
__device__ __forceinline__ int source_mode(int kind, const PointsView& src, int64_t n, float* red) {
    if (kind != RSI_STAGE_PISTON || n < 4096) return 0;
    const int warp = threadIdx.x >> 5, run = warp >> 1, mode = warp & 1;  // 8 warps: a run in one of the orders each
    // places without a common factor with the cells' sizes
    const int64_t i0 = n / 1024 * ((317 + 631 * run) % 1021) / 256 * 256;
    float e[6] = {INFINITY, INFINITY, INFINITY, INFINITY, INFINITY, INFINITY};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int64_t j = rsi_fp32::source_slot(i0 + q * 32 + (threadIdx.x & 31), n, mode);
        const float x = src.xh[j], y = src.yh[j], z = src.zh[j];
        e[0] = fminf(e[0], x), e[1] = fminf(e[1], y), e[2] = fminf(e[2], z);
        e[3] = fminf(e[3], -x), e[4] = fminf(e[4], -y), e[5] = fminf(e[5], -z);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
        for (int o = 16; o; o >>= 1) e[q] = fminf(e[q], __shfl_xor_sync(0xffffffffu, e[q], o));
    const float x = -e[3] - e[0], y = -e[4] - e[1], z = -e[5] - e[2];
    if ((threadIdx.x & 31) == 0) red[warp] = fmaf(x, x, fmaf(y, y, z * z));
    __syncthreads();
    float size[2] = {0.0f, 0.0f};
    for (int q = 0; q < 8; ++q) size[q & 1] += red[q];
    __syncthreads();
    return size[1] < 0.9f * size[0] ? 1 : 0;
}

// The rectangles of one block of 256 TPT targets and of its quarters; one CTA of 256 threads.
template <int TPT>
__device__ __forceinline__ void make_boxes(const TgtView& tgt, int64_t n_tgt, int64_t t0, int L, int h, Box* out,
                                           float* red) {
    int64_t j[TPT];
#pragma unroll
    for (int q = 0; q < TPT; ++q)
        j[q] = strip_slot(min(t0 + int64_t(block_pos<TPT>(q * kThreads + int(threadIdx.x), h)), n_tgt - 1), n_tgt, L, h);
    const int64_t jr = strip_slot(t0, n_tgt, L, h);  // all offsets from the block's first target
    const float rh[3] = {tgt.xh[jr], tgt.yh[jr], tgt.zh[jr]}, rl[3] = {tgt.xl[jr], tgt.yl[jr], tgt.zl[jr]};
    float p[TPT][3], lo, ext[6];
    int wrong = 0;  // bit q: a target of quarter q has a coordinate that is not a number
#pragma unroll
    for (int q = 0; q < TPT; ++q) {
        df_diff(tgt.xh[j[q]], tgt.xl[j[q]], rh[0], rl[0], p[q][0], lo);
        df_diff(tgt.yh[j[q]], tgt.yl[j[q]], rh[1], rl[1], p[q][1], lo);
        df_diff(tgt.zh[j[q]], tgt.zl[j[q]], rh[2], rl[2], p[q][2], lo);
        if (!(isfinite(p[q][0]) && isfinite(p[q][1]) && isfinite(p[q][2]))) wrong |= 1 << q;
    }
    int ax3 = 0;
    float whole[6];
    for (int b = 0; b < (TPT > 1 ? 1 + TPT : 1); ++b) {
        // minima pass over NaN, and the clustered sum does not read a target's third
        // coordinate: such a rectangle is left to the direct sum, which reports it
        const bool numbers = !__syncthreads_or(b == 0 ? wrong : wrong & (1 << (b - 1)));
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            float a = INFINITY, c = INFINITY;
#pragma unroll
            for (int q = 0; q < TPT; ++q)
                if (b == 0 || b == 1 + q) a = fminf(a, p[q][d]), c = fminf(c, -p[q][d]);
            ext[d] = a, ext[3 + d] = c;
        }
        rsi_fp32::block_min6(ext, red);
        if (b == 0) {
#pragma unroll
            for (int d = 0; d < 6; ++d) whole[d] = ext[d];
            const float w[3] = {-ext[3] - ext[0], -ext[4] - ext[1], -ext[5] - ext[2]};
            // the thinnest axis of the whole block is every rectangle's normal
            ax3 = (w[2] <= w[0] && w[2] <= w[1]) ? 2 : w[1] <= w[0] ? 1 : 0;
        }
        if (threadIdx.x == 0) {
            Box o = {};
            o.ax1 = ax3 == 0 ? 1 : 0;
            o.ax2 = ax3 == 2 ? 1 : 2;
            float mid[3], half[3], wm[3];
            for (int d = 0; d < 3; ++d) {
                mid[d] = 0.5f * (ext[d] - ext[3 + d]), half[d] = 0.5f * (-ext[3 + d] - ext[d]);
                wm[d] = 0.5f * (whole[d] - whole[3 + d]);
                df_diff(rh[d], rl[d], -mid[d], 0.0f, o.c[2 * d], o.c[2 * d + 1]);
            }
            o.q1 = half[o.ax1], o.q2 = half[o.ax2], o.q3 = numbers ? half[ax3] : INFINITY;
            o.o1 = o.q1 > 0.0f ? (wm[o.ax1] - mid[o.ax1]) / o.q1 : 0.0f;
            o.o2 = o.q2 > 0.0f ? (wm[o.ax2] - mid[o.ax2]) / o.q2 : 0.0f;
            out[b] = o;
        }
    }
}

// Rows of the target set: L = the first slot at which x and y return to slot
// 0's, and the strip height h that makes a block of `per` targets about as wide
// as high; L = 0 where there are no such rows.  Every thread of the CTA.
__device__ __forceinline__ void find_rows(const TgtView& tgt, int64_t n, int per, int& L, int& h) {
    __shared__ int first;
    if (threadIdx.x == 0) first = 0x7fffffff;
    __syncthreads();
    const float x0 = tgt.xh[0], y0 = tgt.yh[0], z0 = tgt.zh[0], x0l = tgt.xl[0], y0l = tgt.yl[0];
    const int lim = int(n < 65536 ? n : 65536);
    // rows start with three points evenly spaced on a line; QMC points do not
    const float ax = tgt.xh[1] - x0, ay = tgt.yh[1] - y0, az = tgt.zh[1] - z0;
    const float bx = tgt.xh[2] - tgt.xh[1], by = tgt.yh[2] - tgt.yh[1], bz = tgt.zh[2] - tgt.zh[1];
    const float step = fabsf(ax) + fabsf(ay) + fabsf(az);
    const bool line = fabsf(bx - ax) + fabsf(by - ay) + fabsf(bz - az) <= 1e-2f * step;
    for (int j = line ? 3 + int(threadIdx.x) : lim; j < lim && j < *static_cast<volatile int*>(&first); j += blockDim.x)
        if (tgt.xh[j] == x0 && tgt.xl[j] == x0l && tgt.yh[j] == y0 && tgt.yl[j] == y0l) atomicMin(&first, j);
    __syncthreads();
    L = h = 0;
    if (first < lim && n % first == 0 && n < (int64_t(1) << 31)) {
        const float dz = fabsf(tgt.zh[first] - z0);
        if (step > 0.0f && dz > 0.0f) {
            L = first;
            h = 1;
            while (h < per && 2.0f * float(h) * float(h) * dz < float(per) * step) h <<= 1;
        }
    }
}

// Adds one CTA's share of the cost estimate: a block of targets against up to
// 256 tiles, one a thread.  `weight`: of the clustered kernel's instructions
// beside the direct sum's.
template <class M, int TPT>
__device__ __forceinline__ void estimate(const M& model, const Node* nodes, int n_tiles, int S, int top,
                                         const Box* box, float weight, unsigned cta,
                                         StageGate* gate) {
    const int samples = min(n_tiles, kThreads);
    const Node* lev[kLevels] = {nodes, nodes + n_tiles, nodes + n_tiles + (n_tiles + 3) / 4};
    float cost = 0.0f;
    if (int(threadIdx.x) < samples) {
        const int tile =
            int((int64_t(threadIdx.x) * n_tiles / samples + int64_t(cta) * n_tiles / (16 * samples)) % n_tiles);
        int n = 0, l = top;
        for (; l >= 0; --l)
            if ((n = model.choose(lev[l][tile >> (2 * l)], box[0])) != 0) break;
        if (n) {
            const float units = float(1 << (2 * l));
            cost = weight * M::cost(float(S) * units, float(TPT * kThreads), n) / (units * TPT);
        } else {
            const int m = TPT > 1 ? model.choose(lev[0][tile], box[1 + threadIdx.x % TPT]) : 0;
            cost = m ? weight * M::cost(float(S), float(kThreads), m) : float(M::kDirectCost) * S;
        }
    }
    __shared__ unsigned sum;
    if (threadIdx.x == 0) sum = 0;
    __syncthreads();
    atomicAdd(&sum, unsigned(cost));
    __syncthreads();
    if (threadIdx.x == 0) {
        atomicAdd(&gate->cost, (unsigned long long)sum);
        atomicAdd(&gate->pairs, (unsigned long long)samples);
    }
}

}  // namespace rsi_cluster
