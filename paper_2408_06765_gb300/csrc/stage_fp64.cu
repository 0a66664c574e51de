// stage_fp64.cu -- double-precision source x target kernel (steps a3, a5),
// the path for runs validated at 1e-5 against the FP64 oracle.  Same tiling
// and bulk-copy pipeline as the FP32C kernel; the paper's terms with an FP64
// phase and 48-bit amplitudes (stage_fp64_body.cuh), summed in pairs of floats
// over 32 terms and in doubles with Neumaier compensation over those.
// 2^12 x 2^12 pairs of a piston stage: 2.08 ms with every operation in doubles
// (54 double instructions per pair), 0.40 ms now with 9.7, 0.91 of what the
// pipe's rate allows for them; of an interface stage 2.36 and 0.41 (per-point
// normals, 3 operations more: 2.45 and 0.50).
#include <math.h>

#include "stage_fp64_body.cuh"

namespace {

constexpr int kThreads = 128;

struct Neu {
    double s, c;
};
__device__ __forceinline__ void neu_add(Neu& a, double v) {
    double t = a.s + v;
    if (fabs(a.s) >= fabs(v))
        a.c += (a.s - t) + v;
    else
        a.c += (v - t) + a.s;
    a.s = t;
}

using namespace rsi_fp64;
__device__ const Tab kTab = make_tab();

template <int KIND, int NORM>
__global__ void __launch_bounds__(kThreads)
    stage_fp64_kernel(StageArgs a) {
    __shared__ TabEntry tab[kTabSize];
    extern __shared__ __align__(128) uint8_t smem[];
    const int tid = threadIdx.x;
    const int split = blockIdx.y;
    const int t_begin = split * a.tiles_per_split;
    const int t_end = min(a.n_tiles, t_begin + a.tiles_per_split);
    const int ntile = max(0, t_end - t_begin);
    const uint32_t tile_bytes = uint32_t(a.tile_bytes);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + RSI_PIPE_STAGES * a.tile_bytes);

    const int64_t j_raw = int64_t(blockIdx.x) * kThreads + tid;
    const int64_t j = j_raw < a.n_tgt ? j_raw : a.n_tgt - 1;
    const double qx = a.tgt.x[j], qy = a.tgt.y[j], qz = a.tgt.z[j];
    for (int i = tid; i < kTabSize; i += kThreads) tab[i] = kTab.e[i];
    Wave w = make_wave(a.k);
    if (a.variant == 1) w.span = 0u;  // every term in doubles

    if (tid == 0) {
        for (int s = 0; s < RSI_PIPE_STAGES; ++s) mbar_init(smem_u32(&bars[s]), 1);
        fence_mbar_init();
    }
    __syncthreads();
    if (tid == 0) {
        for (int s = 0; s < RSI_PIPE_STAGES && s < ntile; ++s) {
            uint32_t bar = smem_u32(&bars[s]);
            mbar_expect_tx(bar, tile_bytes);
            bulk_g2s(smem_u32(smem + s * a.tile_bytes), a.tiles + size_t(t_begin + s) * a.tile_bytes, tile_bytes,
                     bar);
        }
    }

    Neu re = {0.0, 0.0}, im = {0.0, 0.0};
    int failed_at = -1;
    for (int it = 0; it < ntile; ++it) {
        const int buf = it % RSI_PIPE_STAGES;
        const uint32_t parity = uint32_t(it / RSI_PIPE_STAGES) & 1u;
        bool ok = mbar_wait_bounded(smem_u32(&bars[buf]), parity);
        if (__syncthreads_or(!ok)) {
            failed_at = it;
            break;
        }
        const double scale = *reinterpret_cast<const double*>(smem + buf * a.tile_bytes);
        const double fast_scale = KIND == RSI_STAGE_PISTON ? scale : scale * w.k;
        const Record* rec = reinterpret_cast<const Record*>(smem + buf * a.tile_bytes + RSI_TILE_HDR_BYTES);
        for (int i0 = 0; i0 < a.S; i0 += 32) {
            DF sr = {0.0f, 0.0f}, si = {0.0f, 0.0f};
#pragma unroll 1
            for (int i = i0; i < i0 + 32; ++i) {
                const Record& r = rec[i];
                const double dx = qx - r.x, dy = qy - r.y, dz = qz - r.z;
                const double r2 = dx * dx + dy * dy + dz * dz;
                const double nd = (KIND == RSI_STAGE_PISTON) ? 0.0
                                  : (NORM == RSI_NORMALS_Z)  ? dz
                                                             : (r.nx * dx + r.ny * dy + r.nz * dz);
                if (in_range(w, r2)) {
                    DF fr, fi;
                    fast_term<KIND>(w, r2, nd, r.a, r.b, tab, fr, fi);
                    sr = df_add(sr, fr);
                    si = df_add(si, fi);
                } else {
                    const double2 v = slow_term<KIND>(w.k, r2, nd, double(r.a.h) + double(r.a.l),
                                                      double(r.b.h) + double(r.b.l));
                    neu_add(re, scale * v.x);
                    neu_add(im, scale * v.y);
                }
            }
            neu_add(re, fast_scale * (double(sr.h) + double(sr.l)));
            neu_add(im, fast_scale * (double(si.h) + double(si.l)));
        }
        __syncthreads();
        if (tid == 0 && it + RSI_PIPE_STAGES < ntile) {
            uint32_t bar = smem_u32(&bars[buf]);
            mbar_expect_tx(bar, tile_bytes);
            bulk_g2s(smem_u32(smem + buf * a.tile_bytes),
                     a.tiles + size_t(t_begin + it + RSI_PIPE_STAGES) * a.tile_bytes, tile_bytes, bar);
        }
    }
    if (failed_at >= 0) {
        if (tid == 0) {
            atomicExch(a.status, RSI_DEV_TIMEOUT);
            for (int it = failed_at; it < ntile && it < failed_at + RSI_PIPE_STAGES; ++it)
                mbar_wait_bounded(smem_u32(&bars[it % RSI_PIPE_STAGES]), uint32_t(it / RSI_PIPE_STAGES) & 1u);
        }
        return;
    }
    if (j_raw < a.n_tgt) {
        double2* out = a.out + (a.splits > 1 ? size_t(split) * size_t(a.n_tgt) : 0);
        double vr = re.s + re.c, vi = im.s + im.c;
        if (!isfinite(vr) || !isfinite(vi)) atomicExch(a.status, RSI_DEV_NONFINITE);
        out[j_raw] = make_double2(vr, vi);
    }
}

// One CTA per tile: its records, with the amplitudes over a power of two near
// the largest, so that they are floats of full precision whatever their unit.
constexpr int kPrepThreads = 128;
__global__ void __launch_bounds__(kPrepThreads)
    prep_fp64_kernel(int kind, int S, int64_t n_src, PointsView src, const double2* __restrict__ sigma,
                     double amp_scale, uint8_t* tiles, size_t tile_bytes) {
    __shared__ int top;
    uint8_t* tile = tiles + size_t(blockIdx.x) * tile_bytes;
    Record* rec = reinterpret_cast<Record*>(tile + RSI_TILE_HDR_BYTES);
    const int64_t first = int64_t(blockIdx.x) * S;
    auto amplitude = [&](int64_t q, double& a, double& b) {
        a = b = 0.0;
        if (q >= n_src) return;
        a = amp_scale * src.w[q];
        if (kind == RSI_STAGE_PISTON) return;
        const double2 sg = sigma[q];
        b = a * sg.y;
        a *= sg.x;
    };
    if (threadIdx.x == 0) top = 0;
    __syncthreads();
    int largest = 0;
    for (int i = threadIdx.x; i < S; i += kPrepThreads) {
        double a, b;
        amplitude(first + i, a, b);
        largest = max(largest, max(__double2hiint(a) & 0x7fffffff, __double2hiint(b) & 0x7fffffff));
    }
    atomicMax(&top, largest);
    __syncthreads();
    // 2^e for 2^e <= largest < 2^(e+1); 1 where there is none or it is not finite
    const int e = top >> 20;
    const bool usable = e > 0 && e < 0x7ff;
    const double scale = usable ? __hiloint2double(e << 20, 0) : 1.0;
    if (threadIdx.x == 0) {
        double* hdr = reinterpret_cast<double*>(tile);
        hdr[0] = scale;
        hdr[1] = hdr[2] = hdr[3] = 0.0;
    }
    // 2^-e would overflow for the smallest e: in two factors
    const int e1 = usable ? (1023 - e) / 2 : 0, e2 = usable ? 1023 - e - e1 : 0;
    const double f1 = __hiloint2double((1023 + e1) << 20, 0), f2 = __hiloint2double((1023 + e2) << 20, 0);
    auto pair = [&](double v) {
        v = v * f1 * f2;
        const float h = float(v);
        return DF{h, isfinite(h) ? float(v - double(h)) : 0.0f};
    };
    for (int i = threadIdx.x; i < S; i += kPrepThreads) {
        const int64_t q = first + i;
        Record r;
        double a, b;
        amplitude(q, a, b);
        r.a = pair(a);
        r.b = pair(b);
        const bool real = q < n_src;
        r.x = real ? src.x[q] : 4.0;
        r.y = real ? src.y[q] : 4.0;
        r.z = real ? src.z[q] : 4.0;
        r.nx = real ? src.nx[q] : 0.0;
        r.ny = real ? src.ny[q] : 0.0;
        r.nz = real ? src.nz[q] : 1.0;
        rec[i] = r;
    }
}

template <int KIND, int NORM>
int launch_t(const StageArgs& a, cudaStream_t s) {
    size_t smem = RSI_PIPE_STAGES * a.tile_bytes + RSI_PIPE_STAGES * sizeof(uint64_t);
    static RsiCtxOnce attr_set;
    if (attr_set.needed()) {
        RSI_CUDA_TRY(cudaFuncSetAttribute(stage_fp64_kernel<KIND, NORM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          200 * 1024),
                     "cudaFuncSetAttribute(stage_fp64)");
        attr_set.done();
    }
    dim3 grid(unsigned((a.n_tgt + kThreads - 1) / kThreads), unsigned(a.splits));
    stage_fp64_kernel<KIND, NORM><<<grid, kThreads, smem, s>>>(a);
    RSI_CHECK_LAUNCH("stage_fp64_kernel");
    return RSI_OK;
}

template <int KIND, int NORM>
int occupancy_t(const StageArgs& a) {
    size_t smem = RSI_PIPE_STAGES * a.tile_bytes + RSI_PIPE_STAGES * sizeof(uint64_t);
    int blocks = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, stage_fp64_kernel<KIND, NORM>, kThreads, smem) !=
        cudaSuccess)
        return 1;
    return blocks > 0 ? blocks : 1;
}

int dispatch(const StageArgs& a, cudaStream_t s, bool occ) {
    if (a.kind == RSI_STAGE_PISTON)
        return occ ? occupancy_t<RSI_STAGE_PISTON, RSI_NORMALS_Z>(a) : launch_t<RSI_STAGE_PISTON, RSI_NORMALS_Z>(a, s);
    if (a.normals == RSI_NORMALS_POINTS)
        return occ ? occupancy_t<RSI_STAGE_RSI, RSI_NORMALS_POINTS>(a)
                   : launch_t<RSI_STAGE_RSI, RSI_NORMALS_POINTS>(a, s);
    return occ ? occupancy_t<RSI_STAGE_RSI, RSI_NORMALS_Z>(a) : launch_t<RSI_STAGE_RSI, RSI_NORMALS_Z>(a, s);
}

}  // namespace

size_t fp64_record_bytes() { return sizeof(Record); }
int fp64_threads() { return kThreads; }

int launch_prep_fp64(const rsi_stage& st, const PointsView& src, int64_t n_src, const double2* sigma, int S,
                     uint8_t* tiles, size_t tile_bytes, int n_tiles, cudaStream_t s) {
    const double amp_scale = stage_amp_scale(st);
    prep_fp64_kernel<<<unsigned(n_tiles), kPrepThreads, 0, s>>>(st.kind, S, n_src, src, sigma, amp_scale, tiles,
                                                                tile_bytes);
    RSI_CHECK_LAUNCH("prep_fp64_kernel");
    return RSI_OK;
}

int launch_stage_fp64(const StageArgs& a, cudaStream_t s) { return dispatch(a, s, false); }
int stage_occupancy_fp64(const StageArgs& a) { return dispatch(a, nullptr, true); }
