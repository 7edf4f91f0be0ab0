// The three steps as separate calls: dat_quantize (Algorithm A1 Step 7), dat_aggregate /
// dat_average (Step 9, Eq. grad_agg) and dat_lalr_step (Step 12, Eq. 3).  Codes, scales and
// g_hat are materialised in device memory between the calls.
#include <cmath>

#include "dat_internal.cuh"

// ------------------------------------------------------------------------------------------
// S1: quantizer norms.  One fp64 partial sum of squares per (tile, worker); the CTA that finishes a layer's last
// tile adds the layer's partials in a fixed order: nu_{i,l}, nu_l = max_i, S/nu.  Squares of fp32 values are exact
// in fp64, so the result does not depend on the tiling beyond the last bits of an fp64 sum.
// HBM-bound: 122 us for the 818 MB of ResNet-50, M = 8 (139 as two launches and a copy).
// ------------------------------------------------------------------------------------------
#define SUMSQ_KEEP_BYTES (64ll << 20)             // of the last tiles' gradients, that stay in L2
#define SUMSQ_JOBS 8                              // sums (of a tile and a worker) of a CTA, at most (a warp's partials: <= 32)

// The separate calls follow one another on a stream: a kernel that is launched by dat_launch_after may be set up while the one
// before it ends, and waits for that end (dat_after_previous) before it touches memory that a kernel writes.  It lets the next
// one start only then, so a launch never overlaps with more than the launch before it -- whatever that was: after a kernel
// that does not take part it starts when that one has ended.
__device__ __forceinline__ void dat_after_previous()
{
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}
template <class K, class... ARGS>
static cudaError_t dat_launch_after(K kernel, dim3 grid, cudaStream_t s, const ARGS &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(DAT_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    // (recorded into a graph, whose nodes before may be no kernels, a launch waits for them as any other does)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    const bool known = cudaStreamIsCapturing(s, &cap) == cudaSuccess;
    if (!known) (void)cudaGetLastError();
    cfg.numAttrs = (known && cap == cudaStreamCaptureStatusNone) ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

struct NormOut {
    float S_f;
    float *worker_norms, *scales, *qmul;
    float *dq, *scales_out;                       // nu/(S M) and a copy of the norms, if wanted
    float SM_f;
    uint32_t *count, *status;
    bool per_worker;
};

__device__ __forceinline__ void sumsq_finish(int l, int64_t t0, int64_t t1, int h, int M, const double *partials, const NormOut &o)
{
    __shared__ float s_norm[DAT_MAX_WORKERS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i = warp; i < M; i += DAT_THREADS / 32) {
        double acc = 0.0;
        for (int64_t t = t0 + lane; t < t1; t += 32) acc += __ldcg(partials + t * M + i);
        acc = dat_warp_sum(acc);
        if (lane == 0) {
            const float nrm = (float)sqrt(acc);
            s_norm[i] = nrm;
            o.worker_norms[(int64_t)i * h + l] = nrm;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        float nu = s_norm[0];
        bool bad = !isfinite(nu);
        for (int i = 1; i < M; ++i) {
            bad |= !isfinite(s_norm[i]);
            nu = (s_norm[i] > nu) ? s_norm[i] : nu;
        }
        if (o.per_worker) {
            // every worker keeps its own norm (Eq. rand_q as written): index i*h + l
            for (int i = 0; i < M; ++i) {
                o.scales[(int64_t)i * h + l] = s_norm[i];
                o.qmul[(int64_t)i * h + l] = dat_level_factor(s_norm[i], o.S_f, isfinite(s_norm[i]));
                if (o.scales_out) o.scales_out[(int64_t)i * h + l] = s_norm[i];
            }
        } else {
            o.scales[l] = nu;
            o.qmul[l] = dat_level_factor(nu, o.S_f, !bad);
            if (o.dq) o.dq[l] = (nu == 0.0f) ? 0.0f : nu / o.SM_f;
            if (o.scales_out) o.scales_out[l] = nu;
        }
        if (bad) atomicOr(o.status, DAT_STATUS_NONFINITE);
        o.count[l] = 0u;                          // ready for the next call
    }
}

// A tile's groups of eight that lie partly outside the layer: the first (thread 0) and the last (thread 1).  Returns the
// group's first element, or -1.
__device__ __forceinline__ int64_t sumsq_ragged_at(const TileRange &r)
{
    const int64_t first = r.begin, last = (r.end - 1) & ~(int64_t)7;
    if (threadIdx.x == 0) return (first < r.lo || first + 8 > r.hi) ? first : -1;
    return (last > first && last + 8 > r.hi) ? last : -1;
}
__device__ __noinline__ double sumsq_ragged(const float *g, const TileRange &r)
{
    const int64_t e0 = sumsq_ragged_at(r);
    float v[8];
    dat_load4_masked(g, e0, r.lo, r.hi, v);
    dat_load4_masked(g, e0 + 4, r.lo, r.hi, v + 4);
    double acc = 0.0;
#pragma unroll
    for (int j = 0; j < 8; ++j) acc = fma((double)v[j], (double)v[j], acc);
    return acc;
}

// The tile's sums of workers [w0, w1), one per warp and worker, into s_sum.  NW workers' loads in flight per thread.
// INSIDE: the tile lies wholly in the layer.
template <int NW, bool INSIDE>
__device__ __forceinline__ void sumsq_rows(const GradPtrs &gp, const TileRange &r, int w0, int w1, bool keep, double (*s_sum)[DAT_THREADS / 32])
{
    constexpr int ITERS = DAT_TILE / 8 / DAT_THREADS;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // a group at one of the layer's ends that is not whole (threads 0 and 1 look after the two)
    const bool ragged = !INSIDE && threadIdx.x < 2 && sumsq_ragged_at(r) >= 0;
    for (int i = w0; i < w1; i += NW) {           // every load of NW workers is in flight before the first is used
        float v[NW][ITERS][8];
#pragma unroll
        for (int p = 0; p < NW; ++p) {
            const float *__restrict__ g = gp.p[min(i + p, w1 - 1)];
            const bool wide = dat_aligned32(g);
#pragma unroll
            for (int it = 0; it < ITERS; ++it) {
                const int64_t e0 = r.begin + 8 * (int64_t)(it * DAT_THREADS + threadIdx.x);
                if (i + p < w1 && (INSIDE || (e0 >= r.lo && e0 + 8 <= r.hi))) {
                    if (keep) dat_ld8<EV_NORMAL>(g + e0, wide, v[p][it]);
                    else dat_ld8<EV_FIRST>(g + e0, wide, v[p][it]);
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) v[p][it][j] = 0.0f;
                }
            }
        }
#pragma unroll
        for (int p = 0; p < NW; ++p) {
            double acc = 0.0;
#pragma unroll
            for (int it = 0; it < ITERS; ++it)
#pragma unroll
                for (int j = 0; j < 8; ++j) acc = fma((double)v[p][it][j], (double)v[p][it][j], acc);
            if (ragged && i + p < w1) acc += sumsq_ragged(gp.p[i + p], r);
            acc = dat_warp_sum(acc);
            if (lane == 0 && i + p < w1) s_sum[i + p - w0][warp] = acc;
        }
    }
}

// A CTA sums `per_cta` workers of a tile, or of `tiles_per_cta` consecutive ones (TILES).  What it does once, at its end -- barrier, fence, count,
// a chain of three round trips -- takes longer than a tile's loads, so with few workers a CTA per tile keeps too few bytes
// in flight (us for the norms, a tile per CTA / up to eight sums per CTA / the two launches that these were before: 25.6
// million elements, M = 1: 32.8 / 27.0 / 30.7; 100 million, M = 2: 157 / 133 / 146, M = 3: 216 / 203 / 205; 200 million, M = 1:
// 197 / 157 / 141).  Sixteen sums: 163 in the last, 126 instead of 122 for ResNet-50, M = 8.
template <int NW, bool TILES>
__global__ void __launch_bounds__(DAT_THREADS, NW == 1 ? 6 : 4)
k_sumsq(const __grid_constant__ GradPtrs gp, const TileSource tiles, int M, int per_cta, int tiles_per_cta, int64_t n_tiles, int64_t keep_from,
        double *partials, const __grid_constant__ NormOut out)
{
    constexpr int W = DAT_THREADS / 32;
    __shared__ double s_sum[SUMSQ_JOBS][W];
    __shared__ uint32_t s_last;                   // bit k: the layer of the CTA's tile k is complete
    cudaTriggerProgrammaticLaunchCompletion();    // a step's next phase may set itself up; it waits for this one's end
    const int64_t t0 = TILES ? (int64_t)blockIdx.x * tiles_per_cta : (int64_t)blockIdx.x;
    const int nt = TILES ? (int)min((int64_t)tiles_per_cta, n_tiles - t0) : 1;
    const int w0 = blockIdx.y * per_cta, w1 = min(w0 + per_cta, M), nw = w1 - w0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    TileRange r;                                  // of the last tile, behind the loop
#pragma unroll 1
    for (int k = 0; k < nt; ++k) {                // (no barrier in between: the warps run apart and keep loads in flight)
        r = dat_tile_range(tiles, t0 + k);
        const bool keep = t0 + k >= keep_from;    // read again first thing by the call that follows (which walks back)
        if (r.begin >= r.lo && r.begin + DAT_TILE <= r.hi) sumsq_rows<NW, true>(gp, r, w0, w1, keep, s_sum + k * nw);
        else sumsq_rows<NW, false>(gp, r, w0, w1, keep, s_sum + k * nw);
    }
    __syncthreads();
    if (warp == 0) {                              // (at most 32 sums: the partials are warp 0's)
        if (lane < nt * nw) {
            double s = 0.0;
#pragma unroll
            for (int x = 0; x < W; ++x) s += s_sum[lane][x];
            partials[(t0 + lane / nw) * M + w0 + lane % nw] = s;
        }
        __syncwarp();
        if (lane == 0) {
            uint32_t last = 0;
            TileRange x = r;
            dat_fence();
            for (int i = nt - 1;;) {              // from the last tile on; tiles of one layer are counted in together
                const uint32_t n = (uint32_t)min((int64_t)(i + 1), t0 + i - x.first + 1);
                if (atomicAdd(out.count + x.layer, n) == (uint32_t)(dat_layer_tiles(x) * gridDim.y) - n) last |= 1u << i;
                i -= (int)n;
                if (i < 0) break;
                x = dat_tile_range(tiles, t0 + i);
            }
            if (last) dat_fence();
            s_last = last;
        }
    }
    __syncthreads();
    for (uint32_t last = s_last; last; last &= last - 1) {
        const int i = __ffs(last) - 1;
        const TileRange x = i == nt - 1 ? r : dat_tile_range(tiles, t0 + i);
        sumsq_finish(x.layer, x.first, x.first + dat_layer_tiles(x), tiles.h, M, partials, out);
        __syncthreads();
    }
}

static TileSource plan_tiles(const dat_plan_t *plan) { return TileSource{plan->d_tiles, plan->d_offsets, plan->d_tile_base, (int)plan->h}; }

static int sumsq_go(dat_plan_t *plan, const GradPtrs &gp, int M, const NormOut &o, cudaStream_t s)
{
    // several workers in a CTA (fewer arrivals at the layer's counter, a longer stream per CTA) as long as the CTAs
    // still fill the GPU, then several tiles
    int per_cta = 1, tiles_per_cta = 1;
    auto ctas = [&](int workers, int n) { return (plan->n_tiles + n - 1) / n * ((M + workers - 1) / workers); };
    while (per_cta < SUMSQ_JOBS && per_cta < M && ctas(2 * per_cta, 1) >= 8 * plan->sm_count) per_cta *= 2;
    if (per_cta >= M)
        while (2 * tiles_per_cta * per_cta <= SUMSQ_JOBS && ctas(per_cta, 2 * tiles_per_cta) >= 8 * plan->sm_count) tiles_per_cta *= 2;
    dim3 grid((unsigned)((plan->n_tiles + tiles_per_cta - 1) / tiles_per_cta), (unsigned)((M + per_cta - 1) / per_cta));
    const int64_t keep_from = plan->n_tiles - SUMSQ_KEEP_BYTES / (4 * DAT_TILE * M);
#define DAT_SUMSQ(NW, T) k_sumsq<NW, T><<<grid, DAT_THREADS, 0, s>>>(gp, plan_tiles(plan), M, per_cta, tiles_per_cta, plan->n_tiles, keep_from, plan->d_partials, o)
    if (tiles_per_cta > 1) { if (per_cta == 1) DAT_SUMSQ(1, true); else DAT_SUMSQ(2, true); }
    else if (per_cta == 1) DAT_SUMSQ(1, false);
    else DAT_SUMSQ(2, false);
#undef DAT_SUMSQ
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

static int sumsq_launch(dat_plan_t *plan, const GradPtrs &gp, int M, float *scales, bool per_worker, cudaStream_t s, float *norms_out = nullptr)
{
    const NormOut o = {(float)plan->S, norms_out ? norms_out : plan->d_worker_norms, scales, plan->d_qmul, nullptr, nullptr, 1.0f,
                       plan->d_count, plan->d_status, per_worker};
    return sumsq_go(plan, gp, M, o, s);
}

// The norms as the step's phases want them (dat_pipeline.cu): with the layers' nu/(S M).
int dat_norm_phase(dat_plan_t *plan, const GradPtrs &gp, float *scales_out, cudaStream_t s)
{
    const NormOut o = {(float)plan->S, plan->d_worker_norms, plan->scale_mode == DAT_SCALE_PER_WORKER ? plan->d_worker_norms : plan->d_scales, plan->d_qmul,
                       plan->d_dq, scales_out, (float)((uint64_t)plan->S * (uint64_t)plan->M), plan->d_count, plan->d_status,
                       plan->scale_mode == DAT_SCALE_PER_WORKER};
    return sumsq_go(plan, gp, plan->M, o, s);
}

// ------------------------------------------------------------------------------------------
// S2 + S3: stochastic levels and the packed planes.  A warp takes 256 * `groups` consecutive elements of the flat
// vector (they may span layers) of one worker, a lane a group of eight of every 256 -- one Philox block at 16 bits,
// two at 23.  The packed bits are assembled in the warp's own shared memory and written out with 128-bit stores.
// HBM-bound once the arithmetic is short (4 bytes read and (b+1)/8 written per element; see dat_u1_scaled): 187 us for
// ResNet-50, M = 8, b = 8, 5.6 TB/s.  It was 390 us with four elements per thread (each block of eight drawn twice), the
// plain form of the level and no loads in flight while levels are drawn.
// ------------------------------------------------------------------------------------------
#define QUANT_GROUPS 8                           // groups of eight per lane, at most (a multiple of 2)
#define QUANT_CTAS 4                             // resident CTAs per SM (3: 199 us, 5 with spills: 232 us instead of 187)

struct QuantScale {                              // where a layer's S/nu comes from
    const float *qmul;                           // computed before (scales_in == nullptr), or
    const float *scales_in;                      // the caller's norms, from which it is formed here; they are copied to scales
    float *scales;
    int n_scales;
    float S_f;
    uint32_t *status;
    bool pad;                                    // layer 0 only fills the range up to a multiple of 8: norm 1
};
__device__ __forceinline__ float quant_mul(const QuantScale &q, int64_t k)
{
    if (!q.scales_in) return q.qmul[k];              // (no __ldg: written by a kernel that this one may have been started under)
    const float nu = (q.pad && k == 0) ? 1.0f : __ldg(q.scales_in + k);
    return dat_level_factor(nu, q.S_f, isfinite(nu));
}
// The receiver's factor nu/S (one vector, one norm per layer).
__device__ __forceinline__ float quant_back(const QuantScale &q, int64_t k)
{
    const float nu = __ldg((q.scales_in ? q.scales_in : q.scales) + k);
    return (nu == 0.0f) ? 0.0f : nu / q.S_f;
}

struct QuantRange {                              // one vector (or range of one) and where its message goes
    QuantScale qs;
    const int64_t *off;
    const int32_t *flat_layer;
    uint8_t *levels, *signs;
    float *back;                                 // the receiver's value, if it is wanted
    int64_t d, level_bytes, sign_bytes, elem_base;
    int64_t grad_at;                             // element of the gradient buffers where the range starts
    uint32_t stream_base, cta0, ctas;
    int h, n, groups;
    bool per_worker;
};
#define QUANT_RANGES 32                          // ranges of one launch, at most
template <int N>
struct QuantArgs {
    GradPtrs gp;
    PhiloxKeys keys;
    int n_ranges;
    QuantRange r[N];
};

// A group at the vector's end, across layers, or whose layer's scale is outside the range of the scaled form: the
// plain form of Eq. xi, element by element.  Leaves the group's packed levels and signs in shared memory.
template <int BITS, bool RNG16, bool BACK>
__device__ __forceinline__ void quantize_slow8(const GradPtrs &gp, const PhiloxKeys &keys, const QuantRange &a, int worker, int64_t e0, int l0, int nl, uint8_t *s_level, uint8_t *s_sign)
{
    const float *g = gp.p[worker] + a.grad_at;
    const int64_t q0 = a.per_worker ? (int64_t)worker * a.h : 0;
    uint32_t neg = 0;
    int64_t l_hi = 0;
    float t = 0.0f, f = 0.0f;
#pragma unroll 1
    for (int p = 0; p < 2; ++p) {
        float u1[4];
        uint64_t packed = 0;
        dat_u1x4((uint64_t)(e0 + a.elem_base) + 4 * p, a.stream_base + (uint32_t)worker, keys, RNG16, u1);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int64_t e = e0 + 4 * p + j;
            if (e < a.d) {
                if (e >= l_hi) {                  // (also the first element: l_hi = 0)
                    const int l = l0 + dat_find(a.off + l0, nl, e);
                    l_hi = __ldg(a.off + l + 1);
                    t = quant_mul(a.qs, q0 + l);
                    if (BACK) f = quant_back(a.qs, l);
                }
                const float x = g[e];
                const uint32_t lev = dat_level_u1(x, t, (float)(1u << BITS), u1[j]);
                packed |= (uint64_t)lev << (BITS * j);
                neg |= (uint32_t)(x < 0.0f) << (4 * p + j);
                if (BACK) a.back[e] = (float)((x < 0.0f) ? -(int)lev : (int)lev) * f;
            }
        }
        if (BITS == 16) reinterpret_cast<uint64_t *>(s_level)[p] = packed;
        else if (BITS == 8) reinterpret_cast<uint32_t *>(s_level)[p] = (uint32_t)packed;
        else if (BITS == 4) reinterpret_cast<uint16_t *>(s_level)[p] = (uint16_t)packed;
        else if (BITS == 2) s_level[p] = (uint8_t)packed;
        else s_level[0] = (uint8_t)((p ? s_level[0] : 0u) | (uint32_t)packed << (4 * p));
    }
    *s_sign = (uint8_t)neg;
}

// Packed levels and signs of one group from its eight elements (lowest first) and random words, by the scaled form:
// min(y, S + 1) 2^-b is the clamp to S.  (A minimum and no saturation, which would make a NaN 0, that is level -1, and
// take it from the word's other levels: the caller's norms say nothing about single elements.)
// BACK: v becomes the receiver's value, sign * level * f.
template <int BITS, bool RNG16, bool BACK>
__device__ __forceinline__ void quantize8(float v[8], float ts, float f, const uint32_t w[8], uint8_t *s_level, uint8_t *s_sign)
{
    constexpr float TWO_B = (float)(1u << BITS);
    constexpr uint32_t UBITS = (uint32_t)(127 - BITS) << 23;
    constexpr int PER = (BITS == 16) ? 2 : (BITS == 8) ? 4 : 8;        // levels in a 32-bit word (b <= 4: all eight)
    uint32_t word[8 / PER], neg = 0;
#pragma unroll
    for (int a = 8 / PER - 1; a >= 0; --a) {
        uint32_t bias = 0;                        // the float bits carry 0x4B000000 each: a constant modulo 2^32
        word[a] = 0;
#pragma unroll
        for (int j = PER - 1; j >= 0; --j) {
            const float x = v[a * PER + j] + 0.0f;           // -0 becomes +0: its sign bit is 0
            const float ys = fminf(__fmaf_rn(fabsf(x), ts, dat_u1_scaled<RNG16>(w, a * PER + j, UBITS)), 1.0f);
            const float q = __fmaf_rz(ys, TWO_B, 8388607.0f);
            word[a] += __float_as_uint(q) * (1u << (BITS * j));
            if (BACK)                             // (a level of 0 gives +0, whatever the sign)
                v[a * PER + j] = __fmaf_rn(q - 8388608.0f, __uint_as_float((__float_as_uint(x) & 0x80000000u) | 0x3F800000u), 0.0f) * f;
            bias += 0x4B000000u * (1u << (BITS * j));
            neg = __funnelshift_l(__float_as_uint(x), neg, 1);
        }
        word[a] -= bias;
    }
    if (BITS == 16) *reinterpret_cast<uint4 *>(s_level) = make_uint4(word[0], word[1 % (8 / PER)], word[2 % (8 / PER)], word[3 % (8 / PER)]);
    else if (BITS == 8) *reinterpret_cast<uint2 *>(s_level) = make_uint2(word[0], word[1 % (8 / PER)]);
    else if (BITS == 4) *reinterpret_cast<uint32_t *>(s_level) = word[0];
    else if (BITS == 2) *reinterpret_cast<uint16_t *>(s_level) = (uint16_t)word[0];
    else *s_level = (uint8_t)word[0];
    *s_sign = (uint8_t)neg;
}

// A warp's part that is not the plain case of the kernel below: several layers, the vector's end, a 16-byte aligned
// buffer.  (A call, so that what it keeps in registers is its own.)
template <int BITS, bool RNG16, bool BACK, int N>
__device__ __noinline__ void quantize_mixed(const QuantArgs<N> &all, int range, int worker, int64_t e_piece, uint8_t *s_level, uint8_t *s_sign)
{
    const GradPtrs &gp = all.gp;
    const PhiloxKeys &keys = all.keys;
    const QuantRange &a = all.r[range];
    const int lane = threadIdx.x & 31;
    const int64_t piece = e_piece / DAT_FLAT, last = min(e_piece + 256 * a.groups, a.d - 1) / DAT_FLAT;
    const int l0 = __ldg(a.flat_layer + piece), nl = __ldg(a.flat_layer + last + 1) - l0 + 1;   // the layers are among [l0, l0 + nl)
    const int64_t q0 = a.per_worker ? (int64_t)worker * a.h : 0;
    const float *const g = gp.p[worker] + a.grad_at;
    const bool wide = dat_aligned32(g);
    const bool page = dat_one_counter_page<RNG16>((uint64_t)(e_piece + a.elem_base), 256 * a.groups);
    const PhiloxWorker pw = dat_philox_worker((uint32_t)((uint64_t)(e_piece + a.elem_base) >> (RNG16 ? 35 : 34)), a.stream_base + (uint32_t)worker, keys);
    int64_t l_hi = 0;
    int l = l0;
    float t = 0.0f;
#pragma unroll 1
    for (int k = 0; k < a.groups; ++k) {
        const int64_t e0 = e_piece + 8 * lane + 256 * k;
        uint8_t *const my_level = s_level + (lane + 32 * k) * BITS, *const my_sign = s_sign + lane + 32 * k;
        if (e0 < a.d && e0 >= l_hi) {                        // the group's layer
            l = l0 + dat_find(a.off + l0, nl, e0);
            l_hi = __ldg(a.off + l + 1);
            t = quant_mul(a.qs, q0 + l);
        }
        if (page && dat_scaled_factor(t, (float)(1u << BITS)) && e0 + 8 <= l_hi) {
            float x[8];
            uint32_t w[8];
            dat_ld8<EV_FIRST>(g + e0, wide, x);
            dat_group_words<RNG16>(dat_philox_group<RNG16>((uint64_t)(e0 + a.elem_base), keys), pw, keys, w);
            quantize8<BITS, RNG16, BACK>(x, t * (1.0f / (float)(1u << BITS)), BACK ? quant_back(a.qs, l) : 0.0f, w, my_level, my_sign);
            if (BACK) dat_st8<EV_LAST>(a.back + e0, wide, x);
        } else {
            quantize_slow8<BITS, RNG16, BACK>(gp, keys, a, worker, e0, l0, nl, my_level, my_sign);
        }
    }
}

// N > 1: several ranges of the vectors in one launch (a rank's messages to all owners).
template <int BITS, bool RNG16, bool BACK, int N>
__global__ void __launch_bounds__(DAT_THREADS, QUANT_CTAS)
k_quantize(const __grid_constant__ QuantArgs<N> all)
{
    constexpr int MOST = 256 * QUANT_GROUPS;                 // elements of a warp, at most
    __shared__ uint4 s_level[DAT_THREADS / 32][MOST * BITS / 8 / 16];
    __shared__ uint4 s_sign[DAT_THREADS / 32][MOST / 8 / 16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int range = 0;
    if (N > 1)
        while (range + 1 < all.n_ranges && blockIdx.x >= all.r[range + 1].cta0) ++range;
    const QuantRange &a = all.r[range];
    // back from the vector's end, the workers side by side: k_sumsq walked forward, tile by tile over the workers, and
    // what it read last is still in L2
    const unsigned cta = a.ctas - 1u - (blockIdx.x - a.cta0);
    const int worker = (int)(cta % (unsigned)a.n);
    if (a.qs.scales_in) {                                    // copy of the caller's norms, and their check
        for (int64_t k = (int64_t)cta * DAT_THREADS + threadIdx.x; k < a.qs.n_scales; k += (int64_t)a.ctas * DAT_THREADS) {
            const float nu = a.qs.scales_in[k];
            if (a.qs.scales && a.qs.scales != a.qs.scales_in) a.qs.scales[k] = nu;
            if (!isfinite(nu)) atomicOr(a.qs.status, DAT_STATUS_NONFINITE);
        }
    }
    const int64_t part = (int64_t)(cta / (unsigned)a.n) * (DAT_THREADS / 32) + warp, e_piece = part * (256 * a.groups);
    if (e_piece >= a.d) return;
    const float *ahead = all.gp.p[worker] + a.grad_at + e_piece + 8 * lane;
    const bool whole = dat_aligned32(all.gp.p[worker] + a.grad_at) && e_piece + 256 * a.groups <= a.d;
    float v[2][8];
    if (whole) {                                             // two groups per lane are always in flight
        dat_ld8<EV_FIRST>(ahead, true, v[0]);
        dat_ld8<EV_FIRST>(ahead + 256, true, v[1]);
    }
    // (the norms, where k_sumsq runs just before.  The next launch may not start under this one: its CTAs would take the
    // places of the last ones here -- dat_quantize of 20 thousand elements, M = 16: 16.1 us instead of 15.0; dat_quantize,
    // dat_aggregate and dat_lalr_step of 500 thousand, M = 40, b = 8: 73.8 instead of 70.9)
    cudaGridDependencySynchronize();
    const int l0 = __ldg(a.flat_layer + e_piece / DAT_FLAT);
    const float t = quant_mul(a.qs, (a.per_worker ? (int64_t)worker * a.h : 0) + l0);
    if (whole && __ldg(a.off + l0 + 1) >= e_piece + 256 * a.groups && dat_scaled_factor(t, (float)(1u << BITS)) &&
        dat_one_counter_page<RNG16>((uint64_t)(e_piece + a.elem_base), 256 * a.groups)) {
        const float ts = t * (1.0f / (float)(1u << BITS)), f = BACK ? quant_back(a.qs, l0) : 0.0f;
        const PhiloxWorker pw = dat_philox_worker((uint32_t)((uint64_t)(e_piece + a.elem_base) >> (RNG16 ? 35 : 34)), a.stream_base + (uint32_t)worker, all.keys);
        uint32_t counter = (uint32_t)((uint64_t)(e_piece + a.elem_base) >> (RNG16 ? 3 : 2)) + (RNG16 ? 1u : 2u) * lane;
        uint8_t *to_level = reinterpret_cast<uint8_t *>(s_level[warp]) + lane * BITS, *to_sign = reinterpret_cast<uint8_t *>(s_sign[warp]) + lane;
        float *back = BACK ? a.back + e_piece + 8 * lane : nullptr;
        ahead += 512;
#pragma unroll 1
        for (int k = a.groups; k > 0; k -= 2) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
                uint32_t w[8];
                PhiloxGroup<RNG16> pg;
                pg.e[0] = dat_philox_elem(counter, all.keys);
                if (!RNG16) pg.e[RNG16 ? 0 : 1] = dat_philox_elem(counter + 1u, all.keys);
                dat_group_words<RNG16>(pg, pw, all.keys, w);
                quantize8<BITS, RNG16, BACK>(v[p], ts, f, w, to_level + p * 32 * BITS, to_sign + p * 32);
                if (BACK) dat_st8<EV_LAST>(back + 256 * p, true, v[p]);
                if (k > 2) dat_ld8<EV_FIRST>(ahead + 256 * p, true, v[p]);
                counter += RNG16 ? 32u : 64u;
            }
            ahead += 512;
            if (BACK) back += 512;
            to_level += 64 * BITS;
            to_sign += 64;
        }
    } else {
        quantize_mixed<BITS, RNG16, BACK, N>(all, range, worker, e_piece, reinterpret_cast<uint8_t *>(s_level[warp]), reinterpret_cast<uint8_t *>(s_sign[warp]));
    }
    __syncwarp();

    // 128-bit stores of the finished part (planes are padded to 16 bytes, so whole uint4 fit)
    {
        const int64_t bytes = 32 * BITS * a.groups, base = part * bytes, left = a.level_bytes - base;
        const int n16 = (int)((left < bytes ? left : bytes) / 16);
        uint4 *dst = reinterpret_cast<uint4 *>(a.levels + (int64_t)worker * a.level_bytes + base);
        for (int k = lane; k < n16; k += 32) dst[k] = s_level[warp][k];
    }
    {
        const int64_t bytes = 32 * a.groups, base = part * bytes, left = a.sign_bytes - base;
        const int n16 = (int)((left < bytes ? left : bytes) / 16);
        uint4 *dst = reinterpret_cast<uint4 *>(a.signs + (int64_t)worker * a.sign_bytes + base);
        for (int k = lane; k < n16; k += 32) dst[k] = s_sign[warp][k];
    }
}

// Levels of `n` vectors (workers of the plan's streams from `stream_base` on); scales_in as in dat_quantize.  back: the
// one vector's receiver's value overwrites it (Algorithm A1 Step 10).
static int64_t quant_ctas(int64_t d, int groups) { return (d + groups * (int64_t)(8 * DAT_THREADS) - 1) / (groups * (int64_t)(8 * DAT_THREADS)); }

static QuantRange quant_range(const dat_plan_t *plan, int n, uint8_t *levels, uint8_t *signs, float *scales, const float *scales_in, int n_scales,
                              bool per_worker, uint32_t stream_base)
{
    QuantRange a = {};
    a.qs = QuantScale{plan->d_qmul, scales_in, scales, n_scales, (float)plan->S, plan->d_status, false};
    a.off = plan->d_offsets;
    a.flat_layer = plan->d_flat_layer;
    a.levels = levels;
    a.signs = signs;
    a.d = plan->d;
    a.level_bytes = plan->level_bytes;
    a.sign_bytes = plan->sign_bytes;
    a.elem_base = plan->elem_base;
    a.stream_base = stream_base;
    a.h = (int)plan->h;
    a.n = n;
    a.per_worker = per_worker;
    return a;
}

// Sets the ranges' shares of the grid and launches.  after_norms: k_sumsq runs just before; this launch may be set up and
// load its first gradients while that one ends (300 thousand elements, M = 3, b = 4: 18.5 -> 16.5 us, 3 million, M = 2:
// 28.8 -> 26.3, ResNet-50, M = 8: 323 -> 319).  Not dat_requantize, which has a fraction of the CTAs: 22.7 -> 28.8 us for
// 3 million elements.
template <int N>
static int quant_go(dat_plan_t *plan, QuantArgs<N> &a, uint64_t seed, uint64_t step, cudaStream_t s, bool after_norms = false)
{
    a.keys = dat_make_keys(seed, step);
    // long runs per warp (the set-up is paid once) while there are four waves of CTAs; shorter ones for small problems
    int groups = QUANT_GROUPS;
    auto ctas = [&](int g) {
        int64_t c = 0;
        for (int k = 0; k < a.n_ranges; ++k) c += quant_ctas(a.r[k].d, g) * a.r[k].n;
        return c;
    };
    while (groups > 2 && ctas(groups) < 4ll * QUANT_CTAS * plan->sm_count) groups /= 2;
    uint32_t grid = 0;
    for (int k = 0; k < a.n_ranges; ++k) {
        a.r[k].groups = groups;
        a.r[k].cta0 = grid;
        a.r[k].ctas = (uint32_t)(quant_ctas(a.r[k].d, groups) * a.r[k].n);
        grid += a.r[k].ctas;
    }
    const bool back = a.r[0].back != nullptr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(DAT_THREADS);
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = after_norms ? 1 : 0;
#define DAT_Q(B, R, K) DAT_CUDA(plan, cudaLaunchKernelEx(&cfg, k_quantize<B, R, K, N>, a))
#define DAT_QK(B, R) do { if (N == 1 && back) DAT_Q(B, R, N == 1); else DAT_Q(B, R, false); } while (0)
#define DAT_QR(B) do { if (plan->rng_bits == 16) DAT_QK(B, true); else DAT_QK(B, false); } while (0)
    switch (plan->bits) {
    case 1: DAT_QR(1); break;
    case 2: DAT_QR(2); break;
    case 4: DAT_QR(4); break;
    case 8: DAT_QR(8); break;
    default: DAT_QR(16); break;
    }
#undef DAT_QR
#undef DAT_QK
#undef DAT_Q
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

static int quantize_launch(dat_plan_t *plan, const GradPtrs &gp, int n, uint64_t seed, uint64_t step, uint8_t *levels, uint8_t *signs,
                           float *scales, const float *scales_in, int n_scales, bool per_worker, uint32_t stream_base, cudaStream_t s, float *back = nullptr)
{
    QuantArgs<1> a;
    a.gp = gp;
    a.n_ranges = 1;
    a.r[0] = quant_range(plan, n, levels, signs, scales, scales_in, n_scales, per_worker, stream_base);
    a.r[0].back = back;
    return quant_go(plan, a, seed, step, s, !scales_in && !back);
}

// dat_quantize for several ranges of the same vectors: one launch per QUANT_RANGES.  A rank of a sharded step sends each
// owner the codes of that owner's range; as eight calls, ResNet-50 over eight ranks took eight launches of 11.5 us for
// 2 us of traffic each.
extern "C" int dat_quantize_ranges(int num_ranges, dat_plan_t *const *plans, const int64_t *first_layer, const int32_t *padded,
                                   const float *const *grads, uint64_t seed, uint64_t step, const float *norms,
                                   uint8_t *const *levels, uint8_t *const *signs, void *stream)
{
    if (num_ranges < 1 || !plans || !first_layer || !padded || !grads || !norms || !levels || !signs || (step >> 32)) return DAT_ERR_ARG;
    for (int k = 0; k < num_ranges; ++k) {
        const int rc = dat_check_plan(plans[k]);
        if (rc != DAT_OK) return rc;
        const dat_plan_t *p = plans[k], *q = plans[0];
        if (p->bits == 32) return DAT_ERR_BITS;
        if (p->M != q->M || p->bits != q->bits || p->rng_bits != q->rng_bits || p->worker_base != q->worker_base ||
            p->scale_mode != DAT_SCALE_SHARED_MAX || !levels[k] || !signs[k] || first_layer[k] < 0 || (padded[k] && first_layer[k] < 1)) return DAT_ERR_ARG;
        if (!dat_aligned16(levels[k]) || !dat_aligned16(signs[k])) return DAT_ERR_ALIGN;
    }
    QuantArgs<QUANT_RANGES> a;
    int rc = dat_check_grads(plans[0], grads, &a.gp);
    if (rc != DAT_OK) return rc;
    for (int k0 = 0; k0 < num_ranges && rc == DAT_OK; k0 += QUANT_RANGES) {
        a.n_ranges = num_ranges - k0 < QUANT_RANGES ? num_ranges - k0 : QUANT_RANGES;
        for (int j = 0; j < a.n_ranges; ++j) {
            const int k = k0 + j;
            const dat_plan_t *p = plans[k];
            a.r[j] = quant_range(p, p->M, levels[k], signs[k], nullptr, norms + first_layer[k] - (padded[k] ? 1 : 0), (int)p->h, false, p->worker_base);
            a.r[j].qs.pad = padded[k] != 0;
            a.r[j].grad_at = p->elem_base;
        }
        rc = quant_go(plans[k0], a, seed, step, (cudaStream_t)stream);
    }
    return rc;
}

extern "C" int dat_quantize(dat_plan_t *plan, const float *const *grads, uint64_t seed, uint64_t step,
                            uint8_t *levels, uint8_t *signs, float *scales, const float *scales_in,
                            void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (plan->bits == 32) return DAT_ERR_BITS;
    if (!levels || !signs || !scales) return DAT_ERR_ARG;
    if (step >> 32) return DAT_ERR_ARG;
    if (!dat_aligned16(levels) || !dat_aligned16(signs) || !dat_aligned16(scales)) return DAT_ERR_ALIGN;
    if (scales_in && !dat_aligned16(scales_in)) return DAT_ERR_ALIGN;
    GradPtrs gp;
    rc = dat_check_grads(plan, grads, &gp);
    if (rc != DAT_OK) return rc;

    cudaStream_t s = (cudaStream_t)stream;
    const bool per_worker = (plan->scale_mode == DAT_SCALE_PER_WORKER);
    if (!scales_in) {
        rc = sumsq_launch(plan, gp, plan->M, scales, per_worker, s);
        if (rc != DAT_OK) return rc;
    }
    return quantize_launch(plan, gp, plan->M, seed, step, levels, signs, scales, scales_in, (int)(per_worker ? plan->h * plan->M : plan->h),
                           per_worker, plan->worker_base, s);
}

// S1 by itself: the quantizer norm of every (worker, layer), nu_{i,l} = ||g_l^(i)||_2 (Eq. rand_q).
extern "C" int dat_worker_norms(dat_plan_t *plan, const float *const *grads, float *norms_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!norms_out) return DAT_ERR_ARG;
    if (!dat_aligned16(norms_out)) return DAT_ERR_ALIGN;
    GradPtrs gp;
    rc = dat_check_grads(plan, grads, &gp);
    if (rc != DAT_OK) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    return sumsq_launch(plan, gp, plan->M, plan->d_scales, false, s, norms_out);
}

// ------------------------------------------------------------------------------------------
// S4 + S5: unpack, integer sum over workers, one scaling.
// ------------------------------------------------------------------------------------------
template <int BITS>
__device__ __forceinline__ void dat_unpack8(const uint8_t *__restrict__ plane, int64_t e0, uint32_t lev[8])
{
    const uint8_t *p = plane + e0 * BITS / 8;
    if (BITS == 16) {
        const uint4 q = *reinterpret_cast<const uint4 *>(p);
        lev[0] = q.x & 0xFFFF; lev[1] = q.x >> 16; lev[2] = q.y & 0xFFFF; lev[3] = q.y >> 16;
        lev[4] = q.z & 0xFFFF; lev[5] = q.z >> 16; lev[6] = q.w & 0xFFFF; lev[7] = q.w >> 16;
    } else if (BITS == 8) {
        const uint2 q = *reinterpret_cast<const uint2 *>(p);
#pragma unroll
        for (int j = 0; j < 4; ++j) { lev[j] = (q.x >> (8 * j)) & 0xFF; lev[4 + j] = (q.y >> (8 * j)) & 0xFF; }
    } else {
        uint32_t q;
        if (BITS == 4) q = *reinterpret_cast<const uint32_t *>(p);
        else if (BITS == 2) q = *reinterpret_cast<const uint16_t *>(p);
        else q = *p;
#pragma unroll
        for (int j = 0; j < 8; ++j) lev[j] = (q >> (BITS * j)) & ((1u << BITS) - 1u);
    }
}

// Where the M workers' planes are: one buffer with worker i at i * level_bytes (what dat_quantize writes), or
// one pointer per worker -- this GPU's memory or a peer's mapped into the process, read with plain loads:
// the owner of a layer range pulls the other ranks' planes itself instead of waiting for them to be sent.
struct PlanesFlat {
    const uint8_t *levels, *signs;
    int64_t level_bytes, sign_bytes;
    __device__ __forceinline__ const uint8_t *lv(int i) const { return levels + (int64_t)i * level_bytes; }
    __device__ __forceinline__ const uint8_t *sg(int i) const { return signs + (int64_t)i * sign_bytes; }
};
struct PlanesTable {
    const uint8_t *levels[DAT_MAX_WORKERS], *signs[DAT_MAX_WORKERS];
    __device__ __forceinline__ const uint8_t *lv(int i) const { return levels[i]; }
    __device__ __forceinline__ const uint8_t *sg(int i) const { return signs[i]; }
};

// A thread owns 16 consecutive elements and takes four workers at a time: their bytes are transposed, so that one
// four-way dot product (DP4A, two at 16 bits) adds the four workers' signed levels of an element -- per element and
// worker about one issue slot instead of five for unpacking, negating and adding one level at a time, which limited
// this kernel (75 us for 332 MB at M = 8, b = 8; 50 us for 157 MB at M = 16, b = 4).
// The words of one worker: 16 levels, two sign bytes.
template <int BITS> struct AggWords { uint32_t lv[BITS / 2 > 0 ? BITS / 2 : 1]; uint32_t sg; };

template <int BITS, class SRC>
__device__ __forceinline__ AggWords<BITS> agg_load(const SRC &src, int i, int M, int64_t e0, bool tail)
{
    AggWords<BITS> w = {};
    if (i >= M) return w;                        // absent workers add level 0
    const uint8_t *p = src.lv(i) + e0 * BITS / 8;
    const uint8_t *q = src.sg(i) + (e0 >> 3);
    if (BITS == 16) {
        const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(p));
        w.lv[0] = a.x; w.lv[1 % (BITS / 2 + 1)] = a.y; w.lv[2 % (BITS / 2 + 1)] = a.z; w.lv[3 % (BITS / 2 + 1)] = a.w;
        if (!tail) {                             // (the plane's padding ends with the first eight elements)
            const uint4 b = __ldcs(reinterpret_cast<const uint4 *>(p) + 1);
            w.lv[4 % (BITS / 2 + 1)] = b.x; w.lv[5 % (BITS / 2 + 1)] = b.y; w.lv[6 % (BITS / 2 + 1)] = b.z; w.lv[7 % (BITS / 2 + 1)] = b.w;
        }
    } else if (BITS == 8) {                      // planes are padded to 16 bytes: whatever the group holds, its words exist
        const uint4 a = __ldcs(reinterpret_cast<const uint4 *>(p));
        w.lv[0] = a.x; w.lv[1 % (BITS / 2 + 1)] = a.y; w.lv[2 % (BITS / 2 + 1)] = a.z; w.lv[3 % (BITS / 2 + 1)] = a.w;
    } else if (BITS == 4) {
        const uint2 a = __ldcs(reinterpret_cast<const uint2 *>(p));
        w.lv[0] = a.x; w.lv[1 % (BITS / 2 + 1)] = a.y;
    } else if (BITS == 2) {
        w.lv[0] = __ldcs(reinterpret_cast<const uint32_t *>(p));
    } else {
        w.lv[0] = __ldcs(reinterpret_cast<const uint16_t *>(p));
    }
    w.sg = __ldcs(reinterpret_cast<const uint16_t *>(q));
    return w;
}

// out[k] = byte k of the four words, one byte per word: a 4x4 transpose.
__device__ __forceinline__ void agg_transpose(uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t out[4])
{
    const uint32_t ab0 = __byte_perm(a, b, 0x5140), ab1 = __byte_perm(a, b, 0x7362);
    const uint32_t cd0 = __byte_perm(c, d, 0x5140), cd1 = __byte_perm(c, d, 0x7362);
    out[0] = __byte_perm(ab0, cd0, 0x5410);
    out[1] = __byte_perm(ab0, cd0, 0x7632);
    out[2] = __byte_perm(ab1, cd1, 0x5410);
    out[3] = __byte_perm(ab1, cd1, 0x7632);
}

__device__ __forceinline__ int agg_dp4(uint32_t u, uint32_t s, int c)      // c + sum of unsigned bytes times signed bytes
{
    int r;
    asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(u), "r"(s), "r"(c));
    return r;
}
__device__ __forceinline__ int agg_dp2(uint32_t u, uint32_t s, int c)      // c + sum of unsigned halves times the low signed bytes
{
    int r;
    asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(r) : "r"(u), "r"(s), "r"(c));
    return r;
}

template <int BITS>
__device__ __forceinline__ void agg_add4(const AggWords<BITS> w[4], int sum[16])
{
    uint32_t sg[4];
    agg_transpose(w[0].sg, w[1].sg, w[2].sg, w[3].sg, sg);                  // sg[0], sg[1]: the sign bytes of elements 0-7, 8-15
    constexpr int PER = (BITS < 8) ? 8 / BITS : 1;                          // levels in a byte
    constexpr uint32_t MASK = (BITS >= 8) ? 0xFFFFFFFFu : ((1u << BITS) - 1u) * 0x01010101u;
    uint32_t by[4];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
        // the workers' signs as bytes +1 / -1
        const uint32_t s = ((sg[j >> 3] >> (j & 7)) & 0x01010101u) * 0xFEu + 0x01010101u;
        if (BITS == 16) {
            const uint32_t a = __byte_perm(w[0].lv[(j >> 1) % (BITS / 2 + 1)], w[1].lv[(j >> 1) % (BITS / 2 + 1)], (j & 1) ? 0x7632 : 0x5410);
            const uint32_t b = __byte_perm(w[2].lv[(j >> 1) % (BITS / 2 + 1)], w[3].lv[(j >> 1) % (BITS / 2 + 1)], (j & 1) ? 0x7632 : 0x5410);
            sum[j] = agg_dp2(b, s >> 16, agg_dp2(a, s, sum[j]));
        } else {
            const int byte = j / PER;                                       // of the worker's 2 * BITS level bytes
            if (byte % 4 == 0 && j % PER == 0) agg_transpose(w[0].lv[byte / 4], w[1].lv[byte / 4], w[2].lv[byte / 4], w[3].lv[byte / 4], by);
            sum[j] = agg_dp4((by[byte % 4] >> (BITS * (j % PER) % 8)) & MASK, s, sum[j]);
        }
    }
}

template <int BITS, class SRC>
__global__ void __launch_bounds__(DAT_THREADS, 4)
k_aggregate(const __grid_constant__ SRC src, int M, const int64_t *__restrict__ off, const int32_t *__restrict__ flat_layer, int64_t d,
            const float *scales, float SM_f, bool wide, int32_t *__restrict__ code_sum, float *__restrict__ g_hat)
{
    dat_after_previous();
    const int64_t e0 = 16 * ((int64_t)blockIdx.x * DAT_THREADS + threadIdx.x);
    if (e0 >= d) return;
    const bool tail = BITS == 16 && e0 + 8 >= d;
    int sum[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) sum[j] = 0;
#pragma unroll 1
    for (int i = 0; i < M; i += 4) {
        AggWords<BITS> w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = agg_load<BITS>(src, i + k, M, e0, tail);
        agg_add4<BITS>(w, sum);
    }
    const int64_t piece = e0 / DAT_FLAT;
    const int l0 = __ldg(flat_layer + piece), nl = __ldg(flat_layer + piece + 1) - l0 + 1;
    int l = l0 + ((nl > 1) ? dat_find(off + l0, nl, e0) : 0);
    int64_t l_hi = __ldg(off + l + 1);
    float nu = scales[l], f = (nu == 0.0f) ? 0.0f : nu / SM_f;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
        const int64_t e = e0 + 8 * p;
        if (e >= d) break;
        float out[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            while (e + j >= l_hi && e + j < d) {
                ++l;
                l_hi = __ldg(off + l + 1);
                nu = scales[l];
                f = (nu == 0.0f) ? 0.0f : nu / SM_f;
            }
            out[j] = (float)sum[8 * p + j] * f;
        }
        if (e + 8 <= d) {
            dat_st8<EV_LAST>(g_hat + e, wide, out);          // the update that follows reads it
            if (code_sum) {
                reinterpret_cast<int4 *>(code_sum + e)[0] = make_int4(sum[8 * p], sum[8 * p + 1], sum[8 * p + 2], sum[8 * p + 3]);
                reinterpret_cast<int4 *>(code_sum + e)[1] = make_int4(sum[8 * p + 4], sum[8 * p + 5], sum[8 * p + 6], sum[8 * p + 7]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (e + j < d) {
                    g_hat[e + j] = out[j];
                    if (code_sum) code_sum[e + j] = sum[8 * p + j];
                }
        }
    }
}

// The same with one norm per worker (Eq. grad_agg as written): no integer sum exists;
// g_hat = (sum_i nu_{i,l} * signed level_i) / (S*M), accumulated in fp32 with one fused
// multiply-add per worker, in ascending worker order.  The norms are read by plain loads: not by __ldg, for a kernel that this
// one may have been started under writes them, and not past L1 (500 thousand elements, M = 40, b = 8: 60 us; 13 with plain loads
// of one norm per worker, four workers at a time, where a warp lies in one layer).  Six CTAs per SM: with few workers a thread
// has little in flight (60 million elements, b = 4, M = 1: 185 us with four, 163 with five, 148; M = 16: 419, 415, 418).
template <int BITS, class SRC>
__global__ void __launch_bounds__(DAT_THREADS, 6)
k_aggregate_per_worker(const __grid_constant__ SRC src, int M, const int64_t *__restrict__ off, const int32_t *__restrict__ flat_layer, int h,
                       int64_t d, const float *scales, float SM_f, float *__restrict__ g_hat)
{
    dat_after_previous();
    const int64_t e0 = 8 * ((int64_t)blockIdx.x * DAT_THREADS + threadIdx.x);
    const unsigned live = __ballot_sync(0xFFFFFFFFu, e0 < d);
    if (e0 >= d) return;
    int lidx[8];
    {
        const int64_t piece = e0 / DAT_FLAT;
        const int l0 = __ldg(flat_layer + piece), nl = __ldg(flat_layer + piece + 1) - l0 + 1;
        int l = l0 + ((nl > 1) ? dat_find(off + l0, nl, e0) : 0);
        int64_t l_hi = __ldg(off + l + 1);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            while (e0 + j >= l_hi && l + 1 < h) {
                ++l;
                l_hi = __ldg(off + l + 1);
            }
            lidx[j] = l;
        }
    }
    float acc[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.0f;
    auto add = [&](int i, auto &&nu) {
        uint32_t lev[8];
        dat_unpack8<BITS>(src.lv(i), e0, lev);
        const uint32_t sg = src.sg(i)[e0 >> 3];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            // (float)level without the conversion unit: 2^23 + level is exact, the sign bit goes on afterwards
            const float mag = __uint_as_float(0x4B000000u | lev[j]) - 8388608.0f;
            const float code = __uint_as_float(__float_as_uint(mag) | (((sg >> j) & 1u) << 31));
            acc[j] = __fmaf_rn(nu(j), code, acc[j]);
        }
    };
    // (one way for the whole warp: as two ways, a warp at a layer's end goes through the workers twice)
    if (!__any_sync(live, lidx[0] != lidx[7])) {
#pragma unroll 4
        for (int i = 0; i < M; ++i) {
            const float nu = scales[(int64_t)i * h + lidx[0]];
            add(i, [&](int) { return nu; });
        }
    } else {
#pragma unroll 1
        for (int i = 0; i < M; ++i) {
            float nu[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) nu[j] = scales[(int64_t)i * h + lidx[j]];
            add(i, [&](int j) { return nu[j]; });
        }
    }
    float out[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) out[j] = acc[j] / SM_f;
    if (e0 + 8 <= d) {
        reinterpret_cast<float4 *>(g_hat + e0)[0] = make_float4(out[0], out[1], out[2], out[3]);
        reinterpret_cast<float4 *>(g_hat + e0)[1] = make_float4(out[4], out[5], out[6], out[7]);
    } else {
        for (int j = 0; j < 8 && e0 + j < d; ++j) g_hat[e0 + j] = out[j];
    }
}

// ------------------------------------------------------------------------------------------
// Algorithm A1 Step 10 (two-sided quantisation): g_hat <- Q(g_hat) at the server.  The kernels of Step 7 on ONE
// vector: norm per layer, levels on the random stream of index M (the first one no worker uses), packed message; the
// receiver's value nu_l * sign * level / S is written back by the kernel that draws the level.
// ------------------------------------------------------------------------------------------
extern "C" int dat_requantize(dat_plan_t *plan, float *g_hat, uint64_t seed, uint64_t step,
                              uint8_t *levels, uint8_t *signs, float *scales, const float *scales_in,
                              void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (plan->bits == 32) return DAT_ERR_BITS;
    if (!g_hat || !levels || !signs || !scales) return DAT_ERR_ARG;
    if (step >> 32) return DAT_ERR_ARG;
    if (!dat_aligned16(g_hat) || !dat_aligned16(levels) || !dat_aligned16(signs) || !dat_aligned16(scales) ||
        (scales_in && !dat_aligned16(scales_in)))
        return DAT_ERR_ALIGN;
    GradPtrs gp;
    for (int i = 0; i < DAT_MAX_WORKERS; ++i) gp.p[i] = nullptr;
    gp.p[0] = g_hat;

    cudaStream_t s = (cudaStream_t)stream;
    if (!scales_in) {
        rc = sumsq_launch(plan, gp, 1, scales, false, s);
        if (rc != DAT_OK) return rc;
    }
    return quantize_launch(plan, gp, 1, seed, step, levels, signs, scales, scales_in, (int)plan->h, false,
                           plan->worker_base + (uint32_t)plan->M, s, g_hat);
}

static bool dat_aligned32_host(const void *p) { return ((uintptr_t)p & 31u) == 0; }

template <class SRC>
static int aggregate_launch(dat_plan_t *plan, const SRC &src, const float *scales, int32_t *code_sum, float *g_hat, void *stream)
{
    cudaStream_t s = (cudaStream_t)stream;
    const int h = (int)plan->h;
    const float SM_f = (float)((uint64_t)plan->S * (uint64_t)plan->M);
    const unsigned grid = (unsigned)((plan->d + DAT_THREADS * 8 - 1) / (DAT_THREADS * 8));
    if (plan->scale_mode == DAT_SCALE_PER_WORKER) {
        if (code_sum) return DAT_ERR_ARG;        // differently scaled codes have no integer sum
#define DAT_APW(B)                                                                                                  \
    DAT_CUDA(plan, dat_launch_after(k_aggregate_per_worker<B, SRC>, dim3(grid), s, src, plan->M, (const int64_t *)plan->d_offsets,       \
                                    (const int32_t *)plan->d_flat_layer, h, plan->d, scales, SM_f, g_hat))
        switch (plan->bits) {
        case 1: DAT_APW(1); break;
        case 2: DAT_APW(2); break;
        case 4: DAT_APW(4); break;
        case 8: DAT_APW(8); break;
        default: DAT_APW(16); break;
        }
#undef DAT_APW
        DAT_LAUNCHED(plan);
        return DAT_OK;
    }
    const unsigned grid16 = (unsigned)((plan->d + DAT_THREADS * 16 - 1) / (DAT_THREADS * 16));
#define DAT_A(B)                                                                                                                 \
    DAT_CUDA(plan, dat_launch_after(k_aggregate<B, SRC>, dim3(grid16), s, src, plan->M, (const int64_t *)plan->d_offsets,                 \
                                    (const int32_t *)plan->d_flat_layer, plan->d, scales, SM_f, dat_aligned32_host(g_hat), code_sum, g_hat))
    switch (plan->bits) {
    case 1: DAT_A(1); break;
    case 2: DAT_A(2); break;
    case 4: DAT_A(4); break;
    case 8: DAT_A(8); break;
    default: DAT_A(16); break;
    }
#undef DAT_A
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

extern "C" int dat_aggregate(dat_plan_t *plan, const uint8_t *levels, const uint8_t *signs,
                             const float *scales, int32_t *code_sum, float *g_hat, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (plan->bits == 32) return DAT_ERR_BITS;
    if (!levels || !signs || !scales || !g_hat) return DAT_ERR_ARG;
    if (!dat_aligned16(levels) || !dat_aligned16(signs) || !dat_aligned16(scales) || !dat_aligned16(g_hat) ||
        (code_sum && !dat_aligned16(code_sum)))
        return DAT_ERR_ALIGN;
    return aggregate_launch(plan, PlanesFlat{levels, signs, plan->level_bytes, plan->sign_bytes}, scales, code_sum, g_hat, stream);
}

extern "C" int dat_aggregate_gather(dat_plan_t *plan, const uint8_t *const *level_planes, const uint8_t *const *sign_planes,
                                    const float *scales, int32_t *code_sum, float *g_hat, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (plan->bits == 32) return DAT_ERR_BITS;
    if (!level_planes || !sign_planes || !scales || !g_hat) return DAT_ERR_ARG;
    if (!dat_aligned16(scales) || !dat_aligned16(g_hat) || (code_sum && !dat_aligned16(code_sum))) return DAT_ERR_ALIGN;
    PlanesTable t;
    for (int i = 0; i < DAT_MAX_WORKERS; ++i) { t.levels[i] = nullptr; t.signs[i] = nullptr; }
    for (int i = 0; i < plan->M; ++i) {
        if (!level_planes[i] || !sign_planes[i]) return DAT_ERR_ARG;
        if (!dat_aligned16(level_planes[i]) || !dat_aligned16(sign_planes[i])) return DAT_ERR_ALIGN;
        t.levels[i] = level_planes[i];
        t.signs[i] = sign_planes[i];
    }
    return aggregate_launch(plan, t, scales, code_sum, g_hat, stream);
}

// Eq. grad_agg with Q = identity: ordered fp32 sum over workers, then one division by M.
__global__ void __launch_bounds__(DAT_THREADS)
k_average(GradPtrs gp, int M, int64_t d, float *__restrict__ g_hat)
{
    const int64_t e0 = 4 * ((int64_t)blockIdx.x * DAT_THREADS + threadIdx.x);
    if (e0 >= d) return;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    for (int i = 0; i < M; ++i) {
        float v[4];
        dat_load4(gp.p[i], e0, 0, d, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[j] += v[j];
    }
    const float Mf = (float)M;
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[j] = acc[j] / Mf;
    dat_store4(g_hat, e0, 0, d, acc);
}

extern "C" int dat_average(dat_plan_t *plan, const float *const *grads, float *g_hat, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!g_hat) return DAT_ERR_ARG;
    if (!dat_aligned16(g_hat)) return DAT_ERR_ALIGN;
    GradPtrs gp;
    rc = dat_check_grads(plan, grads, &gp);
    if (rc != DAT_OK) return rc;
    const unsigned grid = (unsigned)((plan->d + DAT_THREADS * 4 - 1) / (DAT_THREADS * 4));
    k_average<<<grid, DAT_THREADS, 0, (cudaStream_t)stream>>>(gp, plan->M, plan->d, g_hat);
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

// ------------------------------------------------------------------------------------------
// S6-S8: LALR (Eq. 3), and LAMB (Algorithm A2) with the same update.  Pass 1 (per-layer tiles): m' -- for LAMB m' and
// v', with the direction u = m^/(sqrt(v^) + zeta) + wd*theta formed on the fly -- and the fp64 partial sums of theta^2
// and u^2; the CTA that finishes a layer's last tile forms a_l = lr * tau(||theta_l||)/||u_l||.  Pass 2:
// theta -= a_l * u (LAMB: u once more from the stored moments; the same fp32 operations give the same bits).
// HBM-bound.  Pass 1 walks the tiles back from the last, pass 2 forward from the first: what pass 1 touched last
// (theta and the moments, kept in L2 with evict-last) is what pass 2 reads first.
// ------------------------------------------------------------------------------------------
enum { OPT_MOMENTUM = 0, OPT_LAMB = 1 };
#define UPDATE_CTAS 5                            // resident CTAs per SM (4: 71.6 + 39.4 us, 6: 72.3 + 41.0, 5: 67.8 + 40.2 for ResNet-50)

struct UpdateArgs {
    TileSource tiles;
    float *theta, *mom, *var;
    const float *g_hat;
    LambConst lamb;
    float mu, wd, lr, c_l, c_u;
    bool wide;
    double *partials;
    float *step_a, *norms_out;
    uint32_t *count, *status;
};

template <int EV>
__device__ __forceinline__ void update_ld8(const float *p, bool full, bool wide, int64_t e0, int64_t lo, int64_t hi, float v[8])
{
    if (full) {
        dat_ld8<EV>(p + e0, wide, v);
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = (e0 + j >= lo && e0 + j < hi) ? p[e0 + j] : 0.0f;
    }
}
template <int EV>
__device__ __forceinline__ void update_st8(float *p, bool full, bool wide, int64_t e0, int64_t lo, int64_t hi, const float v[8])
{
    if (full) {
        dat_st8<EV>(p + e0, wide, v);
    } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (e0 + j >= lo && e0 + j < hi) p[e0 + j] = v[j];
    }
}

// Per layer, from the partial sums of its tiles: a_l (every thread of the CTA).
__device__ __forceinline__ void update_finish(const UpdateArgs &a, int l, int64_t t0, int64_t t1, double *scratch)
{
    double x = 0.0, y = 0.0;
    for (int64_t t = t0 + threadIdx.x; t < t1; t += DAT_THREADS) { x += __ldcg(a.partials + 2 * t); y += __ldcg(a.partials + 2 * t + 1); }
    x = dat_block_sum(x, scratch);
    y = dat_block_sum(y, scratch);
    if (threadIdx.x == 0) {
        const float n_theta = (float)sqrt(x), n_u = (float)sqrt(y);
        const float tau = fminf(fmaxf(n_theta, a.c_l), a.c_u);
        const float ratio = (n_u == 0.0f) ? 0.0f : tau / n_u;
        a.step_a[l] = a.lr * ratio;
        if (a.norms_out) { a.norms_out[2 * l] = n_theta; a.norms_out[2 * l + 1] = n_u; }
        if (!isfinite(n_theta) || !isfinite(n_u)) atomicOr(a.status, DAT_STATUS_NONFINITE);
        a.count[l] = 0u;                          // ready for the next call
    }
}

// The tile's two sums (every thread), counted in; the layer's last tile finishes the layer.
__device__ __forceinline__ void update_count_in(const UpdateArgs &a, const TileRange &r, int64_t tile, double ss_theta, double ss_u, double *scratch, bool *s_last)
{
    const double x = dat_block_sum(ss_theta, scratch);
    const double y = dat_block_sum(ss_u, scratch);
    const int64_t T = dat_layer_tiles(r);
    if (threadIdx.x == 0) {
        a.partials[2 * tile] = x;
        a.partials[2 * tile + 1] = y;
        *s_last = dat_count_in(a.count + r.layer, (uint32_t)T);
    }
    __syncthreads();
    if (*s_last) update_finish(a, r.layer, r.first, r.first + T, scratch);
}

template <int OPT>
__global__ void __launch_bounds__(DAT_THREADS, UPDATE_CTAS)
k_update_pass1(const __grid_constant__ UpdateArgs a)
{
    __shared__ double scratch[DAT_THREADS / 32];
    __shared__ bool s_last;
    const int64_t tile = (int64_t)gridDim.x - 1 - blockIdx.x;
    dat_after_previous();
    const TileRange r = dat_tile_range(a.tiles, tile);
    double ss_theta = 0.0, ss_u = 0.0;
#pragma unroll 1
    for (int it = 0; it < DAT_TILE / 8 / DAT_THREADS; ++it) {
        const int64_t e0 = r.begin + 8 * (int64_t)(it * DAT_THREADS + threadIdx.x);
        if (e0 >= r.end) continue;
        const bool full = e0 >= r.lo && e0 + 8 <= r.hi;
        float th[8], m[8], g[8];
        update_ld8<EV_LAST>(a.theta, full, a.wide, e0, r.lo, r.hi, th);
        update_ld8<EV_FIRST>(a.mom, full, a.wide, e0, r.lo, r.hi, m);
        update_ld8<EV_FIRST>(a.g_hat, full, a.wide, e0, r.lo, r.hi, g);
        if (OPT == OPT_LAMB) {
            float v[8];
            update_ld8<EV_FIRST>(a.var, full, a.wide, e0, r.lo, r.hi, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                m[j] = __fmaf_rn(a.lamb.beta1, m[j], __fmul_rn(a.lamb.om1, g[j]));
                v[j] = __fmaf_rn(a.lamb.beta2, v[j], __fmul_rn(a.lamb.om2, __fmul_rn(g[j], g[j])));
                const float u = (full || (e0 + j >= r.lo && e0 + j < r.hi)) ? dat_lamb_direction(a.lamb, m[j], v[j], th[j]) : 0.0f;
                ss_theta = fma((double)th[j], (double)th[j], ss_theta);
                ss_u = fma((double)u, (double)u, ss_u);
            }
            update_st8<EV_LAST>(a.var, full, a.wide, e0, r.lo, r.hi, v);
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                m[j] = __fmaf_rn(a.mu, m[j], __fmaf_rn(a.wd, th[j], g[j]));
                ss_theta = fma((double)th[j], (double)th[j], ss_theta);
                ss_u = fma((double)m[j], (double)m[j], ss_u);
            }
        }
        update_st8<EV_LAST>(a.mom, full, a.wide, e0, r.lo, r.hi, m);
    }
    update_count_in(a, r, tile, ss_theta, ss_u, scratch, &s_last);
}

template <int OPT>
__global__ void __launch_bounds__(DAT_THREADS, UPDATE_CTAS)
k_update_pass2(const __grid_constant__ UpdateArgs a)
{
    dat_after_previous();
    const TileRange r = dat_tile_range(a.tiles, blockIdx.x);
    const float na = -__ldcg(a.step_a + r.layer);        // (no __ldg: written by a kernel that this one may have been started under)
#pragma unroll
    for (int it = 0; it < DAT_TILE / 8 / DAT_THREADS; ++it) {
        const int64_t e0 = r.begin + 8 * (int64_t)(it * DAT_THREADS + threadIdx.x);
        if (e0 >= r.end) continue;
        const bool full = e0 >= r.lo && e0 + 8 <= r.hi;
        float th[8], m[8];
        update_ld8<EV_FIRST>(a.theta, full, a.wide, e0, r.lo, r.hi, th);
        update_ld8<EV_FIRST>(a.mom, full, a.wide, e0, r.lo, r.hi, m);
        if (OPT == OPT_LAMB) {
            float v[8];
            update_ld8<EV_FIRST>(a.var, full, a.wide, e0, r.lo, r.hi, v);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const float u = (full || (e0 + j >= r.lo && e0 + j < r.hi)) ? dat_lamb_direction(a.lamb, m[j], v[j], th[j]) : 0.0f;
                th[j] = __fmaf_rn(na, u, th[j]);
            }
        } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) th[j] = __fmaf_rn(na, m[j], th[j]);
        }
        update_st8<EV_FIRST>(a.theta, full, a.wide, e0, r.lo, r.hi, th);
    }
}

static bool update_wide(const void *a, const void *b, const void *c, const void *d)
{
    return (((uintptr_t)a | (uintptr_t)b | (uintptr_t)c | (uintptr_t)d) & 31u) == 0;
}

// The arguments of a plan's two passes.
static UpdateArgs update_args(const dat_plan_t *plan, float *theta, float *mom, float *var, const float *g_hat, float lr, float c_l, float c_u, float *norms_out)
{
    UpdateArgs a = {};
    a.tiles = plan_tiles(plan);
    a.theta = theta;
    a.mom = mom;
    a.var = var;
    a.g_hat = g_hat;
    a.lr = lr;
    a.c_l = c_l;
    a.c_u = c_u;
    a.wide = update_wide(theta, mom, var, g_hat);
    a.partials = plan->d_partials;
    a.step_a = plan->d_step_a;
    a.norms_out = norms_out;
    a.count = plan->d_count;
    a.status = plan->d_status;
    return a;
}

extern "C" int dat_lalr_step(dat_plan_t *plan, float *theta, float *mom, const float *g_hat,
                             const dat_hparams_t *hp, float *layer_norms_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !g_hat || !hp) return DAT_ERR_ARG;
    if (!dat_aligned16(theta) || !dat_aligned16(mom) || !dat_aligned16(g_hat) ||
        (layer_norms_out && !dat_aligned16(layer_norms_out)))
        return DAT_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    UpdateArgs a = update_args(plan, theta, mom, nullptr, g_hat, hp->lr, hp->c_l, hp->c_u, layer_norms_out);
    a.mu = hp->momentum;
    a.wd = hp->weight_decay;
    DAT_CUDA(plan, dat_launch_after(k_update_pass1<OPT_MOMENTUM>, dim3((unsigned)plan->n_tiles), s, a));
    DAT_LAUNCHED(plan);
    DAT_CUDA(plan, dat_launch_after(k_update_pass2<OPT_MOMENTUM>, dim3((unsigned)plan->n_tiles), s, a));
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

extern "C" int dat_lamb_step(dat_plan_t *plan, float *theta, float *mom, float *var, const float *g_hat,
                             const dat_lamb_hparams_t *hp, int64_t t, float *layer_norms_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta || !mom || !var || !g_hat || !hp || t < 1) return DAT_ERR_ARG;
    if (!(hp->beta1 > 0.0f && hp->beta1 < 1.0f && hp->beta2 > 0.0f && hp->beta2 < 1.0f)) return DAT_ERR_ARG;
    if (!dat_aligned16(theta) || !dat_aligned16(mom) || !dat_aligned16(var) || !dat_aligned16(g_hat) ||
        (layer_norms_out && !dat_aligned16(layer_norms_out)))
        return DAT_ERR_ALIGN;
    cudaStream_t s = (cudaStream_t)stream;
    UpdateArgs a = update_args(plan, theta, mom, var, g_hat, hp->lr, hp->c_l, hp->c_u, layer_norms_out);
    a.lamb = dat_lamb_const(hp, t);
    DAT_CUDA(plan, dat_launch_after(k_update_pass1<OPT_LAMB>, dim3((unsigned)plan->n_tiles), s, a));
    DAT_LAUNCHED(plan);
    DAT_CUDA(plan, dat_launch_after(k_update_pass2<OPT_LAMB>, dim3((unsigned)plan->n_tiles), s, a));
    DAT_LAUNCHED(plan);
    return DAT_OK;
}

// ------------------------------------------------------------------------------------------
// dat_lalr_step_static: the LALR update for callers that cannot allocate device memory.
// No plan, no cudaMalloc: the layer table, the per-tile partial sums and the per-layer step
// lengths live in one fixed array that is part of the library image on every device.
// ------------------------------------------------------------------------------------------
struct StaticScratch {
    int64_t off[DAT_STATIC_MAX_LAYERS + 1];
    int64_t tile_base[DAT_STATIC_MAX_LAYERS + 1];
    double partials[2 * (DAT_STATIC_MAX_TILES + DAT_STATIC_MAX_LAYERS)];      // (see below)
    float step_a[DAT_STATIC_MAX_LAYERS];
    uint32_t status, count[DAT_STATIC_MAX_LAYERS];
};

static __device__ __align__(256) unsigned char g_static_scratch[sizeof(StaticScratch)];

// In host code `g_static_scratch` is only a handle; the device address has to be asked for,
// once per device, with that device current.
#define DAT_STATIC_MAX_DEVICES 64
static StaticScratch *g_static_ptr[DAT_STATIC_MAX_DEVICES];

extern "C" int dat_lalr_step_static(int64_t num_layers, const int64_t *layer_offsets, float *theta, float *mom,
                                    const float *g_hat, const dat_hparams_t *hp, float *layer_norms_out,
                                    void *stream)
{
    if (!layer_offsets || !theta || !mom || !g_hat || !hp) return DAT_ERR_ARG;
    if (num_layers < 1) return DAT_ERR_ARG;
    if (num_layers > DAT_STATIC_MAX_LAYERS) return DAT_ERR_TOO_LARGE;
    if (!dat_aligned16(theta) || !dat_aligned16(mom) || !dat_aligned16(g_hat) ||
        (layer_norms_out && !dat_aligned16(layer_norms_out)))
        return DAT_ERR_ALIGN;
    if (layer_offsets[0] != 0) return DAT_ERR_LAYOUT;
    int64_t tile_base[DAT_STATIC_MAX_LAYERS + 1];              // host stack, 32 KB
    int64_t nt = 0, counted = 0;
    for (int64_t l = 0; l < num_layers; ++l) {
        if (layer_offsets[l + 1] <= layer_offsets[l]) return DAT_ERR_LAYOUT;
        tile_base[l] = nt;
        // the documented limit counts tiles from multiples of 4 on; the kernels' start on multiples of 8, one more in a layer at most
        counted += (layer_offsets[l + 1] - (layer_offsets[l] & ~(int64_t)3) + DAT_TILE - 1) / DAT_TILE;
        nt += (layer_offsets[l + 1] - (layer_offsets[l] & ~(int64_t)7) + DAT_TILE - 1) / DAT_TILE;
        if (counted > DAT_STATIC_MAX_TILES) return DAT_ERR_TOO_LARGE;
    }
    tile_base[num_layers] = nt;

    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) { (void)cudaGetLastError(); return DAT_ERR_CUDA; }
    if (dev < 0 || dev >= DAT_STATIC_MAX_DEVICES) return DAT_ERR_UNSUPPORTED;
    if (!g_static_ptr[dev]) {
        StaticScratch *p = nullptr;
        if (cudaGetSymbolAddress((void **)&p, g_static_scratch) != cudaSuccess || !p) {
            (void)cudaGetLastError();
            return DAT_ERR_CUDA;
        }
        g_static_ptr[dev] = p;
    }
    StaticScratch *sc = g_static_ptr[dev];
    cudaStream_t s = (cudaStream_t)stream;
    // the tables are copied from host memory (one of them from this function's stack) on every call:
    // a captured graph would replay those copies from dead memory
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) { (void)cudaGetLastError(); return DAT_ERR_CUDA; }
    if (cap != cudaStreamCaptureStatusNone) return DAT_ERR_UNSUPPORTED;
    const size_t table = (size_t)(num_layers + 1) * sizeof(int64_t);
    cudaError_t e = cudaMemcpyAsync(sc->off, layer_offsets, table, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(sc->tile_base, tile_base, table, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(&sc->status, 0, sizeof(uint32_t) * (size_t)(1 + num_layers), s);   // status and counters start at zero
    if (e != cudaSuccess) { (void)cudaGetLastError(); return DAT_ERR_CUDA; }
    UpdateArgs a = {};
    a.tiles = TileSource{nullptr, sc->off, sc->tile_base, (int)num_layers};
    a.theta = theta;
    a.mom = mom;
    a.g_hat = g_hat;
    a.mu = hp->momentum;
    a.wd = hp->weight_decay;
    a.lr = hp->lr;
    a.c_l = hp->c_l;
    a.c_u = hp->c_u;
    a.wide = update_wide(theta, mom, nullptr, g_hat);
    a.partials = sc->partials;
    a.step_a = sc->step_a;
    a.norms_out = layer_norms_out;
    a.count = sc->count;
    a.status = &sc->status;
    k_update_pass1<OPT_MOMENTUM><<<(unsigned)nt, DAT_THREADS, 0, s>>>(a);
    (void)dat_launch_after(k_update_pass2<OPT_MOMENTUM>, dim3((unsigned)nt), s, a);
    if (cudaGetLastError() != cudaSuccess) return DAT_ERR_CUDA;
    return DAT_OK;
}
