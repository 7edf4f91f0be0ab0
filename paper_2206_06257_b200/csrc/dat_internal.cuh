// Internal declarations shared by the translation units of libdat.so (not installed).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "dat.h"

// Elements per tile of the per-layer tiling (tiles never cross a layer boundary; they start on 8-element boundaries
// of the flat vector: 32-byte accesses, and whole Philox blocks).
#define DAT_TILE 4096
#define DAT_THREADS 256
// Pieces of the flat vector (they may span layers) of which a warp quantizes one, two or four.
#define DAT_FLAT 512

struct GradPtrs {
    const float *p[DAT_MAX_WORKERS];
};

// The ten round keys of Philox4x32-10 for one (seed, step): the same for every thread.
struct PhiloxKeys {
    uint32_t k0[10];
    uint32_t k1[10];
    uint32_t seed_hi;   // fourth counter word
};

struct PipeSchedule;    // dat_pipeline.cu

// One per-layer tile of the separate-call kernels (see dat_tile_range): what a CTA needs to know, in one load.
struct TileDesc {
    int64_t lo, hi, begin;             // the layer's bounds; first element of the tile (a multiple of 8)
    int32_t layer, first;              // first: the layer's first tile
};

// LAMB (Algorithm A2): what the kernels need of the hyper-parameters at iteration t.
// Division by a constant 0 < y <= 1 as x*hi + x*lo, hi + lo = 1/y to 2^-48: see dat_const_div (dat_plan.cu) and dat_div_short.
struct ConstDiv {
    double inv;                        // 1/y
    float hi, lo;
    bool exact;                        // the two-operation form rounds correctly for every significand
};
struct LambConst {
    float beta1, beta2, om1, om2, zeta, wd;
    ConstDiv bc1, bc2;                 // 1 - beta1^t, 1 - beta2^t
};
ConstDiv dat_const_div(float y);                             // dat_plan.cu
LambConst dat_lamb_const(const dat_lamb_hparams_t *hp, int64_t t);   // dat_plan.cu

struct dat_plan {
    int device = 0;
    int64_t h = 0, d = 0;
    int M = 0, bits = 0, scale_mode = 0, rng_bits = 16;
    int64_t elem_base = 0;             // global index of the plan's element 0 and of its worker 0 in the random
    uint32_t worker_base = 0;          // streams (dat_plan_set_origin: a plan that covers a slice of a larger problem)
    uint32_t S = 0;
    std::vector<int64_t> offsets;      // host copy, h+1
    std::vector<int64_t> tile_base;    // host copy, h+1: first per-layer tile of each layer
    int64_t n_tiles = 0;               // per-layer tiles in total
    int64_t level_bytes = 0, sign_bytes = 0;

    // device workspace (one allocation, carved up)
    char *ws = nullptr;
    size_t ws_bytes = 0;
    int64_t *d_offsets = nullptr;      // h+1
    int64_t *d_tile_base = nullptr;    // h+1
    TileDesc *d_tiles = nullptr;       // n_tiles
    int32_t *d_flat_layer = nullptr;   // pieces of DAT_FLAT elements + 1: the layer of each piece's first element (last entry: h-1)
    uint32_t *d_count = nullptr;       // h     tiles of the layer that have been summed (k_sumsq; zero between calls)
    double *d_partials = nullptr;      // n_tiles * max(M,2)
    float *d_worker_norms = nullptr;   // M*h
    float *d_scales = nullptr;         // h     nu_l (fused path / scratch)
    float *d_qmul = nullptr;           // h (shared scale) or M*h (per-worker scales): S/nu (0 if nu = 0)
    float *d_dq = nullptr;             // h     nu_l/(S*M)
    float *d_step_a = nullptr;         // h     lr * tau/||u||
    float *d_norms = nullptr;          // 2h
    uint32_t *d_status = nullptr;      // 1

    PipeSchedule *pipe = nullptr;      // work items and tables of dat_step_pipelined, built with the plan

    // dat_step_host: staging buffers, streams for the copies in and out, events
    float *stage = nullptr;
    cudaStream_t copy_in = nullptr, copy_out = nullptr;
    std::vector<cudaEvent_t> events;

    int sm_count = 0;
    int64_t launches = 0;
    int last_cuda = 0;
};

// ---- host helpers (dat_plan.cu) -------------------------------------------------------------
int dat_check_plan(dat_plan_t *plan);                       // device current, non-null
int dat_cuda_fail(dat_plan_t *plan, cudaError_t e);          // records e, returns DAT_ERR_CUDA
bool dat_aligned16(const void *p);
int dat_check_grads(const dat_plan_t *plan, const float *const *grads, GradPtrs *out);
bool dat_grads_wide(const dat_plan_t *plan, const float *const *grads);   // every buffer on a 32-byte boundary
PhiloxKeys dat_make_keys(uint64_t seed, uint64_t step);
struct PhiloxWorkers;
void dat_make_worker_table(const PhiloxKeys &keys, int M, PhiloxWorkers *out);
int dat_pipe_build(dat_plan_t *plan);                        // dat_pipeline.cu (device current)
void dat_pipe_destroy(dat_plan_t *plan);
cudaError_t dat_pipe_reset(dat_plan_t *plan, cudaStream_t s);
int dat_norm_phase(dat_plan_t *plan, const GradPtrs &gp, float *scales_out, cudaStream_t s);      // dat_unfused.cu
int dat_pipe_groups(dat_plan_t *plan, int most);             // the step group by group (dat_step_host)
int dat_pipe_group_count(const dat_plan_t *plan);
void dat_pipe_group_range(const dat_plan_t *plan, int k, int64_t *e0, int64_t *e1);
int dat_pipe_step_group(dat_plan_t *plan, int k, float *theta, float *mom, const float *const *grads, uint64_t seed, uint64_t step,
                        const dat_hparams_t *hp, cudaStream_t s);

#define DAT_CUDA(plan, call)                                              \
    do {                                                                  \
        cudaError_t e__ = (call);                                         \
        if (e__ != cudaSuccess) return dat_cuda_fail((plan), e__);        \
    } while (0)

#define DAT_LAUNCHED(plan)                                                \
    do {                                                                  \
        cudaError_t e__ = cudaGetLastError();                             \
        if (e__ != cudaSuccess) return dat_cuda_fail((plan), e__);        \
        (plan)->launches++;                                               \
    } while (0)

// ---- device helpers ---------------------------------------------------------------------------
#ifdef __CUDACC__

// One Philox4x32-10 block (Salmon et al., SC'11): ten rounds of two 32x32->64 multiplies and
// two three-way XORs; round keys precomputed on the host.
__device__ __forceinline__ void dat_philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                           const PhiloxKeys &k, uint32_t out[4])
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k.k0[r];
        const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k.k1[r];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
        c0 = n0;
        c2 = n2;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// The random words of the four elements 4q .. 4q+3 of `worker`.
__device__ __forceinline__ void dat_random_words(uint64_t q, uint32_t worker, const PhiloxKeys &k,
                                                 uint32_t out[4])
{
    dat_philox((uint32_t)q, (uint32_t)(q >> 32), worker, k.seed_hi, k, out);
}

// The quantizer's random number u1 = 1 + u in [1, 2), u uniform on a 2^-23 grid: the low 23 bits
// of a random word become the mantissa.
__device__ __forceinline__ float dat_u1_from_word(uint32_t w)
{
    return __uint_as_float(0x3F800000u | (w & 0x007FFFFFu));
}

// The same on a 2^-16 grid, from a 16-bit half word: 1 + half / 2^16.
__device__ __forceinline__ float dat_u1_from_half(uint32_t half)
{
    return __uint_as_float(0x3F800000u | (half << 7));
}

// Philox with what does not change along the loops taken out.  Of the counter (q, q_hi, worker, seed_hi) the first
// two rounds multiply words that depend on the element alone or on the worker alone: with those products kept, the
// block of one (element group, worker) pair is two XORs and rounds 2..9 -- 16 of the 20 wide multiplies, which cost
// four issue cycles of the multiply pipe each on sm_100 (measured; LOP3, PRMT and shifts cost two of the ALU pipe,
// FFMA one, a DP2A two of the multiply pipe).
struct PhiloxElem { uint32_t a, b, c; };         // from the element group's counter word q
struct PhiloxWorker { uint32_t x, y, z; };       // from the worker (and q_hi, which is the same for a whole tile)

__device__ __forceinline__ PhiloxElem dat_philox_elem(uint32_t q, const PhiloxKeys &k)
{
    const uint64_t p0 = (uint64_t)0xD2511F53u * q;
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * ((uint32_t)(p0 >> 32) ^ k.seed_hi ^ k.k1[0]);
    return PhiloxElem{(uint32_t)(p1 >> 32), (uint32_t)p1, (uint32_t)p0};
}
__host__ __device__ __forceinline__ PhiloxWorker dat_philox_worker(uint32_t q_hi, uint32_t worker, const PhiloxKeys &k)
{
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * worker;
    const uint64_t p0 = (uint64_t)0xD2511F53u * ((uint32_t)(p1 >> 32) ^ q_hi ^ k.k0[0]);
    return PhiloxWorker{(uint32_t)p1 ^ k.k0[1], (uint32_t)(p0 >> 32) ^ k.k1[1], (uint32_t)p0};
}
__device__ __forceinline__ void dat_philox_block(const PhiloxElem &e, const PhiloxWorker &w, const PhiloxKeys &k, uint32_t out[4])
{
    uint32_t c0 = e.a ^ w.x, c1 = e.b, c2 = e.c ^ w.y, c3 = w.z;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
        const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
        c0 = (uint32_t)(p1 >> 32) ^ c1 ^ k.k0[r];
        c2 = (uint32_t)(p0 >> 32) ^ c3 ^ k.k1[r];
        c1 = (uint32_t)p1;
        c3 = (uint32_t)p0;
    }
    out[0] = c0; out[1] = c1; out[2] = c2; out[3] = c3;
}

// (1 + u) 2^-b of element j of a group of eight, from the group's random words, in one instruction: the exponent
// field of 2^-b plus the uniform number in the mantissa -- half * 128 + ubits as a two-way dot product (multiply
// pipe, no ALU) at 16 bits, low 23 bits OR ubits at 23 bits.  Exact: 1 + u has at most 24 significant bits.
template <bool RNG16>
__device__ __forceinline__ float dat_u1_scaled(const uint32_t *w, int j, uint32_t ubits)
{
    if (RNG16) return __uint_as_float(__dp2a_lo(w[j >> 1], (j & 1) ? 0x8000u : 0x0080u, ubits));
    return __uint_as_float(ubits | (w[j] & 0x007FFFFFu));
}

// The random words of the eight elements of one group: one block at 16 bits, two at 23 bits.
template <bool RNG16> struct PhiloxGroup { PhiloxElem e[RNG16 ? 1 : 2]; };
template <bool RNG16>
__device__ __forceinline__ PhiloxGroup<RNG16> dat_philox_group(uint64_t e0, const PhiloxKeys &k)
{
    PhiloxGroup<RNG16> g;
    g.e[0] = dat_philox_elem((uint32_t)(e0 >> (RNG16 ? 3 : 2)), k);
    if (!RNG16) g.e[RNG16 ? 0 : 1] = dat_philox_elem((uint32_t)(e0 >> 2) + 1u, k);
    return g;
}
template <bool RNG16>
__device__ __forceinline__ void dat_group_words(const PhiloxGroup<RNG16> &g, const PhiloxWorker &w, const PhiloxKeys &k, uint32_t out[8])
{
    dat_philox_block(g.e[0], w, k, out);
    if (!RNG16) dat_philox_block(g.e[RNG16 ? 0 : 1], w, k, out + 4);
}
// Counter words above 32 bits: the same for every group of [begin, begin + n) unless this says so.
template <bool RNG16>
__device__ __forceinline__ bool dat_one_counter_page(uint64_t begin, uint64_t n)
{
    constexpr int SH = 32 + (RNG16 ? 3 : 2);
    return (begin >> SH) == ((begin + n - 1) >> SH);
}

// u1 of the four elements e0 .. e0+3 (e0 a multiple of 4) of `worker`.  rng16 = false: one
// Philox block per four elements, word j for element e0+j.  rng16 = true: one block per EIGHT
// elements (counter e/8); element e takes word (e/2) mod 4, low half if e is even, high if odd.
__device__ __forceinline__ void dat_u1x4(uint64_t e0, uint32_t worker, const PhiloxKeys &k, bool rng16, float u1[4])
{
    uint32_t w[4];
    if (!rng16) {
        dat_random_words(e0 >> 2, worker, k, w);
#pragma unroll
        for (int j = 0; j < 4; ++j) u1[j] = dat_u1_from_word(w[j]);
    } else {
        dat_random_words(e0 >> 3, worker, k, w);
        const uint32_t wa = (e0 & 4u) ? w[2] : w[0], wb = (e0 & 4u) ? w[3] : w[1];
        u1[0] = dat_u1_from_half(wa & 0xFFFFu);
        u1[1] = dat_u1_from_half(wa >> 16);
        u1[2] = dat_u1_from_half(wb & 0xFFFFu);
        u1[3] = dat_u1_from_half(wb >> 16);
    }
}

// Stochastic level of one element (Eq. xi): level = min(floor(|g|*qmul + u), S) with u uniform
// on [0,1).  With u1 = 1 + u in [1,2), y = fma(|g|, qmul, u1) is clamped to S+1 and
// level = floor(y) - 1.  y lies in [1, 65537): adding 2^23 - 1 with rounding toward -inf leaves
// floor(y) - 1 in the low mantissa bits.  Returns those float bits, 0x4B000000 + level.  (A NaN has level S.)
__device__ __forceinline__ uint32_t dat_level_bits_u1(float g, float qmul, float S1_f, float u1)
{
    const float y = fminf(__fmaf_rn(fabsf(g), fabsf(qmul), u1), S1_f);
    return __float_as_uint(__fadd_rd(y, 8388607.0f));
}

// The factor S/nu of a layer with norm nu (0 for a zero layer).  Its sign bit set says that some gradient of the layer is
// not finite: the scaled form of the level, which knows neither NaN nor infinity times 0, is then left alone.
__device__ __forceinline__ float dat_level_factor(float nu, float S_f, bool finite)
{
    const float t = (nu == 0.0f) ? 0.0f : S_f / nu;
    return finite ? t : __uint_as_float(__float_as_uint(t) | 0x80000000u);
}
// Whether the scaled form applies: t 2^-b is 0 or a normal number.
__device__ __forceinline__ bool dat_scaled_factor(float t, float two_b)
{
    return __float_as_uint(t) == 0u || (t >= 1.17549435e-38f * two_b && t <= 3.402823466e38f);
}

__device__ __forceinline__ uint32_t dat_level_u1(float g, float qmul, float S1_f, float u1)
{
    return dat_level_bits_u1(g, qmul, S1_f, u1) & 0x007FFFFFu;
}

// Largest l in [0, h) with table[l] <= x (table[0] <= x < table[h] assumed).
__device__ __forceinline__ int dat_find(const int64_t *__restrict__ table, int h, int64_t x)
{
    int lo = 0, hi = h;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(table + mid) <= x) lo = mid; else hi = mid;
    }
    return lo;
}

// The same by a whole warp: every lane looks at an entry of its own, so 32 layers take one access and 4096 three, one
// after the other, instead of 5 and 12 (dat_lalr_step_static, 20 million elements: 3000 layers 133.7 -> 116.1 us).
__device__ __forceinline__ int dat_find_warp(const int64_t *__restrict__ table, int h, int64_t x)
{
    const int lane = threadIdx.x & 31;
    int lo = 0, n = h;
    while (n > 1) {
        const int step = (n + 31) / 32, at = lane * step;
        const unsigned le = __ballot_sync(0xFFFFFFFFu, at < n && __ldg(table + lo + min(at, n - 1)) <= x);
        const int k = 31 - __clz(le);             // (lane 0's entry is not above x)
        lo += k * step;
        n = min(step, n - k * step);
    }
    return lo;
}

// One thread's release / acquire point at GPU scope.  What the CTA's other threads wrote before a barrier that this
// thread has passed is released with it (and what it acquires holds for threads behind a later barrier), so one thread
// per CTA fences, and with the acquire-release fence: __threadfence() is the sequentially consistent one.
__device__ __forceinline__ void dat_fence() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

// One thread, the CTA's part of a count being complete: counts it in; returns whether it was the last of `total`
// (what the others released before counting is then visible to this CTA's threads after their next barrier).
__device__ __forceinline__ bool dat_count_in(uint32_t *count, uint32_t total, uint32_t n = 1u)
{
    dat_fence();
    const bool last = atomicAdd(count, n) == total - n;
    if (last) dat_fence();
    return last;
}

__device__ __forceinline__ double dat_warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}

// Sum over a block of DAT_THREADS threads in a fixed order; result valid in thread 0.
// `scratch` holds at least DAT_THREADS/32 doubles; safe to call repeatedly.
__device__ __forceinline__ double dat_block_sum(double v, double *scratch)
{
    v = dat_warp_sum(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) scratch[warp] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int w = 0; w < DAT_THREADS / 32; ++w) r += scratch[w];
    }
    return r;
}

// ------------------------------------------------------------------------------------------
// Per-layer tiling shared by the norm kernels: tile t belongs to layer l = find(tile_base, t);
// it covers the flat elements [a + k*DAT_TILE, a + (k+1)*DAT_TILE) ∩ [lo, hi) where
// lo/hi are the layer's bounds, a = lo rounded down to a multiple of 8 and k = t - tile_base[l].
// ------------------------------------------------------------------------------------------
struct TileRange {
    int layer;
    int64_t first;         // the layer's first tile
    int64_t lo, hi;        // layer bounds
    int64_t begin, end;    // begin is a multiple of 8; elements outside [lo, hi) are masked
};

// The tiles of a plan come from its table; without a plan (dat_lalr_step_static) they are found in the layer table, by
// whole warps.
struct TileSource {
    const TileDesc *tiles;
    const int64_t *off, *tile_base;
    int h;
};

__device__ __forceinline__ TileRange dat_tile_range(const TileSource &src, int64_t tile)
{
    TileRange r;
    if (src.tiles) {
        const longlong2 a = __ldg(reinterpret_cast<const longlong2 *>(src.tiles + tile)), b = __ldg(reinterpret_cast<const longlong2 *>(src.tiles + tile) + 1);
        r.lo = a.x;
        r.hi = a.y;
        r.begin = b.x;
        r.layer = (int)(uint32_t)b.y;
        r.first = (int64_t)(b.y >> 32);
    } else {
        r.layer = dat_find_warp(src.tile_base, src.h, tile);
        r.first = __ldg(src.tile_base + r.layer);
        r.lo = __ldg(src.off + r.layer);
        r.hi = __ldg(src.off + r.layer + 1);
        r.begin = (r.lo & ~(int64_t)7) + (tile - r.first) * DAT_TILE;
    }
    r.end = min(r.begin + (int64_t)DAT_TILE, r.hi);
    return r;
}

// Tiles of the layer.
__device__ __forceinline__ int64_t dat_layer_tiles(const TileRange &r)
{
    return (r.hi - (r.lo & ~(int64_t)7) + DAT_TILE - 1) / DAT_TILE;
}

// Loads the four elements e0..e0+3 (e0 a multiple of 4) that lie in [lo, hi); others read 0.
__device__ __forceinline__ void dat_load4(const float *__restrict__ p, int64_t e0, int64_t lo,
                                          int64_t hi, float v[4])
{
    if (e0 >= lo && e0 + 4 <= hi) {
        const float4 f = *reinterpret_cast<const float4 *>(p + e0);
        v[0] = f.x; v[1] = f.y; v[2] = f.z; v[3] = f.w;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (e0 + j >= lo && e0 + j < hi) ? p[e0 + j] : 0.0f;
    }
}

// The same without a branch: reads inside the layer only, what lies outside is 0.  Several of these stay in flight.
__device__ __forceinline__ void dat_load4_masked(const float *__restrict__ p, int64_t e0, int64_t lo, int64_t hi, float v[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int64_t e = e0 + j;
        const float x = p[max(lo, min(e, hi - 1))];
        v[j] = (e >= lo && e < hi) ? x : 0.0f;
    }
}

__device__ __forceinline__ void dat_store4(float *__restrict__ p, int64_t e0, int64_t lo,
                                           int64_t hi, const float v[4])
{
    if (e0 >= lo && e0 + 4 <= hi) {
        *reinterpret_cast<float4 *>(p + e0) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (e0 + j >= lo && e0 + j < hi) p[e0 + j] = v[j];
    }
}

// x / y for 0 < y <= 1, correctly rounded, in two forms.  x*hi + RN(x*lo) is that for finite x of at least 2^-98 (x*lo
// keeps its bits: the denormal grid is below 2^-52 of the quotient).
__device__ __forceinline__ bool dat_div_short(float x, const ConstDiv &c)
{
    return c.exact && (__float_as_uint(x) & 0x7FFFFFFFu) - (29u << 23) < ((255u - 29u) << 23);
}
// Any x: the product with 1/y in double precision, less than 2^-52 of the quotient off, rounded once.  No quotient is a
// midpoint of the float grid, and none is that close to one: for a result of 24 bits the distance is at least 2^-49 of
// it; on the denormal grid, x = k and y = Y 2^-p (Y odd, p >= 1 or Y = 1) in its units, k 2^p / Y = j + 1/2 would make
// an even number odd, and the distance is at least 1 / 2Y > 2^-25 with the error below 2^-28.
__device__ __forceinline__ float dat_div_any(float x, const ConstDiv &c) { return (float)((double)x * c.inv); }

// The LAMB direction of one element from the stored moments: u = m^/(sqrt(v^) + zeta) + wd*theta with the
// bias-corrected m^ = m'/(1 - beta1^t), v^ = v'/(1 - beta2^t) (Algorithm A2; one rounding per operation).
// First moments of elements whose aggregate stays zero decay below 2^-98 and stay among the denormal numbers, where the
// division operator leaves its short path: a server step on ResNet-18, M = 16, b = 4, with most of them decayed takes
// 216 us with it and 184 with the product (177 with the two-operation form for every x, which rounds wrongly there).  One
// branch for both quotients (a branch each: 3 to 5 % of dat_lamb_step and dat_step_lamb; 187 in the server step).
__device__ __forceinline__ float dat_lamb_direction(const LambConst &c, float m_new, float v_new, float theta)
{
    float m_hat, v_hat;
    if (dat_div_short(m_new, c.bc1) && dat_div_short(v_new, c.bc2)) {
        m_hat = __fmaf_rn(m_new, c.bc1.hi, __fmul_rn(m_new, c.bc1.lo));
        v_hat = __fmaf_rn(v_new, c.bc2.hi, __fmul_rn(v_new, c.bc2.lo));
    } else {
        m_hat = dat_div_any(m_new, c.bc1);
        v_hat = dat_div_any(v_new, c.bc2);
    }
    return __fmaf_rn(c.wd, theta, m_hat / (sqrtf(v_hat) + c.zeta));
}

// ------------------------------------------------------------------------------------------
// 16-byte global loads and stores that stay out of L1 and carry an L2 eviction priority.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint64_t dat_policy_evict_last()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t dat_policy_evict_first()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ uint64_t dat_policy_evict_normal()
{
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ float4 dat_ld4_hint(const float *p, uint64_t pol)
{
    float4 v;
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "l"(pol));
    return v;
}
__device__ __forceinline__ void dat_st4_hint(float *p, float4 v, uint64_t pol)
{
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %5;"
                 :: "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "l"(pol) : "memory");
}

// Eight consecutive floats past L1 with an L2 eviction priority.  sm_100 has 32-byte loads and stores: half the
// instructions of two 16-byte ones, and no sector is asked for twice.  They want a 32-byte boundary, which a 16-byte
// aligned buffer may not have (wide: the buffers do; element indices are multiples of 8).
enum { EV_NORMAL = 0, EV_FIRST = 1, EV_LAST = 2 };
template <int EV> __device__ __forceinline__ uint64_t dat_policy()
{
    return EV == EV_FIRST ? dat_policy_evict_first() : EV == EV_LAST ? dat_policy_evict_last() : dat_policy_evict_normal();
}
#define DAT_LD8(Q)                                                                                                          \
    asm volatile("ld.global.L1::no_allocate" Q ".v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"                                   \
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p))
#define DAT_ST8(Q)                                                                                                          \
    asm volatile("st.global" Q ".v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};"                                                   \
                 :: "l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory")
template <int EV> __device__ __forceinline__ void dat_ld8(const float *p, bool wide, float v[8])
{
    if (wide) {
        if (EV == EV_FIRST) DAT_LD8(".L2::evict_first");
        else if (EV == EV_LAST) DAT_LD8(".L2::evict_last");
        else DAT_LD8("");
    } else {
        const float4 a = dat_ld4_hint(p, dat_policy<EV>()), b = dat_ld4_hint(p + 4, dat_policy<EV>());
        v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
}
template <int EV> __device__ __forceinline__ void dat_st8(float *p, bool wide, const float v[8])
{
    if (wide) {
        if (EV == EV_FIRST) DAT_ST8(".L2::evict_first");
        else if (EV == EV_LAST) DAT_ST8(".L2::evict_last");
        else DAT_ST8("");
    } else {
        dat_st4_hint(p, make_float4(v[0], v[1], v[2], v[3]), dat_policy<EV>());
        dat_st4_hint(p + 4, make_float4(v[4], v[5], v[6], v[7]), dat_policy<EV>());
    }
}
#undef DAT_LD8
#undef DAT_ST8
__device__ __forceinline__ bool dat_aligned32(const void *p) { return ((uintptr_t)p & 31u) == 0; }

// ------------------------------------------------------------------------------------------
// Levels and signed sum over the workers for one thread's group of eight consecutive elements
// (Eq. xi, Eq. grad_agg), shared by the kernels that keep codes and sums in registers.
// ------------------------------------------------------------------------------------------
struct QuConst {
    float t, ts, two_b, inv_two_b, den_b;         // S/nu_l, S/nu_l 2^-b, 2^b, 2^-b, 2^(b-149)
    uint32_t ubits;                               // the bits of 2^-b
    bool wide;
};
__device__ __forceinline__ QuConst dat_qu_const(float t, float S_f, bool wide)
{
    const float two_b = S_f + 1.0f, inv_two_b = 1.0f / two_b;
    return QuConst{t, t * inv_two_b, two_b, inv_two_b, two_b * __uint_as_float(1u), __float_as_uint(inv_two_b), wide};
}
// Outside the scaled form's range, or beyond the counters of the worker table.
template <bool RNG16>
__device__ __forceinline__ bool dat_qu_plain(const QuConst &q, int64_t begin, int64_t n)
{
    return !dat_scaled_factor(q.t, q.two_b) || ((begin + n) >> (RNG16 ? 35 : 34)) != 0;
}

// The worker-dependent products of the Philox blocks (counter word q_hi = 0), formed on the host per call.
struct PhiloxWorkers {
    PhiloxWorker w[DAT_MAX_WORKERS + 1];          // the last: the server's stream (index M) of the two-sided step
};

// The M gradient rows of one group of eight elements: levels and signed sum.
//
// Scaled form (S + 1 = 2^b): y = sat(fma(|g|, t 2^-b, (1 + u) 2^-b)) is min(fma(|g|, t, 1 + u), S + 1) 2^-b exactly, and
// one fma towards zero onto the grid of the denormal numbers, y 2^(b-149) - 2^-149, truncates to level 2^-149: the sums
// are then exact sums of denormal numbers (|sum| < 2^23 units), brought back by an exact scaling at the end.  Per
// element: one DP2A for (1 + u) 2^-b, three fused multiply-adds and one LOP3 for the sign.  The issue-limited time of
// this loop per group and worker went from 165 to about 115 cycles per scheduler (both multiply pipe and ALU full).
template <bool RNG16, int UNROLL>
__device__ __forceinline__ void qu_rows(const GradPtrs &gp, const PhiloxKeys &keys, const PhiloxWorkers &pw, const QuConst &qc, int M, int64_t e0, float acc[8])
{
    const PhiloxGroup<RNG16> pg = dat_philox_group<RNG16>((uint64_t)e0, keys);
#pragma unroll UNROLL
    for (int i = 0; i < M; ++i) {          // UNROLL workers' loads and Philox blocks in flight together
        float v[8];
        dat_ld8<EV_FIRST>(gp.p[i] + e0, qc.wide, v);         // a gradient is dead once its level is drawn
        uint32_t w[8];
        dat_group_words<RNG16>(pg, pw.w[i], keys, w);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            const float ys = __saturatef(__fmaf_rn(fabsf(v[j]), qc.ts, dat_u1_scaled<RNG16>(w, j, qc.ubits)));
            const float lev = __fmaf_rz(ys, qc.den_b, __uint_as_float(0x80000001u));
            const float sg = __uint_as_float((__float_as_uint(v[j]) & 0x80000000u) | 0x3F800000u);
            acc[j] = __fmaf_rn(lev, sg, acc[j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = (acc[j] * 0x1p100f) * 0x1p49f;
}

// The same by the plain form of Eq. xi with whole Philox blocks, for a group at a layer's ragged ends or outside the
// scaled form's range (same integers).  Sums in units of one level, four at a time (the call passes no array).
template <bool RNG16, int UNROLL>
__device__ __noinline__ float4 qu_rows_slow4(const GradPtrs &gp, const PhiloxKeys &keys, float t, float two_b, int M, int64_t e0, int64_t lo, int64_t hi)
{
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll UNROLL
    for (int i = 0; i < M; ++i) {              // (one lane here holds up its warp)
        float v[4], u1[4];
        if (UNROLL > 1) dat_load4_masked(gp.p[i], e0, lo, hi, v);
        else dat_load4(gp.p[i], e0, lo, hi, v);
        dat_u1x4((uint64_t)e0, (uint32_t)i, keys, RNG16, u1);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float lf = (float)dat_level_u1(v[j], t, two_b, u1[j]);
            acc[j] += (v[j] < 0.0f) ? -lf : lf;
        }
    }
    return make_float4(acc[0], acc[1], acc[2], acc[3]);
}
template <bool RNG16, int UNROLL>
__device__ __forceinline__ void qu_rows_slow(const GradPtrs &gp, const PhiloxKeys &keys, const QuConst &qc, int M, int64_t e0, int64_t lo, int64_t hi, float acc[8])
{
    const float4 a = qu_rows_slow4<RNG16, UNROLL>(gp, keys, qc.t, qc.two_b, M, e0, lo, hi), b = qu_rows_slow4<RNG16, UNROLL>(gp, keys, qc.t, qc.two_b, M, e0 + 4, lo, hi);
    acc[0] = a.x; acc[1] = a.y; acc[2] = a.z; acc[3] = a.w; acc[4] = b.x; acc[5] = b.y; acc[6] = b.z; acc[7] = b.w;
}

// The signed levels of the four elements e0 .. e0+3 of one worker by the plain form, elements outside the layer 0.
template <bool RNG16>
__device__ __forceinline__ void dat_signed_levels4(const float *g, uint32_t worker, const PhiloxKeys &keys, float t, float two_b, int64_t e0, int64_t lo, int64_t hi, int lev[4])
{
    float v[4], u1[4];
    dat_load4_masked(g, e0, lo, hi, v);
    dat_u1x4((uint64_t)e0, worker, keys, RNG16, u1);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int l = (int)dat_level_u1(v[j], t, two_b, u1[j]);
        lev[j] = (v[j] < 0.0f) ? -l : l;
    }
}

// A group at a layer's ragged end, by its whole warp: a lane takes a worker (of the 64 two), and the signed levels are
// added as integers (four at a time: the call passes no array).  By the group's own lane, worker after worker, the
// warp and its CTA wait for a chain of 2 M loads and blocks; many tiles of a model of small odd layers
// have such a group (by phases, 300 thousand elements in 40 odd layers, M = 64: 121 -> 70 us; 2.1 million in 98, M = 22: 103 -> 90).
template <bool RNG16>
__device__ __noinline__ float4 qu_rows_ragged4(const GradPtrs &gp, const PhiloxKeys &keys, float t, float two_b, int M, int64_t e0, int64_t lo, int64_t hi)
{
    int sum[4] = {0, 0, 0, 0};
    for (int i = threadIdx.x & 31; i < M; i += 32) {
        int lev[4];
        dat_signed_levels4<RNG16>(gp.p[i], (uint32_t)i, keys, t, two_b, e0, lo, hi, lev);
#pragma unroll
        for (int j = 0; j < 4; ++j) sum[j] += lev[j];
    }
    __syncwarp();
    return make_float4((float)__reduce_add_sync(0xFFFFFFFFu, sum[0]), (float)__reduce_add_sync(0xFFFFFFFFu, sum[1]),
                       (float)__reduce_add_sync(0xFFFFFFFFu, sum[2]), (float)__reduce_add_sync(0xFFFFFFFFu, sum[3]));
}

#endif  // __CUDACC__
