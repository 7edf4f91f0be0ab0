// Plan object, argument validation, status word and the host-buffer entry point.
#include <algorithm>
#include <cmath>
#include <new>

#include "dat_internal.cuh"

#define HOST_GROUPS 8                            // groups of layers of dat_step_host, at most
#define HOST_GROUP_BYTES (4ll << 20)             // of a vector, at least

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

bool dat_aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int dat_cuda_fail(dat_plan_t *plan, cudaError_t e)
{
    if (plan) plan->last_cuda = (int)e;
    (void)cudaGetLastError();   // clear the sticky-less error state for the next call
    return DAT_ERR_CUDA;
}

int dat_check_plan(dat_plan_t *plan)
{
    if (!plan) return DAT_ERR_ARG;
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return dat_cuda_fail(plan, e);
    if (dev != plan->device) return DAT_ERR_ARG;
    return DAT_OK;
}

int dat_check_grads(const dat_plan_t *plan, const float *const *grads, GradPtrs *out)
{
    if (!grads) return DAT_ERR_ARG;
    for (int i = 0; i < plan->M; ++i) {
        if (!grads[i]) return DAT_ERR_ARG;
        if (!dat_aligned16(grads[i])) return DAT_ERR_ALIGN;
        out->p[i] = grads[i];
    }
    for (int i = plan->M; i < DAT_MAX_WORKERS; ++i) out->p[i] = nullptr;
    return DAT_OK;
}

bool dat_grads_wide(const dat_plan_t *plan, const float *const *grads)
{
    uintptr_t all = 0;
    for (int i = 0; i < plan->M; ++i) all |= (uintptr_t)grads[i];
    return (all & 31u) == 0;
}

// Correctly rounded division by a number that is known in advance, after Brisebarre, Muller and Raina, "Accelerating
// correctly rounded floating-point division when the divisor is known in advance" (IEEE Trans. Computers 53(8), 2004):
// with hi = RN(1/y) and lo = RN(1/y - hi), RN(x*hi + RN(x*lo)) differs from x/y by less than 2^-47 of it before the last
// rounding, so it can only be wrong for an x whose quotient lies that close to the middle of two floats.  With the
// 24-bit integers X, Y of the operands' significands, such a quotient has |X 2^s - (2k+1) Y| = e <= 4 for s = 24 or 25;
// the few X that satisfy one of these congruences are found and tried here.  If one of them fails (none has been seen
// for 1 - beta^t), and where x*lo would lose bits to the denormal grid, the kernels form the quotient in double precision
// (dat_div_any).
ConstDiv dat_const_div(float y)
{
    ConstDiv c = {1.0 / (double)y, 0.0f, 0.0f, false};
    if (!(y > 1e-30f && y < 1e30f)) return c;
    c.exact = true;
    c.hi = 1.0f / y;
    c.lo = fmaf(-y, c.hi, 1.0f) / y;
    int ex;
    const uint64_t Y = (uint64_t)(frexpf(y, &ex) * 16777216.0f);         // 2^23 <= Y < 2^24
    uint64_t odd = Y;
    int tz = 0;
    while (!(odd & 1)) { odd >>= 1; ++tz; }
    uint64_t inv = odd;                                                  // inverse of `odd` modulo 2^64 (Newton)
    for (int i = 0; i < 6; ++i) inv *= 2 - odd * inv;
    for (int s = 24; s <= 25; ++s)
        for (int e = -4; e <= 4; ++e) {
            if (e == 0 || (e & ((1 << tz) - 1))) continue;              // 2^tz divides X 2^s and (2k+1) Y, so it divides e
            if (tz > 2) continue;
            const uint64_t mod = 1ull << (s - tz);
            const uint64_t q0 = (uint64_t)(int64_t)(e >> tz) * inv & (mod - 1);     // (2k+1) = e/2^tz * odd^-1 (mod 2^(s-tz))
            for (uint64_t q = q0; q < (1ull << 25); q += mod) {
                if (!(q & 1) || q < (1ull << 24)) continue;             // midpoints have 25 significant bits
                const uint64_t num = q * Y - (uint64_t)(int64_t)e;      // = X 2^s
                if (num & ((1ull << s) - 1)) continue;
                const uint64_t X = num >> s;
                if (X < (1ull << 23) || X >= (1ull << 24)) continue;
                const float x = (float)X;
                if (fmaf(x, c.hi, x * c.lo) != x / y) c.exact = false;
            }
        }
    return c;
}

LambConst dat_lamb_const(const dat_lamb_hparams_t *hp, int64_t t)
{
    LambConst c;
    c.beta1 = hp->beta1;
    c.beta2 = hp->beta2;
    c.om1 = 1.0f - hp->beta1;
    c.om2 = 1.0f - hp->beta2;
    c.bc1 = dat_const_div((float)(1.0 - pow((double)hp->beta1, (double)t)));      // 1 - beta^t in double, rounded once
    c.bc2 = dat_const_div((float)(1.0 - pow((double)hp->beta2, (double)t)));
    c.zeta = hp->zeta;
    c.wd = hp->weight_decay;
    return c;
}

PhiloxKeys dat_make_keys(uint64_t seed, uint64_t step)
{
    PhiloxKeys k;
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)step;
    for (int r = 0; r < 10; ++r) {
        k.k0[r] = k0;
        k.k1[r] = k1;
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    k.seed_hi = (uint32_t)(seed >> 32);
    return k;
}

void dat_make_worker_table(const PhiloxKeys &keys, int M, PhiloxWorkers *out)
{
    for (int i = 0; i <= M; ++i) out->w[i] = dat_philox_worker(0u, (uint32_t)i, keys);
}

extern "C" int dat_plan_create(dat_plan_t **out, int64_t num_layers, const int64_t *layer_offsets,
                               int num_workers, int bits, int scale_mode, int rng_bits)
{
    if (!out) return DAT_ERR_ARG;
    *out = nullptr;
    if (!layer_offsets || num_layers < 1 || num_layers > (1 << 24)) return DAT_ERR_ARG;
    if (num_workers < 1 || num_workers > DAT_MAX_WORKERS) return DAT_ERR_ARG;
    if (!(bits == 1 || bits == 2 || bits == 4 || bits == 8 || bits == 16 || bits == 32)) return DAT_ERR_BITS;
    if (scale_mode != DAT_SCALE_SHARED_MAX && scale_mode != DAT_SCALE_PER_WORKER) return DAT_ERR_ARG;
    if (rng_bits != DAT_RNG_BITS_16 && rng_bits != DAT_RNG_BITS_23) return DAT_ERR_ARG;
    if (layer_offsets[0] != 0) return DAT_ERR_LAYOUT;
    for (int64_t l = 0; l < num_layers; ++l)
        if (layer_offsets[l + 1] <= layer_offsets[l]) return DAT_ERR_LAYOUT;
    if (layer_offsets[num_layers] > ((int64_t)1 << 40)) return DAT_ERR_ARG;

    dat_plan_t *p = new (std::nothrow) dat_plan_t();
    if (!p) return DAT_ERR_NOMEM;
    cudaError_t e = cudaGetDevice(&p->device);
    if (e != cudaSuccess) { delete p; (void)cudaGetLastError(); return DAT_ERR_CUDA; }
    e = cudaDeviceGetAttribute(&p->sm_count, cudaDevAttrMultiProcessorCount, p->device);
    if (e != cudaSuccess) { delete p; (void)cudaGetLastError(); return DAT_ERR_CUDA; }

    p->h = num_layers;
    p->d = layer_offsets[num_layers];
    p->M = num_workers;
    p->bits = bits;
    p->scale_mode = scale_mode;
    p->rng_bits = rng_bits;
    p->S = (bits == 32) ? 0u : (uint32_t)((1ull << bits) - 1ull);
    try {
        p->offsets.assign(layer_offsets, layer_offsets + num_layers + 1);
        p->tile_base.resize(num_layers + 1);
    } catch (...) { delete p; return DAT_ERR_NOMEM; }
    int64_t nt = 0;
    for (int64_t l = 0; l < num_layers; ++l) {
        p->tile_base[l] = nt;
        const int64_t a = p->offsets[l] & ~(int64_t)7;
        nt += (p->offsets[l + 1] - a + DAT_TILE - 1) / DAT_TILE;
    }
    p->tile_base[num_layers] = nt;
    p->n_tiles = nt;
    const int eff_bits = (bits == 32) ? 0 : bits;
    p->level_bytes = (int64_t)align_up((size_t)((p->d * eff_bits + 7) / 8), 16);
    p->sign_bytes = (bits == 32) ? 0 : (int64_t)align_up((size_t)((p->d + 7) / 8), 16);

    // carve the workspace
    const size_t h1 = (size_t)num_layers + 1, h = (size_t)num_layers;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 256); return o; };
    const int64_t pieces = (p->d + DAT_FLAT - 1) / DAT_FLAT;
    const size_t o_off = take(h1 * 8), o_tb = take(h1 * 8), o_fl = take(((size_t)pieces + 1) * 4), o_td = take((size_t)nt * sizeof(TileDesc)), o_ct = take(h * 4);
    const size_t o_part = take((size_t)nt * (size_t)(num_workers > 2 ? num_workers : 2) * 8);
    const size_t o_wn = take((size_t)num_workers * h * 4);
    const size_t o_sc = take(h * 4), o_qm = take((size_t)num_workers * h * 4), o_dq = take(h * 4), o_sa = take(h * 4);
    const size_t o_nr = take(2 * h * 4), o_st = take(256);
    p->ws_bytes = off;

    // the tables, laid out as on the device (one copy): layers, per-layer tiles, the layer of every flat piece's first element
    std::vector<char> tables;
    try { tables.resize(o_ct); } catch (...) { delete p; return DAT_ERR_NOMEM; }
    std::copy(p->offsets.begin(), p->offsets.end(), (int64_t *)(tables.data() + o_off));
    std::copy(p->tile_base.begin(), p->tile_base.end(), (int64_t *)(tables.data() + o_tb));
    TileDesc *tile = (TileDesc *)(tables.data() + o_td);
    for (int64_t l = 0; l < num_layers; ++l)
        for (int64_t t = p->tile_base[l]; t < p->tile_base[l + 1]; ++t)
            *tile++ = TileDesc{p->offsets[l], p->offsets[l + 1], (p->offsets[l] & ~(int64_t)7) + (t - p->tile_base[l]) * DAT_TILE, (int32_t)l,
                               (int32_t)p->tile_base[l]};
    int32_t *flat_layer = (int32_t *)(tables.data() + o_fl);
    for (int64_t t = 0, l = 0; t < pieces; ++t) {
        while (p->offsets[l + 1] <= t * DAT_FLAT) ++l;
        flat_layer[t] = (int32_t)l;
    }
    flat_layer[pieces] = (int32_t)(num_layers - 1);

    e = cudaMalloc((void **)&p->ws, p->ws_bytes);
    if (e != cudaSuccess) { delete p; (void)cudaGetLastError(); return DAT_ERR_NOMEM; }
    p->d_offsets = (int64_t *)(p->ws + o_off);
    p->d_tile_base = (int64_t *)(p->ws + o_tb);
    p->d_tiles = (TileDesc *)(p->ws + o_td);
    p->d_flat_layer = (int32_t *)(p->ws + o_fl);
    p->d_count = (uint32_t *)(p->ws + o_ct);
    p->d_partials = (double *)(p->ws + o_part);
    p->d_worker_norms = (float *)(p->ws + o_wn);
    p->d_scales = (float *)(p->ws + o_sc);
    p->d_qmul = (float *)(p->ws + o_qm);
    p->d_dq = (float *)(p->ws + o_dq);
    p->d_step_a = (float *)(p->ws + o_sa);
    p->d_norms = (float *)(p->ws + o_nr);
    p->d_status = (uint32_t *)(p->ws + o_st);
    e = cudaMemset(p->ws + o_ct, 0, p->ws_bytes - o_ct);
    if (e == cudaSuccess) e = cudaMemcpy(p->ws, tables.data(), tables.size(), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaFree(p->ws);
        delete p;
        (void)cudaGetLastError();
        return DAT_ERR_CUDA;
    }
    const int rc = dat_pipe_build(p);
    if (rc != DAT_OK) {
        dat_pipe_destroy(p);
        cudaFree(p->ws);
        delete p;
        return rc;
    }
    *out = p;
    return DAT_OK;
}

extern "C" int dat_plan_set_origin(dat_plan_t *plan, int64_t elem_base, int64_t worker_base)
{
    if (!plan || elem_base < 0 || (elem_base & 7) || worker_base < 0 || worker_base + plan->M > ((int64_t)1 << 32)) return DAT_ERR_ARG;
    plan->elem_base = elem_base;
    plan->worker_base = (uint32_t)worker_base;
    return DAT_OK;
}

extern "C" int dat_plan_destroy(dat_plan_t *plan)
{
    if (!plan) return DAT_OK;
    int rc = DAT_OK;
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != plan->device) cudaSetDevice(plan->device);
    if (cudaDeviceSynchronize() != cudaSuccess) rc = DAT_ERR_CUDA;
    dat_pipe_destroy(plan);
    if (plan->stage) cudaFree(plan->stage);
    if (plan->copy_in) cudaStreamDestroy(plan->copy_in);
    if (plan->copy_out) cudaStreamDestroy(plan->copy_out);
    for (cudaEvent_t ev : plan->events) cudaEventDestroy(ev);
    if (plan->ws) cudaFree(plan->ws);
    if (prev >= 0 && prev != plan->device) cudaSetDevice(prev);
    (void)cudaGetLastError();
    delete plan;
    return rc;
}

extern "C" int dat_plan_sizes(const dat_plan_t *plan, int64_t *level_bytes_per_worker,
                              int64_t *sign_bytes_per_worker, int64_t *num_scales,
                              int64_t *workspace_bytes)
{
    if (!plan) return DAT_ERR_ARG;
    if (level_bytes_per_worker) *level_bytes_per_worker = plan->level_bytes;
    if (sign_bytes_per_worker) *sign_bytes_per_worker = plan->sign_bytes;
    if (num_scales) *num_scales = (plan->scale_mode == DAT_SCALE_PER_WORKER) ? plan->h * plan->M : plan->h;
    if (workspace_bytes) *workspace_bytes = (int64_t)plan->ws_bytes;
    return DAT_OK;
}

extern "C" int dat_get_status(dat_plan_t *plan, uint32_t *flags_out, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!flags_out) return DAT_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    uint32_t v = 0;
    DAT_CUDA(plan, cudaMemcpyAsync(&v, plan->d_status, sizeof v, cudaMemcpyDeviceToHost, s));
    DAT_CUDA(plan, cudaMemsetAsync(plan->d_status, 0, sizeof v, s));
    DAT_CUDA(plan, cudaStreamSynchronize(s));
    if (v & DAT_STATUS_TIMEOUT) {       // the call that gave up left its counters mid-way
        DAT_CUDA(plan, dat_pipe_reset(plan, s));
        DAT_CUDA(plan, cudaStreamSynchronize(s));
    }
    *flags_out = v;
    return DAT_OK;
}

extern "C" int64_t dat_plan_launch_count(const dat_plan_t *plan) { return plan ? plan->launches : 0; }

extern "C" int dat_last_cuda_error(const dat_plan_t *plan) { return plan ? plan->last_cuda : 0; }

extern "C" const char *dat_strerror(int code)
{
    switch (code) {
    case DAT_OK: return "ok";
    case DAT_ERR_ARG: return "invalid argument (null pointer, size or value out of range, wrong device)";
    case DAT_ERR_ALIGN: return "device pointer is not 16-byte aligned";
    case DAT_ERR_BITS: return "bits must be one of 1, 2, 4, 8, 16 (or 32 where no codes are involved)";
    case DAT_ERR_LAYOUT: return "layer offsets must start at 0 and increase strictly";
    case DAT_ERR_CUDA: return "a CUDA runtime call failed";
    case DAT_ERR_NOMEM: return "out of memory";
    case DAT_ERR_UNSUPPORTED: return "not implemented in this build";
    case DAT_ERR_TOO_LARGE: return "problem exceeds the fixed capacity of this entry point (see DAT_STATIC_MAX_*)";
    default: return "unknown error code";
    }
}

// The staging buffers of dat_step_host (first call of a plan).
static int host_stage(dat_plan_t *plan, size_t stride)
{
    if (plan->stage) return DAT_OK;
    const cudaError_t e = cudaMalloc((void **)&plan->stage, (size_t)(plan->M + 2) * stride * 4);
    if (e == cudaSuccess) return DAT_OK;
    plan->stage = nullptr;
    plan->last_cuda = (int)e;
    (void)cudaGetLastError();
    return DAT_ERR_NOMEM;
}

// Groups of layers that the call is cut into: of at least four megabytes per vector, below which the copies' fixed costs
// show, and at most eight; what does not overlap is the last group's step and copies back (ms, one group / 1 MB / 4 MB /
// 8 MB and more, pinned memory):
//   3 million elements, M = 2: 1.39 / 1.35 / 1.28 / 1.36, M = 8: 2.76 / 2.85 / 2.62 / 2.72, M = 32: 8.21 / 8.98 / 8.17 / 8.12
//   1 million, M = 8: 0.99 / 1.05 / one    ResNet-18, M = 6: 8.21 / 7.37 / 7.37 / 7.30 (16, 32 groups: 7.42, 7.65)
// One group where some buffer is pageable: those copies block the host one by one, so nothing overlaps, and they are
// slower in pieces (ResNet-18, M = 3: 25.3 ms in groups, 24.2 in one; 3 million elements, M = 2: 5.5, 4.7).
static int host_groups(const dat_plan_t *plan, const float *theta, const float *mom, const float *const *grads)
{
    const int64_t most = plan->d * 4 / HOST_GROUP_BYTES;
    if (most < 2) return 1;
    for (int i = -2; i < plan->M; ++i) {
        cudaPointerAttributes at;
        const bool known = cudaPointerGetAttributes(&at, i == -2 ? theta : i == -1 ? mom : grads[i]) == cudaSuccess;
        if (!known) (void)cudaGetLastError();
        if (!known || at.type == cudaMemoryTypeUnregistered) return 1;
    }
    return most > HOST_GROUPS ? HOST_GROUPS : (int)most;
}

// The groups' lists, the streams and events (first call in groups).
static int host_prepare(dat_plan_t *plan, int groups)
{
    const int rc = dat_pipe_groups(plan, groups);
    if (rc != DAT_OK) return rc;
    cudaError_t e = cudaSuccess;
    if (!plan->copy_in) e = cudaStreamCreateWithFlags(&plan->copy_in, cudaStreamNonBlocking);
    if (e == cudaSuccess && !plan->copy_out) e = cudaStreamCreateWithFlags(&plan->copy_out, cudaStreamNonBlocking);
    while (e == cudaSuccess && plan->events.size() < 2 + 2 * (size_t)dat_pipe_group_count(plan)) {
        cudaEvent_t ev;
        e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e == cudaSuccess) plan->events.push_back(ev);
    }
    return e == cudaSuccess ? DAT_OK : dat_cuda_fail(plan, e);
}

// All of it on the caller's stream: copies in, the step, copies back.
static int host_in_one(dat_plan_t *plan, float *theta_host, float *mom_host, const float *const *grads_host, size_t stride, uint64_t seed, uint64_t step,
                       const dat_hparams_t *hp, cudaStream_t s)
{
    const size_t bytes = (size_t)plan->d * 4;
    float *d_theta = plan->stage, *d_mom = plan->stage + stride;
    const float *d_grads[DAT_MAX_WORKERS];
    DAT_CUDA(plan, cudaMemcpyAsync(d_theta, theta_host, bytes, cudaMemcpyHostToDevice, s));
    DAT_CUDA(plan, cudaMemcpyAsync(d_mom, mom_host, bytes, cudaMemcpyHostToDevice, s));
    for (int i = 0; i < plan->M; ++i) {
        float *g = plan->stage + (size_t)(i + 2) * stride;
        DAT_CUDA(plan, cudaMemcpyAsync(g, grads_host[i], bytes, cudaMemcpyHostToDevice, s));
        d_grads[i] = g;
    }
    const int rc = dat_step(plan, d_theta, d_mom, d_grads, seed, step, hp, nullptr, nullptr, nullptr, s);
    if (rc != DAT_OK) return rc;
    DAT_CUDA(plan, cudaMemcpyAsync(theta_host, d_theta, bytes, cudaMemcpyDeviceToHost, s));
    DAT_CUDA(plan, cudaMemcpyAsync(mom_host, d_mom, bytes, cudaMemcpyDeviceToHost, s));
    return DAT_OK;
}

// The copies are what this call costs (PCIe); they run group of layers by group of layers on streams of their own, so
// that the step of one group and its copies back run under the copies in of the next (ResNet-18, M = 6: 358 MB in and
// 89 MB out).
static int host_enqueue(dat_plan_t *plan, float *theta_host, float *mom_host, const float *const *grads_host, size_t stride, uint64_t seed, uint64_t step,
                        const dat_hparams_t *hp, cudaStream_t s)
{
    float *d_theta = plan->stage, *d_mom = plan->stage + stride;
    const float *d_grads[DAT_MAX_WORKERS];
    for (int i = 0; i < plan->M; ++i) d_grads[i] = plan->stage + (size_t)(i + 2) * stride;
    const int G = dat_pipe_group_count(plan);
    DAT_CUDA(plan, cudaEventRecord(plan->events[0], s));
    DAT_CUDA(plan, cudaStreamWaitEvent(plan->copy_in, plan->events[0], 0));
    for (int k = 0; k < G; ++k) {
        int64_t a, b;
        dat_pipe_group_range(plan, k, &a, &b);
        const size_t bytes = (size_t)(b - a) * 4;
        cudaEvent_t in = plan->events[2 + 2 * (size_t)k], done = plan->events[3 + 2 * (size_t)k];
        DAT_CUDA(plan, cudaMemcpyAsync(d_theta + a, theta_host + a, bytes, cudaMemcpyHostToDevice, plan->copy_in));
        DAT_CUDA(plan, cudaMemcpyAsync(d_mom + a, mom_host + a, bytes, cudaMemcpyHostToDevice, plan->copy_in));
        for (int i = 0; i < plan->M; ++i)
            DAT_CUDA(plan, cudaMemcpyAsync(plan->stage + (size_t)(i + 2) * stride + a, grads_host[i] + a, bytes, cudaMemcpyHostToDevice, plan->copy_in));
        DAT_CUDA(plan, cudaEventRecord(in, plan->copy_in));
        DAT_CUDA(plan, cudaStreamWaitEvent(s, in, 0));
        const int rc = dat_pipe_step_group(plan, k, d_theta, d_mom, d_grads, seed, step, hp, s);
        if (rc != DAT_OK) return rc;
        DAT_CUDA(plan, cudaEventRecord(done, s));
        DAT_CUDA(plan, cudaStreamWaitEvent(plan->copy_out, done, 0));
        DAT_CUDA(plan, cudaMemcpyAsync(theta_host + a, d_theta + a, bytes, cudaMemcpyDeviceToHost, plan->copy_out));
        DAT_CUDA(plan, cudaMemcpyAsync(mom_host + a, d_mom + a, bytes, cudaMemcpyDeviceToHost, plan->copy_out));
    }
    DAT_CUDA(plan, cudaEventRecord(plan->events[1], plan->copy_out));
    DAT_CUDA(plan, cudaStreamWaitEvent(s, plan->events[1], 0));
    return DAT_OK;
}

extern "C" int dat_step_host(dat_plan_t *plan, float *theta_host, float *mom_host,
                             const float *const *grads_host, uint64_t seed, uint64_t step,
                             const dat_hparams_t *hp, void *stream)
{
    int rc = dat_check_plan(plan);
    if (rc != DAT_OK) return rc;
    if (!theta_host || !mom_host || !grads_host || !hp || (step >> 32)) return DAT_ERR_ARG;
    for (int i = 0; i < plan->M; ++i)
        if (!grads_host[i]) return DAT_ERR_ARG;
    if (plan->elem_base || plan->worker_base) return DAT_ERR_UNSUPPORTED;
    cudaStream_t s = (cudaStream_t)stream;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) { (void)cudaGetLastError(); return DAT_ERR_CUDA; }
    if (cap != cudaStreamCaptureStatusNone) return DAT_ERR_UNSUPPORTED;
    // every staged vector starts on a 256-byte boundary
    const size_t stride = align_up((size_t)plan->d * 4, 256) / 4;
    rc = host_stage(plan, stride);
    if (rc != DAT_OK) return rc;
    const int groups = host_groups(plan, theta_host, mom_host, grads_host);
    if (groups > 1) {
        rc = host_prepare(plan, groups);
        if (rc != DAT_OK) return rc;
        rc = host_enqueue(plan, theta_host, mom_host, grads_host, stride, seed, step, hp, s);
    } else {
        rc = host_in_one(plan, theta_host, mom_host, grads_host, stride, seed, step, hp, s);
    }
    if (rc != DAT_OK) {                             // nothing is left in flight on the caller's buffers
        if (groups > 1) (void)cudaStreamSynchronize(plan->copy_in);
        if (groups > 1) (void)cudaStreamSynchronize(plan->copy_out);
        (void)cudaStreamSynchronize(s);
        return rc;
    }
    DAT_CUDA(plan, cudaStreamSynchronize(s));
    return DAT_OK;
}
