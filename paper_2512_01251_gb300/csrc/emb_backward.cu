// Momentum-exchange force with linear Bouzidi interpolated bounce-back, its
// derivative with respect to q, and the adjoint of q with respect to the
// vertices (Sec. 2.2 cites both methods; Sec. 3.4 builds the q table they use).
//
// All reductions are independent of the order in which the GPU runs: the force takes
// per-thread and per-warp sums of three floats each, per-CTA sums in FP64 and one CTA over
// the partials in index order; the per-vertex sums are integers.  No floating-point atomics
// are used.
#include <mutex>

#include "emb_internal.cuh"

#define MEX_BLOCK 256

// direction index of a block offset (ox, oy, oz) in {-1,0,1}^3, code = (ox+1) + 3(oy+1) + 9(oz+1)
__constant__ int8_t c_dir_of_offset[27] = {20, 16, 26, 12, 6, 13, 24, 17, 21, 8, 4, 9, 2, 0,
                                           1,  10, 3,  7,  22, 18, 23, 14, 5, 11, 25, 15, 19};

// Finest-level cell x_f - c_i, or -1 if its block is missing or the cell is solid.
__device__ __forceinline__ int64_t partner_cell(int64_t cell, int cx, int cy, int cz, const int32_t *__restrict__ nbr,
                                                const uint64_t *__restrict__ mask)
{
    int64_t b = cell >> 6;
    int t = (int)(cell & 63);
    int x = (t & 3) - cx, y = ((t >> 2) & 3) - cy, z = (t >> 4) - cz;
    int ox = x < 0 ? -1 : (x > 3 ? 1 : 0), oy = y < 0 ? -1 : (y > 3 ? 1 : 0), oz = z < 0 ? -1 : (z > 3 ? 1 : 0);
    int64_t nb = b;
    if (ox | oy | oz) {
        int d = c_dir_of_offset[(ox + 1) + 3 * (oy + 1) + 9 * (oz + 1)];
        nb = nbr[b * 26 + d - 1];
        if (nb < 0) return -1;
    }
    int lt = (x & 3) + 4 * (y & 3) + 16 * (z & 3);
    if ((mask[nb] >> lt) & 1ull) return -1;
    return nb * 64 + lt;
}

// The cell's populations that the Bouzidi rule of link k reads: f_i, and f_p (below
// q = 1/2, when the partner cell exists) or f_o (from 1/2 on); the others stay 0.
struct LinkPops {
    float q, f_i, f_o, f_p;
    bool has;
    int cx, cy, cz;
};

__device__ __forceinline__ LinkPops link_pops(int64_t k, const int32_t *__restrict__ cell, const uint8_t *__restrict__ dir,
                                              const float *__restrict__ q, const float *__restrict__ pop, int64_t stride,
                                              const int32_t *__restrict__ nbr, const uint64_t *__restrict__ mask)
{
    LinkPops L;
    const int64_t c = cell[k];
    const int d = dir[k];
    L.q = q[k];
    emb_dir(d, L.cx, L.cy, L.cz);
    L.f_i = pop[(int64_t)d * stride + c];
    L.f_o = L.f_p = 0.0f;
    L.has = false;
    if (L.q < 0.5f) {
        const int64_t p = partner_cell(c, L.cx, L.cy, L.cz, nbr, mask);
        L.has = p >= 0;
        if (L.has) L.f_p = pop[(int64_t)d * stride + p];
    } else {
        L.f_o = pop[(int64_t)((d & 1) ? d + 1 : d - 1) * stride + c];
    }
    return L;
}

// Floats in pairs (h + l, l below half an ulp of h) and in threes, in place of FP64: this chip
// has two FP64 lanes a clock and SM against 128 FP32 ones, and with the terms in FP64 the force
// and dF/dq kernels were bound by them (1.72 M links, D3Q19: 131 and 97 us a call).  The sums and
// products below are the error-free transformations of Knuth (two_sum) and Dekker (two_prod,
// by fma).
//   dF/dq, a single value a link: pairs, about 46 bits, rounded to FP32 at once (25 us).
//   The force, a signed sum over a closed body, most of which cancels: threes, which carry a
//   link's term to about 2^-66 of it and a thread's sums to less than FP64's 2^-53 of theirs.
//   1.72 M links of D3Q19: 131 us with FP64, 43 now (51 from a cold L2), the call; pairs
//   took 43 (52).
// Bound now by the gathers of the populations.
struct F2 {
    float h, l;
};
__device__ __forceinline__ F2 two_sum(float a, float b)
{
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ F2 two_prod(float a, float b)
{
    const float p = __fmul_rn(a, b);
    return {p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ F2 f2_norm(float h, float l)  // |h| >= |l|
{
    const float s = __fadd_rn(h, l);
    return {s, __fsub_rn(l, __fsub_rn(s, h))};
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b)
{
    const F2 s = two_sum(a.h, b.h);
    return f2_norm(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b)
{
    const F2 p = two_prod(a.h, b.h);
    return f2_norm(p.h, __fadd_rn(p.l, __fmaf_rn(a.h, b.l, __fmul_rn(a.l, b.h))));
}
__device__ __forceinline__ F2 f2_div(F2 a, F2 b)
{
    const float x = __fdiv_rn(a.h, b.h);
    const float r = __fadd_rn(__fmaf_rn(-x, b.h, a.h), __fmaf_rn(-x, b.l, a.l));
    return f2_norm(x, __fdiv_rn(r, b.h));
}

// a + b + c: b collects the errors of the sums in a, c those of b.
struct F3 {
    float a, b, c;
};
__device__ __forceinline__ void f3_low(F3 &s, float x)  // x of the size of s.b
{
    const F2 t = two_sum(s.b, x);
    s.b = t.h;
    s.c = __fadd_rn(s.c, t.l);
}
__device__ __forceinline__ void f3_add(F3 &s, float x)
{
    const F2 t = two_sum(s.a, x);
    s.a = t.h;
    f3_low(s, t.l);
}
__device__ __forceinline__ void f3_add(F3 &s, F3 x)
{
    f3_add(s, x.a);
    f3_low(s, x.b);
    s.c = __fadd_rn(s.c, x.c);
}
__device__ __forceinline__ double f3_value(F3 s) { return (double)s.a + ((double)s.b + (double)s.c); }

// Zero, or a magnitude in [2^-40, 2^41): sums, products and quotients of a few such values
// neither overflow nor lose low parts to underflow.
__device__ __forceinline__ bool f2_safe(float a)
{
    const uint32_t e = (__float_as_uint(a) >> 23) & 255u;
    return e - 87u <= 80u || a == 0.0f;
}
__device__ __forceinline__ bool link_safe(const LinkPops &L)
{
    return L.q >= 0.0f && L.q <= 1.0f && f2_safe(L.f_i) && f2_safe(L.f_o) && f2_safe(L.f_p);
}

// Fixed-order block reduction of three doubles; every thread receives the sums.
__device__ __forceinline__ void block_sum3(double &a, double &b, double &c)
{
    __shared__ double s[3][MEX_BLOCK];
    s[0][threadIdx.x] = a;
    s[1][threadIdx.x] = b;
    s[2][threadIdx.x] = c;
    __syncthreads();
    for (int w = MEX_BLOCK / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) {
            s[0][threadIdx.x] += s[0][threadIdx.x + w];
            s[1][threadIdx.x] += s[1][threadIdx.x + w];
            s[2][threadIdx.x] += s[2][threadIdx.x + w];
        }
        __syncthreads();
    }
    a = s[0][0];
    b = s[1][0];
    c = s[2][0];
}

__global__ void __launch_bounds__(MEX_BLOCK) k_mex_partial(const int32_t *__restrict__ cell, const uint8_t *__restrict__ dir,
                                                           const float *__restrict__ q, int64_t n,
                                                           const float *__restrict__ pop, int64_t stride,
                                                           const int32_t *__restrict__ nbr,
                                                           const uint64_t *__restrict__ mask, double *__restrict__ part)
{
    F3 ax = {0.0f, 0.0f, 0.0f}, ay = ax, az = ax;
    double fx = 0, fy = 0, fz = 0;  // links outside the range of the threes (NaN and infinities too)
    bool wild = false;
    int held = 0;
    for (int64_t k = (int64_t)blockIdx.x * MEX_BLOCK + threadIdx.x; k < n; k += (int64_t)gridDim.x * MEX_BLOCK) {
        const LinkPops L = link_pops(k, cell, dir, q, pop, stride, nbr, mask);
        if (link_safe(L)) {
            const float q2 = 2.0f * L.q;
            F3 m = {L.f_i, 0.0f, 0.0f};  // f_i plus the population returned against it
            if (L.q < 0.5f) {
                // 2 f_i, or f_i + 2q f_i + (1 - 2q) f_p
                if (L.has) {
                    const F2 w = two_sum(1.0f, -q2), p = two_prod(q2, L.f_i), b = two_prod(w.h, L.f_p),
                             e = two_prod(w.l, L.f_p);
                    f3_add(m, p.h);
                    f3_add(m, b.h);
                    f3_low(m, p.l);
                    f3_low(m, b.l);
                    f3_low(m, e.h);
                    m.c = __fadd_rn(m.c, e.l);
                } else {
                    m.a = 2.0f * L.f_i;
                }
            } else {
                // f_i + (f_i + (2q - 1) f_o) / 2q; 2q - 1 is exact on [1/2, 1].  The quotient in
                // three steps, each from the remainder of the ones before (the first one's exact)
                const F2 p = two_prod(__fsub_rn(q2, 1.0f), L.f_o), N = two_sum(p.h, L.f_i);
                const float x0 = __fdiv_rn(N.h, q2);
                F3 r = {__fmaf_rn(-x0, q2, N.h), 0.0f, 0.0f};
                f3_add(r, N.l);
                f3_add(r, p.l);
                const float inv = __frcp_rn(q2), x1 = __fmul_rn(r.a, inv);
                const float x2 = __fmul_rn(__fadd_rn(__fmaf_rn(-x1, q2, r.a), __fadd_rn(r.b, r.c)), inv);
                f3_add(m, x0);
                f3_low(m, x1);
                m.c = __fadd_rn(m.c, x2);
            }
            const float sx = (float)L.cx, sy = (float)L.cy, sz = (float)L.cz;  // -1, 0, 1
            f3_add(ax, {sx * m.a, sx * m.b, sx * m.c});
            f3_add(ay, {sy * m.a, sy * m.b, sy * m.c});
            f3_add(az, {sz * m.a, sz * m.b, sz * m.c});
            if (++held == 64) {  // the last float of a three rounds at each sum: few of them
                fx += f3_value(ax);
                fy += f3_value(ay);
                fz += f3_value(az);
                ax = ay = az = {0.0f, 0.0f, 0.0f};
                held = 0;
                wild = true;
            }
        } else {
            const double qq = L.q, f_i = L.f_i;
            double g;
            if (qq < 0.5) g = L.has ? 2.0 * qq * f_i + (1.0 - 2.0 * qq) * (double)L.f_p : f_i;
            else g = f_i / (2.0 * qq) + (2.0 * qq - 1.0) / (2.0 * qq) * (double)L.f_o;
            const double m = f_i + g;
            fx += L.cx * m;
            fy += L.cy * m;
            fz += L.cz * m;
            wild = true;
        }
    }
    // the warps' threes first (FP32), then one FP64 value a warp: a lane keeps x and y or z of
    // itself and the lane 16 on, then one of the three, so that the warp's sums take 6 additions
    // and 18 exchanged floats a lane instead of 15 and 45 (x ends in lane 0, y in 8, z in 16)
    __shared__ double s_warp[3][MEX_BLOCK / 32];
    const int lane = threadIdx.x & 31;
    const bool hi = lane & 16, mid = lane & 8;
    auto other = [&](const F3 &v, int o) -> F3 {
        return {__shfl_xor_sync(0xffffffffu, v.a, o), __shfl_xor_sync(0xffffffffu, v.b, o),
                __shfl_xor_sync(0xffffffffu, v.c, o)};
    };
    F3 s = hi ? az : ax;
    f3_add(s, other(hi ? ax : az, 16));
    f3_add(ay, other(ay, 16));
    const F3 out = hi || mid ? s : ay, in = other(out, 8);
    if (!hi && mid) s = ay;
    f3_add(s, in);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) f3_add(s, other(s, o));
    if ((lane & 7) == 0 && lane < 24) s_warp[lane >> 3][threadIdx.x >> 5] = f3_value(s);
    if (__syncthreads_or(wild)) block_sum3(fx, fy, fz);
    if (threadIdx.x < 3) {
        double v = threadIdx.x == 0 ? s_warp[0][0] : (threadIdx.x == 1 ? s_warp[1][0] : s_warp[2][0]);
        for (int w = 1; w < MEX_BLOCK / 32; ++w) v += s_warp[threadIdx.x][w];
        part[3 * blockIdx.x + threadIdx.x] = v + (threadIdx.x == 0 ? fx : (threadIdx.x == 1 ? fy : fz));
    }
}

__global__ void __launch_bounds__(MEX_BLOCK) k_mex_final(const double *__restrict__ part, int nparts, float *__restrict__ F)
{
    double a = 0, b = 0, c = 0;
    for (int i = threadIdx.x; i < nparts; i += MEX_BLOCK) {
        a += part[3 * i];
        b += part[3 * i + 1];
        c += part[3 * i + 2];
    }
    block_sum3(a, b, c);
    if (threadIdx.x == 0) {
        F[0] = (float)a;
        F[1] = (float)b;
        F[2] = (float)c;
    }
}

__global__ void k_mex_bwd(const int32_t *__restrict__ cell, const uint8_t *__restrict__ dir, const float *__restrict__ q,
                          int64_t n, const float *__restrict__ pop, int64_t stride, const int32_t *__restrict__ nbr,
                          const uint64_t *__restrict__ mask, const float *__restrict__ gF, float *__restrict__ gq)
{
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const LinkPops L = link_pops(k, cell, dir, q, pop, stride, nbr, mask);
    const float gx = gF[0], gy = gF[1], gz = gF[2];
    if (link_safe(L) && f2_safe(gx) && f2_safe(gy) && f2_safe(gz)) {
        const F2 s = f2_add(two_sum(L.cx * gx, L.cy * gy), {L.cz * gz, 0.0f});
        F2 r = {0.0f, 0.0f};
        if (L.q < 0.5f) {
            if (L.has) r = f2_mul(s, two_sum(2.0f * L.f_i, -2.0f * L.f_p));
        } else {
            r = f2_div(f2_mul(s, two_sum(L.f_o, -L.f_i)), two_prod(2.0f * L.q, L.q));
        }
        gq[k] = r.h;
        return;
    }
    const double qq = L.q, f_i = L.f_i;
    double g;
    if (qq < 0.5) g = L.has ? 2.0 * (f_i - (double)L.f_p) : 0.0;
    else g = ((double)L.f_o - f_i) / (2.0 * qq * qq);
    const double s = (double)gx * L.cx + (double)gy * L.cy + (double)gz * L.cz;
    gq[k] = (float)(s * g);
}

static emb_status mex_check(emb_forest f, int lattice, int64_t n, int64_t stride, cudaStream_t s)
{
    if (!f || (lattice != 19 && lattice != 27) || n < 0) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    int L = f->max_level;
    if (f->top != L || !f->lv[L].mask_valid) return EMB_ERR_STATE;
    if (stride < f->lv[L].n * 64) return EMB_ERR_BAD_INPUT;
    return emb_build_neighbors(f->lv[L], s);
}

extern "C" emb_status emb_mex_force(emb_forest f, int32_t lattice, const int32_t *d_cell, const uint8_t *d_dir,
                                    const float *d_q, int64_t n, const float *d_pop, int64_t pop_stride, float *d_F,
                                    void *stream)
{
    cudaStream_t s = emb_stream(stream);
    emb_status rc = mex_check(f, lattice, n, pop_stride, s);
    if (rc != EMB_OK) return rc;
    if (!d_F || (n > 0 && (!d_cell || !d_dir || !d_q || !d_pop))) return EMB_ERR_BAD_INPUT;
    const EmbLevel &lv = f->lv[f->max_level];
    int64_t np64 = (n + MEX_BLOCK - 1) / MEX_BLOCK;
    int nparts = (int)(np64 < 1184 ? np64 : 1184);
    if (nparts < 1) nparts = 1;
    double *part = nullptr;
    EMB_CUDA_TRY(emb_malloc_async(&part, 3 * nparts * sizeof(double), s));
    EMB_LAUNCH((k_mex_partial), nparts, MEX_BLOCK, 0, s)(d_cell, d_dir, d_q, n, d_pop, pop_stride, lv.nbr, lv.mask, part);
    EMB_LAUNCH((k_mex_final), 1, MEX_BLOCK, 0, s)(part, nparts, d_F);
    EMB_CUDA_TRY(cudaGetLastError());
    EMB_CUDA_TRY(cudaFreeAsync(part, s));
    return EMB_OK;
}

extern "C" emb_status emb_mex_force_backward(emb_forest f, int32_t lattice, const int32_t *d_cell, const uint8_t *d_dir,
                                             const float *d_q, int64_t n, const float *d_pop, int64_t pop_stride,
                                             const float *d_gF, float *d_gq, void *stream)
{
    cudaStream_t s = emb_stream(stream);
    emb_status rc = mex_check(f, lattice, n, pop_stride, s);
    if (rc != EMB_OK) return rc;
    if (n == 0) return EMB_OK;
    if (!d_cell || !d_dir || !d_q || !d_pop || !d_gF || !d_gq) return EMB_ERR_BAD_INPUT;
    const EmbLevel &lv = f->lv[f->max_level];
    EMB_LAUNCH((k_mex_bwd), emb_grid(n, 256), 256, 0, s)(d_cell, d_dir, d_q, n, d_pop, pop_stride, lv.nbr, lv.mask, d_gF, d_gq);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}

// ---------------------------------------------------------------------------
// Allocation-free variant of emb_mex_force
// ---------------------------------------------------------------------------
// Some callers cannot call cudaMalloc: a solver time loop that reserved all
// device memory up front through its own pool, or code that must not pay a
// driver allocation (latency, implicit device synchronisation) inside a time
// step.  For them the per-CTA partial sums of the force live in this
// file-scope array instead of a stream-ordered allocation.  Every GPU that loads
// the library holds it (3 x EMB_NOALLOC_MEX_PARTS doubles = 192 KB) until exit.
#define EMB_NOALLOC_MEX_PARTS 8192
static __device__ __align__(256) double g_mex_noalloc_part[3 * EMB_NOALLOC_MEX_PARTS];

static std::mutex g_mex_noalloc_mu;
static double *g_mex_noalloc_ptr[64] = {nullptr};        // device address of the array, per device
static unsigned long long g_mex_noalloc_ctx[64] = {0};   // id of the context it was looked up in

// Unique id of the calling thread's current context (0 when none is current or the
// driver entry points are unavailable).  Context ids are never reused within a
// process, so a reset device (a new primary context) is told apart from the old one.
typedef int (*emb_pfn_ctx_get_current)(void **);
typedef int (*emb_pfn_ctx_get_id)(void *, unsigned long long *);
static unsigned long long current_ctx_id()
{
    static emb_pfn_ctx_get_current get_cur = nullptr;
    static emb_pfn_ctx_get_id get_id = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *a = nullptr, *b = nullptr;
        cudaDriverEntryPointQueryResult qa, qb;
        if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &a, 12000, cudaEnableDefault, &qa) == cudaSuccess &&
            qa == cudaDriverEntryPointSuccess &&
            cudaGetDriverEntryPointByVersion("cuCtxGetId", &b, 12000, cudaEnableDefault, &qb) == cudaSuccess &&
            qb == cudaDriverEntryPointSuccess) {
            get_cur = (emb_pfn_ctx_get_current)a;
            get_id = (emb_pfn_ctx_get_id)b;
        }
    }
    if (!get_cur || !get_id) return 0;
    void *ctx = nullptr;
    unsigned long long id = 0;
    if (get_cur(&ctx) != 0 || !ctx) return 0;
    if (get_id(ctx, &id) != 0) return 0;
    return id;
}

// The array's device address for the current device, looked up once per device
// (and again if that device's context was replaced, e.g. by cudaDeviceReset).  In
// host code the array's name is only a host-side stand-in, so the address must come
// from cudaGetSymbolAddress with the device current.
static emb_status mex_noalloc_scratch(double **out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return EMB_ERR_CUDA;
    std::lock_guard<std::mutex> lk(g_mex_noalloc_mu);
    const unsigned long long ctx = current_ctx_id();
    if (!g_mex_noalloc_ptr[dev] || ctx == 0 || ctx != g_mex_noalloc_ctx[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_mex_noalloc_part);
        if (e != cudaSuccess || !p) {
            emb_note_cuda_error(e, "cudaGetSymbolAddress(g_mex_noalloc_part)", __FILE__, __LINE__);
            return EMB_ERR_CUDA;
        }
        g_mex_noalloc_ptr[dev] = (double *)p;
        // the lookup made the device's primary context current if it was not yet
        g_mex_noalloc_ctx[dev] = ctx ? ctx : current_ctx_id();
    }
    *out = g_mex_noalloc_ptr[dev];
    return EMB_OK;
}

extern "C" emb_status emb_mex_force_noalloc(emb_forest f, int32_t lattice, const int32_t *d_cell, const uint8_t *d_dir,
                                            const float *d_q, int64_t n, const float *d_pop, int64_t pop_stride,
                                            float *d_F, void *stream)
{
    if (!f || (lattice != 19 && lattice != 27) || n < 0 || !d_F) return EMB_ERR_BAD_INPUT;
    if (n > 0 && (!d_cell || !d_dir || !d_q || !d_pop)) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    const int L = f->max_level;
    if (f->top != L || !f->lv[L].mask_valid) return EMB_ERR_STATE;
    const EmbLevel &lv = f->lv[L];
    if (pop_stride < lv.n * 64) return EMB_ERR_BAD_INPUT;
    // the neighbour table must already exist (emb_cutlinks or emb_mex_force built it): building it would allocate
    if (lv.n > 0 && !lv.nbr) return EMB_ERR_STATE;
    // one partial sum per CTA of MEX_BLOCK links
    const int64_t nparts64 = n > 0 ? (n + MEX_BLOCK - 1) / MEX_BLOCK : 1;
    if (nparts64 > EMB_NOALLOC_MEX_PARTS) return EMB_ERR_CAPACITY;  // more than 2,097,152 links
    double *part = nullptr;
    emb_status rc = mex_noalloc_scratch(&part);
    if (rc != EMB_OK) return rc;
    cudaStream_t s = emb_stream(stream);
    const int nparts = (int)nparts64;
    EMB_LAUNCH((k_mex_partial), nparts, MEX_BLOCK, 0, s)(d_cell, d_dir, d_q, n, d_pop, pop_stride, lv.nbr, lv.mask, part);
    EMB_LAUNCH((k_mex_final), 1, MEX_BLOCK, 0, s)(part, nparts, d_F);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}

// ---------------------------------------------------------------------------
// dq/dV adjoint
// ---------------------------------------------------------------------------
// Link k adds gq_k lambda_j n / (h n.c) to vertex j of its triangle (world units).  With
// the vertices relative to the cell centre, V_A = c . (B x C) and so on are integers and
// lambda_j = V_j / (c . n), c . n = V_A + V_B + V_C: the sum over a triangle's links
// needs one scalar S_j = sum gq_k K V_j / (c . n)^2 per vertex (K = 2^20 r_o / h), and
// the normal n multiplies it once.
//
// Sums are taken in integers, so that their order does not matter and the atomics that
// form them give the same result every time:
//   k_qbwd_tile    a CTA takes QB_TILE consecutive links (neighbours in space, so they
//                  share triangles); per (tile, triangle) it finds the largest exponent
//                  of each of the three terms, then adds the terms as multiples of 2^-41
//                  of it.  One entry per (tile, triangle) is written, and the exponent
//                  bound of its nine products S_j n_d is raised into the vertices';
//   k_qbwd_scatter one thread per entry adds the nine products to the vertices, as
//                  multiples of the vertex component's own quantum;
//   k_qbwd_write   the sums as floats.
// Listing every (link, vertex) term and ranking a vertex's list against itself (the
// earlier form) costs c^2 for c terms at a vertex: 8.9 ms on a body of 999 triangles whose
// vertices meet 3,600 links each, and 560 us on 111 K triangles with 1.72 M links, most of
// it FP64 terms.  Now 53 us on the first, bound by the shared-memory atomics and the gathers
// of the tile kernel.  A tile of 512 links keeps three CTAs an SM (29 KB, 80 registers).
#define QB_BLOCK 256
#define QB_PER 2
#define QB_TILE (QB_BLOCK * QB_PER)
#define QB_HASH (2 * QB_TILE)
#define QB_BITS 42  // a term is less than 2^QB_BITS quanta of its entry: two limbs of 21 bits
#define QB_NONE (-(1 << 30))
#define QB_NAN 1u
#define QB_PINF 2u
#define QB_NINF 4u

// S_j = m[j] 2^e[j] of one triangle over one tile; bits 3j .. 3j + 2 of `flag` hold
// QB_NAN, QB_PINF and QB_NINF if a term was not finite.
struct __align__(16) QbEntry {
    int tri;
    uint32_t flag;
    int e[3];
    int pad;
    long long m[3];
};

__device__ __forceinline__ float exp2i(int e) { return __int_as_float((127 + e) << 23); }  // e in [-126, 127]

// v 2^-k as a pair (|v| < 2^62)
__device__ __forceinline__ F2 f2_of_ll(long long v, float scale)
{
    const float h = (float)v;
    return {h * scale, (float)(v - (long long)h) * scale};
}

__device__ __forceinline__ void tri_normal(const int4 &A, const int4 &B, const int4 &C, long long n[3])
{
    const int ux = B.x - A.x, uy = B.y - A.y, uz = B.z - A.z, vx = C.x - A.x, vy = C.y - A.y, vz = C.z - A.z;
    n[0] = (long long)uy * vz - (long long)uz * vy;
    n[1] = (long long)uz * vx - (long long)ux * vz;
    n[2] = (long long)ux * vy - (long long)uy * vx;
}

// a . (b x c) for a lattice direction c: |b x c| < 2^27, |a . (b x c)| < 2^55
__device__ __forceinline__ long long lat_det(const int a[3], const int b[3], int cx, int cy, int cz)
{
    return (long long)a[0] * (b[1] * cz - b[2] * cy) + (long long)a[1] * (b[2] * cx - b[0] * cz) +
           (long long)a[2] * (b[0] * cy - b[1] * cx);
}

// The three terms of one link in FP64 with the hit point taken at the given q, for a q
// that is not the table's value of the crossing, a line parallel to its triangle, and a gq that is no
// normal number; non-finite terms come back as flags.
__device__ __noinline__ uint32_t qb_terms_wide(const int a[3], const int b[3], const int c3[3], const long long n[3],
                                               int cx, int cy, int cz, double s_, double f, F2 t[3], int &ex)
{
    const double bx = (double)b[0] - a[0], by = (double)b[1] - a[1], bz = (double)b[2] - a[2];
    const double qx = (double)c3[0] - a[0], qy = (double)c3[1] - a[1], qz = (double)c3[2] - a[2];
    const double xx = s_ * cx - a[0], xy = s_ * cy - a[1], xz = s_ * cz - a[2];
    const double nx = (double)n[0], ny = (double)n[1], nz = (double)n[2];
    const double nn = nx * nx + ny * ny + nz * nz;
    // X = lB B' + lC C':  X x C' = lB n,  B' x X = lC n
    const double lB = (nx * (xy * qz - xz * qy) + ny * (xz * qx - xx * qz) + nz * (xx * qy - xy * qx)) / nn;
    const double lC = (nx * (by * xz - bz * xy) + ny * (bz * xx - bx * xz) + nz * (bx * xy - by * xx)) / nn;
    f /= nx * cx + ny * cy + nz * cz;
    const double w[3] = {f * (1.0 - lB - lC), f * lB, f * lC};
    uint32_t flag = 0;
    ex = QB_NONE;
    for (int j = 0; j < 3; ++j) {
        if (isnan(w[j])) flag |= QB_NAN << (3 * j);
        else if (isinf(w[j])) flag |= (w[j] > 0 ? QB_PINF : QB_NINF) << (3 * j);
        else if (w[j] != 0.0) ex = max(ex, ilogb(w[j]));
    }
    for (int j = 0; j < 3; ++j) {
        t[j] = {0.0f, 0.0f};
        if (!isfinite(w[j]) || w[j] == 0.0) continue;
        const double m = scalbn(w[j], -ex);
        if (fabs(m) < 0x1p-100) continue;  // its scale would leave the float range
        t[j].h = (float)m;
        t[j].l = (float)(m - (double)t[j].h);
    }
    return flag;
}

__global__ void __launch_bounds__(QB_BLOCK) k_qbwd_tile(const uint64_t *__restrict__ key, LevelGeom g, int r_o,
                                                         const int32_t *__restrict__ cell, const uint8_t *__restrict__ dir,
                                                         const float *__restrict__ q, const int32_t *__restrict__ tri,
                                                         const float *__restrict__ gq, int64_t n,
                                                         const int4 *__restrict__ rec, int64_t T, int64_t nblk,
                                                         int64_t m3, QbEntry *__restrict__ ent, int *__restrict__ tile_n,
                                                         int *__restrict__ vexp, uint32_t *__restrict__ vflag, int *st)
{
    __shared__ int s_key[QB_HASH];                     // triangle of a hash slot (-1: free)
    __shared__ uint16_t s_idx[QB_HASH];                // its entry
    __shared__ int s_tri[QB_TILE], s_emax[3][QB_TILE];
    __shared__ int s_hi[3][QB_TILE], s_lo[3][QB_TILE];
    __shared__ uint32_t s_flag[QB_TILE];
    __shared__ int s_n;
    for (int i = threadIdx.x; i < QB_HASH; i += QB_BLOCK) s_key[i] = -1;
    for (int i = threadIdx.x; i < QB_TILE; i += QB_BLOCK) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            s_emax[j][i] = QB_NONE;
            s_hi[j][i] = s_lo[j][i] = 0;
        }
        s_flag[i] = 0;
    }
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int64_t k0 = (int64_t)blockIdx.x * QB_TILE;
    F2 t[QB_PER][3];
    int ea[QB_PER], slot[QB_PER];
    uint32_t flag[QB_PER];
#pragma unroll
    for (int u = 0; u < QB_PER; ++u) {
        const int64_t k = k0 + u * QB_BLOCK + threadIdx.x;
        slot[u] = -1;
        flag[u] = 0;
        ea[u] = 0;
        if (k >= n) continue;
        const int64_t tr = tri[k];
        if (tr < 0 || tr >= T) {
            emb_set_status(st, EMB_ERR_BAD_INPUT);
            continue;
        }
        // the triangle's slot: at most QB_TILE of the QB_HASH slots are taken
        int s = (int)((uint32_t)tr * 2654435761u >> 16) & (QB_HASH - 1);
        for (;;) {
            int have = *(volatile int *)&s_key[s];
            if (have == -1) {
                have = atomicCAS(&s_key[s], -1, (int)tr);
                if (have == -1) {
                    const int e = atomicAdd(&s_n, 1);
                    s_idx[s] = (uint16_t)e;
                    s_tri[e] = (int)tr;
                    have = (int)tr;
                }
            }
            if (have == (int)tr) break;
            s = (s + 1) & (QB_HASH - 1);
        }
        slot[u] = s;
        const int4 A = rec[3 * tr], B = rec[3 * tr + 1], C = rec[3 * tr + 2];
        const int64_t c = cell[k];
        if (!emb_ck((uint64_t)(c >> 6), (uint64_t)nblk, st)) {
            slot[u] = -1;
            continue;
        }
        const uint64_t bk = key[c >> 6];
        const int tc = (int)(c & 63), half = (int)g.half;
        const int px = (2 * (4 * (int)(bk & EMB_KEY_MASK) + (tc & 3)) + 1) * half;
        const int py = (2 * (4 * (int)((bk >> EMB_KEY_BITS) & EMB_KEY_MASK) + ((tc >> 2) & 3)) + 1) * half;
        const int pz = (2 * (4 * (int)(bk >> (2 * EMB_KEY_BITS)) + (tc >> 4)) + 1) * half;
        int cx, cy, cz;
        emb_dir(dir[k], cx, cy, cz);
        const int a[3] = {A.x - px, A.y - py, A.z - pz}, b[3] = {B.x - px, B.y - py, B.z - pz},
                  d[3] = {C.x - px, C.y - py, C.z - pz};
        const long long V[3] = {lat_det(b, d, cx, cy, cz), lat_det(d, a, cx, cy, cz), lat_det(a, b, cx, cy, cz)};
        const long long nc = V[0] + V[1] + V[2];  // c . n
        long long nn[3];
        tri_normal(A, B, C, nn);
        const float qk = q[k], gk = gq[k];
        // the crossing of the link's line with the plane, D / (h c.n) in steps of the link,
        // rounded as the link table's q is: there the weights are those of the crossing itself,
        // any other q (one ulp off, too) takes the general path with the hit point at that q
        const i128 D = mul128(nn[0], a[0]) + mul128(nn[1], a[1]) + mul128(nn[2], a[2]);
        const long long M = nc < 0 ? -nc : nc;
        const float Nf = D < 0 ? -i128_to_float(-D) : i128_to_float(D);
        const uint32_t ge = (__float_as_uint(gk) >> 23) & 255u;
        const bool usual = M != 0 && qk == __fdiv_rn(nc < 0 ? -Nf : Nf, (float)M * (float)g.h) &&
                           (gk == 0.0f || ge - 1u < 254u);
        if (usual) {
            const int kb = 63 - __clzll(M);
            const float sc = exp2i(-kb);
            const F2 m = f2_of_ll(M, sc);
            // 1 / m to second order, squared; times the mantissa of gq and r_o
            const float r1 = __frcp_rn(m.h);
            const F2 r = f2_norm(r1, r1 * __fadd_rn(__fmaf_rn(-r1, m.h, 1.0f), -r1 * m.l));
            const float gm = gk == 0.0f ? 0.0f : __uint_as_float((__float_as_uint(gk) & 0x807FFFFFu) | 0x3F800000u);
            const F2 w = f2_mul(two_prod(gm, (float)r_o), f2_mul(r, r));
#pragma unroll
            for (int j = 0; j < 3; ++j) t[u][j] = f2_mul(f2_of_ll(V[j], sc), w);
            ea[u] = (int)ge - 127 + (20 - g.lh) - kb;
        } else {
            flag[u] = qb_terms_wide(a, b, d, nn, cx, cy, cz, (double)qk * (double)g.h,
                                    (double)gk * (1048576.0 * (double)r_o) / (double)g.h, t[u], ea[u]);
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < QB_PER; ++u) {
        if (slot[u] < 0) continue;
        const int e = s_idx[slot[u]];
        slot[u] = e;
#pragma unroll
        for (int j = 0; j < 3; ++j)
            if (t[u][j].h != 0.0f)
                atomicMax(&s_emax[j][e], (int)((__float_as_uint(t[u][j].h) >> 23) & 255u) - 127 + ea[u]);
        if (flag[u]) atomicOr(&s_flag[e], flag[u]);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < QB_PER; ++u) {
        if (slot[u] < 0) continue;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // |term| 2^ea < 2^(emax + 1): below 2^21 in units of 2^(emax + 1 - 21), the high limb
            const int sh = ea[u] - s_emax[j][slot[u]] + QB_BITS / 2 - 1;
            if (t[u][j].h == 0.0f || sh < -100) continue;
            const float f = exp2i(sh), x = t[u][j].h * f, hi = floorf(x);
            const int lo = __float2int_rn(__fmaf_rn(t[u][j].l, f, x - hi) * (float)(1 << (QB_BITS / 2)));
            atomicAdd(&s_hi[j][slot[u]], (int)hi);
            atomicAdd(&s_lo[j][slot[u]], lo);
        }
    }
    __syncthreads();
    const int cnt = s_n;
    for (int i = threadIdx.x; i < cnt; i += QB_BLOCK) {
        QbEntry E;
        E.tri = s_tri[i];
        E.flag = s_flag[i];
        E.pad = 0;
        const int4 A = rec[3 * (int64_t)E.tri], B = rec[3 * (int64_t)E.tri + 1], C = rec[3 * (int64_t)E.tri + 2];
        const int vid[3] = {A.w, B.w, C.w};
        long long nn[3];
        tri_normal(A, B, C, nn);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            E.m[j] = ((long long)s_hi[j][i] << (QB_BITS / 2)) + s_lo[j][i];
            E.e[j] = s_emax[j][i] + 1 - QB_BITS;
            const uint32_t fl = (E.flag >> (3 * j)) & 7u;
            if (E.m[j] == 0 && !fl) continue;
            const int mb = 64 - __clzll(E.m[j] < 0 ? -E.m[j] : E.m[j]);
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                const int64_t at = 3 * (int64_t)vid[j] + x;
                if (!emb_ck((uint64_t)at, (uint64_t)m3, st)) continue;
                if (E.m[j] != 0 && nn[x] != 0)
                    atomicMax(vexp + at, E.e[j] + mb + 64 - __clzll(nn[x] < 0 ? -nn[x] : nn[x]));
                // an infinite term times a component of n: its sign, or NaN where that is 0
                if (fl)
                    atomicOr(vflag + at, nn[x] == 0 ? QB_NAN
                                                    : (nn[x] > 0 ? fl : (fl & QB_NAN) | ((fl & QB_PINF) << 1) | ((fl & QB_NINF) >> 1)));
            }
        }
        ent[k0 + i] = E;
    }
    if (threadIdx.x == 0) tile_n[blockIdx.x] = cnt;
}

// A vertex component's quantum is 2^(vexp - qbits): 3n terms of less than 2^vexp each stay
// below 2^63 in it.
__global__ void __launch_bounds__(QB_BLOCK) k_qbwd_scatter(const QbEntry *__restrict__ ent, const int *__restrict__ tile_n,
                                                            const int4 *__restrict__ rec, const int *__restrict__ vexp,
                                                            int qbits, int64_t m3,
                                                            unsigned long long *__restrict__ vacc, int *st)
{
    const int cnt = tile_n[blockIdx.x];
    for (int i = threadIdx.x; i < cnt; i += QB_BLOCK) {
        const QbEntry E = ent[(int64_t)blockIdx.x * QB_TILE + i];
        const int4 A = rec[3 * (int64_t)E.tri], B = rec[3 * (int64_t)E.tri + 1], C = rec[3 * (int64_t)E.tri + 2];
        const int vid[3] = {A.w, B.w, C.w};
        long long nn[3];
        tri_normal(A, B, C, nn);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
            for (int x = 0; x < 3; ++x) {
                if (E.m[j] == 0 || nn[x] == 0) continue;
                const int64_t at = 3 * (int64_t)vid[j] + x;
                if (!emb_ck((uint64_t)at, (uint64_t)m3, st)) continue;
                const int sh = vexp[at] - qbits - E.e[j];  // quanta of E.e per quantum of the vertex, log2
                const i128 P = mul128(E.m[j], nn[x]);
                if (sh > 120) continue;
                const long long v = sh > 0 ? (long long)((P + ((i128)1 << (sh - 1))) >> sh) : (long long)(P << -sh);
                if (v) atomicAdd(vacc + at, (unsigned long long)v);
            }
        }
    }
}

__global__ void k_qbwd_write(const int *__restrict__ vexp, const uint32_t *__restrict__ vflag,
                             const unsigned long long *__restrict__ vacc, int64_t m, int qbits, float *__restrict__ gv)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const long long v = (long long)vacc[i];
    const uint32_t fl = vflag[i];
    float r = 0.0f;
    if (v) r = (float)scalbn((double)v, vexp[i] - qbits);
    if (fl) r = fl == QB_PINF ? INFINITY : (fl == QB_NINF ? -INFINITY : NAN);
    gv[i] = r;
}

extern "C" emb_status emb_cutlinks_backward(emb_mesh m, emb_forest f, const int32_t *d_cell, const uint8_t *d_dir,
                                            const float *d_q, const int32_t *d_tri, int64_t n, const float *d_gq,
                                            float *d_gverts, void *stream)
{
    if (!m || !f || n < 0 || !d_gverts) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    if (m->R != f->R || f->top != f->max_level) return EMB_ERR_STATE;
    if (n > 0 && (!d_cell || !d_dir || !d_q || !d_tri || !d_gq)) return EMB_ERR_BAD_INPUT;
    if (3 * n >= (1ll << 32)) return EMB_ERR_CAPACITY;
    cudaStream_t s = emb_stream(stream);
    int *st = emb_status_word();
    if (!st) return EMB_ERR_CUDA;
    const EmbLevel &lv = f->lv[f->max_level];
    LevelGeom g = level_geom(f, f->max_level);
    // one scratch allocation: vertex sums and flags (3V each, zeroed), their exponents (3V,
    // 0x80 bytes), the entries (QB_TILE a tile) and their counts
    const int64_t nt = (n + QB_TILE - 1) / QB_TILE, m3 = 3 * m->V;
    const size_t a_acc = (size_t)m3 * sizeof(uint64_t), a_v = (size_t)m3 * sizeof(uint32_t),
                 a_tn = (size_t)(nt + 1) * sizeof(int), a_ent = (size_t)(nt * QB_TILE) * sizeof(QbEntry);
    auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
    char *scratch = nullptr;
    EMB_CUDA_TRY(emb_malloc_async((void **)&scratch, up(a_acc) + 2 * up(a_v) + up(a_tn) + a_ent, s));
    unsigned long long *vacc = (unsigned long long *)scratch;
    uint32_t *vflag = (uint32_t *)(scratch + up(a_acc));
    int *vexp = (int *)(scratch + up(a_acc) + up(a_v));
    int *tile_n = (int *)(scratch + up(a_acc) + 2 * up(a_v));
    QbEntry *ent = (QbEntry *)(scratch + up(a_acc) + 2 * up(a_v) + up(a_tn));
    int qbits = 61;
    while (((3 * n) >> (61 - qbits)) != 0) --qbits;
    EMB_CUDA_TRY(cudaMemsetAsync(vacc, 0, up(a_acc) + a_v, s));
    EMB_CUDA_TRY(cudaMemsetAsync(vexp, 0x80, a_v, s));
    if (n > 0) {
        EMB_LAUNCH((k_qbwd_tile), (int)nt, QB_BLOCK, 0, s)(lv.key, g, m->r_o, d_cell, d_dir, d_q, d_tri, d_gq, n, m->rec,
                                                           m->T, lv.n, m3, ent, tile_n, vexp, vflag, st);
        EMB_LAUNCH((k_qbwd_scatter), (int)nt, QB_BLOCK, 0, s)(ent, tile_n, m->rec, vexp, qbits, m3, vacc, st);
    }
    EMB_LAUNCH((k_qbwd_write), emb_grid(m3, 256), 256, 0, s)(vexp, vflag, vacc, m3, qbits, d_gverts);
    EMB_CUDA_TRY(cudaGetLastError());
    EMB_CUDA_TRY(cudaFreeAsync(scratch, s));
    return EMB_OK;
}
