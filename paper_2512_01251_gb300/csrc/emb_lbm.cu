// One lattice-Boltzmann step on the finest level of a forest: the consumer the
// cut-link table is built for (Sec. 2.2 cites interpolated bounce-back with the link
// fractions q and the momentum exchange; Sec. 3.4 lays the table out for lookup during
// computation).  The paper prints neither the collision model nor Bouzidi's rule; the
// textbook BGK collision with the D3Q19 / D3Q27 weights and the linear Bouzidi rule of
// emb_mex_force are used.  Populations are SoA, pop[i * stride + cell], cell = block *
// 64 + x + 4 y + 16 z on the finest level.  The step is
//   pull streaming  f_i(x) = f*_i(x - c_i) when x - c_i is a fluid cell of the level, f*_i(x)
//                   when its block is missing (zero gradient at the edge of the level: the
//                   coupling to coarser levels is out of scope), left open when solid;
//   Bouzidi         per cut link (x, d, q): the population entering x against c_d, from
//                   f*_d(x), f*_d(x - c_d) and f*_-d(x) by the linear rule;
//   collision       BGK f* = f - omega (f - f_eq(rho, u)) at fluid cells, 0 at solid ones.
// The whole step runs as k_lbm_bouzidi and then k_lbm_step, which streams and collides in one
// pass over the cells.  Its parts by themselves (the phases of emb_lbm_step, so that the cost
// of the boundary treatment can be timed against the rest) are k_lbm_stream, k_lbm_bouzidi and
// k_lbm_collide.
#include "emb_internal.cuh"

// direction index of a block offset (ox, oy, oz) in {-1,0,1}^3, code (ox+1) + 3(oy+1) + 9(oz+1)
__constant__ int8_t c_lbm_dir_of_offset[27] = {20, 16, 26, 12, 6, 13, 24, 17, 21, 8, 4, 9, 2, 0,
                                               1,  10, 3,  7,  22, 18, 23, 14, 5, 11, 25, 15, 19};

// Cell x - c of cell (b, t): its id, or -1 if it is solid, -2 if its block is missing.
__device__ __forceinline__ int64_t lbm_source(int64_t b, int t, int cx, int cy, int cz, const int32_t *__restrict__ nbr,
                                              const uint64_t *__restrict__ mask)
{
    const int x = (t & 3) - cx, y = ((t >> 2) & 3) - cy, z = (t >> 4) - cz;
    const int ox = x < 0 ? -1 : (x > 3 ? 1 : 0), oy = y < 0 ? -1 : (y > 3 ? 1 : 0), oz = z < 0 ? -1 : (z > 3 ? 1 : 0);
    int64_t nb = b;
    if (ox | oy | oz) {
        nb = nbr[b * 26 + c_lbm_dir_of_offset[(ox + 1) + 3 * (oy + 1) + 9 * (oz + 1)] - 1];
        if (nb < 0) return -2;
    }
    const int lt = (x & 3) + 4 * (y & 3) + 16 * (z & 3);
    if ((mask[nb] >> lt) & 1ull) return -1;
    return nb * 64 + lt;
}

template <int Q>
__global__ void k_lbm_stream(const float *__restrict__ pop, float *__restrict__ pre, int64_t stride, int64_t ncell,
                             const int32_t *__restrict__ nbr, const uint64_t *__restrict__ mask)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= ncell) return;
    const int64_t b = x >> 6;
    const int t = (int)(x & 63);
    const bool solid = (mask[b] >> t) & 1ull;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        float v = 0.0f;
        if (!solid) {
            int cx, cy, cz;
            emb_dir(i, cx, cy, cz);
            const int64_t s = lbm_source(b, t, cx, cy, cz, nbr, mask);
            v = s >= 0 ? pop[(int64_t)i * stride + s] : (s == -2 ? pop[(int64_t)i * stride + x] : 0.0f);
        }
        pre[(int64_t)i * stride + x] = v;
    }
}

__global__ void k_lbm_bouzidi(const int32_t *__restrict__ cell, const uint8_t *__restrict__ dir,
                              const float *__restrict__ q, int64_t n, const float *__restrict__ pop,
                              float *__restrict__ pre, int64_t stride, int64_t ncell, int lattice,
                              const int32_t *__restrict__ nbr, const uint64_t *__restrict__ mask, uint32_t *bits, int *st)
{
    const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n) return;
    const int64_t c = cell[k];
    const int d = dir[k];
    if (c < 0 || c >= ncell || d < 1 || d >= lattice) {
        emb_set_status(st, EMB_ERR_BAD_INPUT);  // not a link of this level and lattice
        return;
    }
    const int o = (d & 1) ? d + 1 : d - 1;
    int cx, cy, cz;
    emb_dir(d, cx, cy, cz);
    const float f_d = pop[(int64_t)d * stride + c];
    const float qq = q[k];
    float g;
    if (qq < 0.5f) {
        const int64_t p = lbm_source(c >> 6, (int)(c & 63), cx, cy, cz, nbr, mask);  // x - c_d
        g = p >= 0 ? 2.0f * qq * f_d + (1.0f - 2.0f * qq) * pop[(int64_t)d * stride + p] : f_d;
    } else {
        g = f_d / (2.0f * qq) + (2.0f * qq - 1.0f) / (2.0f * qq) * pop[(int64_t)o * stride + c];
    }
    pre[(int64_t)o * stride + c] = g;
    if (bits) atomicOr(bits + c, 1u << o);
}

// BGK relaxation of the populations f[0, Q) of a fluid cell, in place.
template <int Q>
__device__ __forceinline__ void lbm_bgk(float (&f)[Q], float omega)
{
    float rho = 0.0f, jx = 0.0f, jy = 0.0f, jz = 0.0f;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        int cx, cy, cz;
        emb_dir(i, cx, cy, cz);
        rho += f[i];
        jx += cx * f[i];
        jy += cy * f[i];
        jz += cz * f[i];
    }
    const float inv = rho != 0.0f ? 1.0f / rho : 0.0f;
    const float ux = jx * inv, uy = jy * inv, uz = jz * inv;
    const float usq = ux * ux + uy * uy + uz * uz;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        int cx, cy, cz;
        emb_dir(i, cx, cy, cz);
        const int kind = cx * cx + cy * cy + cz * cz;  // 0 rest, 1 axis, 2 edge, 3 corner
        const float w = Q == 19 ? (kind == 0 ? 1.0f / 3 : (kind == 1 ? 1.0f / 18 : 1.0f / 36))
                                : (kind == 0 ? 8.0f / 27 : (kind == 1 ? 2.0f / 27 : (kind == 2 ? 1.0f / 54 : 1.0f / 216)));
        const float cu = cx * ux + cy * uy + cz * uz;
        const float feq = w * rho * (1.0f + 3.0f * cu + 4.5f * cu * cu - 1.5f * usq);
        f[i] = f[i] - omega * (f[i] - feq);
    }
}

template <int Q>
__global__ void k_lbm_collide(const float *__restrict__ pre, float *__restrict__ out, int64_t stride, int64_t ncell,
                              const uint64_t *__restrict__ mask, float omega)
{
    const int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= ncell) return;
    if ((mask[x >> 6] >> (x & 63)) & 1ull) {
#pragma unroll
        for (int i = 0; i < Q; ++i) out[(int64_t)i * stride + x] = 0.0f;
        return;
    }
    float f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) f[i] = pre[(int64_t)i * stride + x];
    lbm_bgk<Q>(f, omega);
#pragma unroll
    for (int i = 0; i < Q; ++i) out[(int64_t)i * stride + x] = f[i];
}

// The whole step in one pass over the cells: the populations are pulled, relaxed in
// registers and stored, so that each is read once and written once (streaming into
// `pre` and colliding from it moves them twice).  k_lbm_bouzidi has run before and left
// the population entering link cell c against c_d in pre[i * stride + c] and bit i in
// word c of `bits` (row 0 of pre, which no link direction uses); bits is NULL without
// links.  A CTA holds LBM_BLOCKS blocks, one thread a cell; their 27 neighbour ids and
// masks are staged in shared memory, so the Q pulls of a cell wait on nothing but each
// other.  Bound by HBM (8 Q bytes a cell) and the loads in flight: two blocks a CTA, ten CTAs
// an SM for D3Q19 (48 registers) and nine for D3Q27 (56), the best of 1 to 8 blocks and all
// register limits (6.2M cells, step with the boundary pass: 211 and 290 us; four blocks
// and no limit 278 and 336; as three passes 400 us for D3Q19).
#define LBM_BLOCKS 2
template <int Q>
__global__ void __launch_bounds__(64 * LBM_BLOCKS, Q == 19 ? 10 : 9) k_lbm_step(const float *__restrict__ pop, const float *__restrict__ pre,
                                                              const uint32_t *__restrict__ bits, float *__restrict__ out,
                                                              int64_t stride, int64_t nblk,
                                                              const int32_t *__restrict__ nbr,
                                                              const uint64_t *__restrict__ mask, float omega, int *st)
{
    __shared__ uint64_t s_mask[LBM_BLOCKS * 27];
    __shared__ int32_t s_id[LBM_BLOCKS * 27];
    const int64_t b0 = (int64_t)blockIdx.x * LBM_BLOCKS;
    if (threadIdx.x < LBM_BLOCKS * 27) {
        const int j = threadIdx.x / 27, code = threadIdx.x - 27 * j;
        int32_t id = -1;
        if (b0 + j < nblk) id = code == 13 ? (int32_t)(b0 + j) : nbr[(b0 + j) * 26 + c_lbm_dir_of_offset[code] - 1];
        if (id >= 0 && !emb_ck((uint64_t)id, (uint64_t)nblk, st)) id = -1;
        s_id[threadIdx.x] = id;
        s_mask[threadIdx.x] = id >= 0 ? mask[id] : 0ull;
    }
    __syncthreads();
    const int j = threadIdx.x >> 6, t = threadIdx.x & 63;
    const int64_t b = b0 + j;
    if (b >= nblk) return;
    const int64_t c = b * 64 + t;
    if ((s_mask[27 * j + 13] >> t) & 1ull) {
#pragma unroll
        for (int i = 0; i < Q; ++i) out[(int64_t)i * stride + c] = 0.0f;
        return;
    }
    const uint32_t lk = bits ? bits[c] : 0u;
    const int x = t & 3, y = (t >> 2) & 3, z = t >> 4;
    float f[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        int cx, cy, cz;
        emb_dir(i, cx, cy, cz);
        const int sx = x - cx, sy = y - cy, sz = z - cz;  // in [-1, 4]
        const int code = 27 * j + 13 + (cx ? sx >> 2 : 0) + (cy ? 3 * (sy >> 2) : 0) + (cz ? 9 * (sz >> 2) : 0);
        const int32_t id = s_id[code];
        const int lt = (sx & 3) + 4 * (sy & 3) + 16 * (sz & 3);
        const bool linked = (lk >> i) & 1u, solid = (s_mask[code] >> lt) & 1ull;
        const float *src = linked ? pre + c : pop + (id >= 0 ? (int64_t)id * 64 + lt : c);
        f[i] = linked || !solid ? src[(int64_t)i * stride] : 0.0f;
    }
    lbm_bgk<Q>(f, omega);
#pragma unroll
    for (int i = 0; i < Q; ++i) out[(int64_t)i * stride + c] = f[i];
}

extern "C" emb_status emb_lbm_step(emb_forest f, int32_t lattice, const int32_t *d_cell, const uint8_t *d_dir,
                                   const float *d_q, int64_t n_links, float omega, const float *d_pop, float *d_pre,
                                   float *d_pop_out, int64_t pop_stride, int32_t phases, void *stream)
{
    if (!f || (lattice != 19 && lattice != 27) || n_links < 0 || !(omega >= 0.0f && omega < 2.0f) || phases < 1 ||
        phases > 7)
        return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    const int L = f->max_level;
    if (f->top != L || !f->lv[L].mask_valid) return EMB_ERR_STATE;
    EmbLevel &lv = f->lv[L];
    const int64_t ncell = lv.n * 64;
    if (pop_stride < ncell) return EMB_ERR_BAD_INPUT;
    if (ncell == 0) return EMB_OK;
    if (!d_pop || !d_pre || !d_pop_out || d_pop == d_pre || d_pre == d_pop_out || d_pop == d_pop_out)
        return EMB_ERR_BAD_INPUT;
    if (n_links > 0 && (!d_cell || !d_dir || !d_q)) return EMB_ERR_BAD_INPUT;
    cudaStream_t s = emb_stream(stream);
    emb_status rc = emb_build_neighbors(lv, s);
    if (rc != EMB_OK) return rc;
    int *st = emb_status_word();
    if (!st) return EMB_ERR_CUDA;
    if (phases == 7) {
        // the boundary populations first, then streaming and collision in one pass
        uint32_t *bits = n_links > 0 ? (uint32_t *)d_pre : nullptr;
        if (bits) {
            EMB_CUDA_TRY(cudaMemsetAsync(bits, 0, ncell * sizeof(uint32_t), s));
            EMB_LAUNCH((k_lbm_bouzidi), emb_grid(n_links, 256), 256, 0, s)(d_cell, d_dir, d_q, n_links, d_pop, d_pre,
                                                                           pop_stride, ncell, lattice, lv.nbr, lv.mask,
                                                                           bits, st);
        }
        const int grid = emb_grid(lv.n, LBM_BLOCKS);
        if (lattice == 19)
            EMB_LAUNCH((k_lbm_step<19>), grid, 64 * LBM_BLOCKS, 0, s)(d_pop, d_pre, bits, d_pop_out, pop_stride, lv.n,
                                                                      lv.nbr, lv.mask, omega, st);
        else
            EMB_LAUNCH((k_lbm_step<27>), grid, 64 * LBM_BLOCKS, 0, s)(d_pop, d_pre, bits, d_pop_out, pop_stride, lv.n,
                                                                      lv.nbr, lv.mask, omega, st);
        EMB_CUDA_TRY(cudaGetLastError());
        return EMB_OK;
    }
    const int grid = emb_grid(ncell, 256);
    if (phases & 1) {
        if (lattice == 19) EMB_LAUNCH((k_lbm_stream<19>), grid, 256, 0, s)(d_pop, d_pre, pop_stride, ncell, lv.nbr, lv.mask);
        else EMB_LAUNCH((k_lbm_stream<27>), grid, 256, 0, s)(d_pop, d_pre, pop_stride, ncell, lv.nbr, lv.mask);
    }
    if ((phases & 2) && n_links > 0)
        EMB_LAUNCH((k_lbm_bouzidi), emb_grid(n_links, 256), 256, 0, s)(d_cell, d_dir, d_q, n_links, d_pop, d_pre, pop_stride,
                                                                       ncell, lattice, lv.nbr, lv.mask, nullptr, st);
    if (phases & 4) {
        if (lattice == 19)
            EMB_LAUNCH((k_lbm_collide<19>), grid, 256, 0, s)(d_pre, d_pop_out, pop_stride, ncell, lv.mask, omega);
        else EMB_LAUNCH((k_lbm_collide<27>), grid, 256, 0, s)(d_pre, d_pop_out, pop_stride, ncell, lv.mask, omega);
    }
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}
