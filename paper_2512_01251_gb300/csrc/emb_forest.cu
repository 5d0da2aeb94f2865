// Forest harness (Sec. 3.2): root grid, top-down creation of children from
// refinement flags, per-level coordinate hash and neighbour links.
//
// Blocks of a level are kept in ascending key order, key = (bz, by, bx), so
// every x-row of blocks is contiguous and ordered along +x (the order the
// voxelizer's row scan needs).  Children are written straight into that order:
// with parents sorted, the rank of a child follows from exclusive counts of
// flagged parents before its parent's plane (bz), row (bz, by) and position.
#include <stdlib.h>

#include "emb_internal.cuh"

// The root level in one launch: every position holds a block, so the bitmap is full and
// the prefix of word w is 64 w.
__global__ void k_root(int64_t R, uint64_t *__restrict__ key, uint64_t *__restrict__ bits, uint32_t *__restrict__ wpre,
                       int64_t nw)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = R * R * R;
    if (i < n) key[i] = emb_key(i % R, (i / R) % R, i / (R * R));
    if (i < nw) bits[i] = n - 64 * i >= 64 ? ~0ull : (1ull << (n - 64 * i)) - 1ull;
    if (i <= nw) wpre[i] = (uint32_t)(64 * i < n ? 64 * i : n);
}

// Blocks of a level at dense positions below lin (at most nb^3).
__device__ __forceinline__ int64_t rank_below(const uint64_t *__restrict__ bits, const uint32_t *__restrict__ wpre,
                                              int64_t lin)
{
    const int sh = (int)(lin & 63);
    const int64_t r = wpre[lin >> 6];
    return sh ? r + __popcll(bits[lin >> 6] & ((1ull << sh) - 1ull)) : r;
}

// Keys past the count in a planned replay that flagged fewer blocks than its buffers hold
// (a replay with headroom, or one whose counts left its plan): a key above every real
// key, so that the level's keys stay sorted for the binary searches over all Cn of
// them; its coordinates (2^21 - 1 on every axis) fail the range checks of the passes
// that decode keys, and the passes over blocks stop at the device count where there
// is one.
#define EMB_KEY_TAIL 0x7FFFFFFFFFFFFFFFull

// The children of the flagged blocks, in order, and their bits in the child level's bitmap
// (cbits, zeroed before; NULL for a level with a hash).  The parents before a block's row
// and plane are counted with the parent's rank bitmap (two loads each) where it has one,
// else by binary search.  A planned replay also fills the keys past the count and stores
// the level's block count at d_n.  (With the bits, the tail and the count in launches of
// their own and the binary searches always: 12 us a level instead of 5.)
__global__ void k_make_children(const EmbLevel P, const uint8_t *__restrict__ flags, const uint32_t *__restrict__ rank,
                                uint64_t *__restrict__ ckey, int64_t Cn, unsigned long long *__restrict__ cbits,
                                bool planned, uint32_t *__restrict__ d_n, int *st)
{
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const uint64_t *__restrict__ key = P.key;
    const int64_t n = P.n, nb = P.nb_axis;
    if (planned) {
        const int64_t m = 8 * (int64_t)rank[n];
        for (int64_t i = m + p; i < Cn; i += (int64_t)gridDim.x * blockDim.x) ckey[i] = EMB_KEY_TAIL;
        if (p == 0 && d_n) {
            if (m > Cn) emb_set_status(st, EMB_ERR_CAPACITY);
            *d_n = (uint32_t)(m < Cn ? m : Cn);
        }
    }
    if (p >= n || !flags[p]) return;
    const uint64_t k = key[p];
    const int64_t bx = (int64_t)(k & EMB_KEY_MASK), by = (int64_t)((k >> EMB_KEY_BITS) & EMB_KEY_MASK),
                  bz = (int64_t)(k >> (2 * EMB_KEY_BITS));
    int64_t rl, rh, pll, plh;
    if (P.bits) {
        if (bx >= nb || by >= nb || bz >= nb) return;  // only a replay whose counts left its plan gets here
        const int64_t row = (bz * nb + by) * nb, plane = bz * nb * nb;
        rl = rank_below(P.bits, P.wpre, row);
        rh = rank_below(P.bits, P.wpre, row + nb);
        pll = rank_below(P.bits, P.wpre, plane);
        plh = rank_below(P.bits, P.wpre, plane + nb * nb);
        // entries of rank, which holds n + 1
        if (!emb_ck((uint64_t)rl, (uint64_t)n + 1, st) || !emb_ck((uint64_t)rh, (uint64_t)n + 1, st) ||
            !emb_ck((uint64_t)pll, (uint64_t)n + 1, st) || !emb_ck((uint64_t)plh, (uint64_t)n + 1, st))
            return;
    } else {
        const uint64_t row0 = k & ~EMB_KEY_MASK, row1 = row0 + (1ull << EMB_KEY_BITS);
        const uint64_t pl0 = k & ~((1ull << (2 * EMB_KEY_BITS)) - 1ull), pl1 = pl0 + (1ull << (2 * EMB_KEY_BITS));
        rl = lower_bound_u64(key, n, row0);
        rh = lower_bound_u64(key, n, row1);
        pll = lower_bound_u64(key, n, pl0);
        plh = lower_bound_u64(key, n, pl1);
    }
    const int64_t r_p = rank[p], r_row = rank[rl], F_row = (int64_t)rank[rh] - r_row;
    const int64_t r_pl = rank[pll], F_pl = (int64_t)rank[plh] - r_pl;
    for (int dz = 0; dz < 2; ++dz)
        for (int dy = 0; dy < 2; ++dy) {
            const int64_t pos = 8 * r_pl + dz * 4 * F_pl + 4 * (r_row - r_pl) + dy * 2 * F_row + 2 * (r_p - r_row);
            const int64_t cy = 2 * by + dy, cz = 2 * bz + dz;
            unsigned long long pair = 0;  // the two children along x: neighbours in a word, 2 bx is even
            for (int dx = 0; dx < 2; ++dx)
                if (pos + dx >= 0 && pos + dx < Cn) {
                    ckey[pos + dx] = emb_key(2 * bx + dx, cy, cz);
                    pair |= 1ull << dx;
                }
            if (cbits && pair) {
                const int64_t lin = (cz * (2 * nb) + cy) * (2 * nb) + 2 * bx;
                atomicOr(cbits + (lin >> 6), pair << (lin & 63));
            }
        }
}

__global__ void k_unpack_keys(const uint64_t *__restrict__ key, int64_t n, int32_t *__restrict__ out)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint64_t k = key[i];
    out[3 * i + 0] = (int32_t)(k & EMB_KEY_MASK);
    out[3 * i + 1] = (int32_t)((k >> EMB_KEY_BITS) & EMB_KEY_MASK);
    out[3 * i + 2] = (int32_t)(k >> (2 * EMB_KEY_BITS));
}

static void free_level(EmbLevel &lv)
{
    if (lv.key) cudaFree(lv.key);
    if (lv.hkey) cudaFree(lv.hkey);
    if (lv.hval) cudaFree(lv.hval);
    if (lv.mask) cudaFree(lv.mask);
    if (lv.nbr) cudaFree(lv.nbr);
    if (lv.bits) cudaFree(lv.bits);
    if (lv.wpre) cudaFree(lv.wpre);
    lv = EmbLevel();
}

extern "C" emb_status emb_forest_root(int32_t R, int32_t max_level, void *stream, emb_forest *out)
{
    if (!out || R < 1 || max_level < 0 || max_level >= EMB_MAX_LEVELS) return EMB_ERR_BAD_INPUT;
    *out = nullptr;
    int32_t r_o = R, k = 0;
    while ((r_o & 1) == 0) {
        r_o >>= 1;
        ++k;
    }
    if (k + max_level > 17 || ((int64_t)R << max_level) >= (1ll << EMB_KEY_BITS) || (int64_t)r_o * (1 << 20) >= (1ll << 25))
        return EMB_ERR_RANGE;
    if ((int64_t)R * R * R > 2147483647ll) return EMB_ERR_BAD_INPUT;
    cudaStream_t s = emb_stream(stream);
    emb_forest f = new emb_forest_s();
    f->R = R;
    f->r_o = r_o;
    f->k = k;
    f->max_level = max_level;
    f->top = 0;
    cudaGetDevice(&f->device);
    EmbLevel &lv = f->lv[0];
    lv.n = (int64_t)R * R * R;
    lv.nb_axis = R;
    const int64_t nw = emb_bitmap_words(R);
    if (emb_malloc_async(&lv.key, lv.n * sizeof(uint64_t), s) != cudaSuccess ||
        emb_malloc_async(&lv.bits, nw * sizeof(uint64_t), s) != cudaSuccess ||
        emb_malloc_async(&lv.wpre, (nw + 1) * sizeof(uint32_t), s) != cudaSuccess) {
        emb_forest_destroy(f);
        return EMB_ERR_CUDA;
    }
    const emb_status rc = emb_enq_root(lv, s);
    if (rc != EMB_OK) {
        emb_forest_destroy(f);
        return rc;
    }
    *out = f;
    return EMB_OK;
}

// Level arrays come from the stream-ordered pool of the calls that built them; the
// teardown synchronises the device once and returns them all.
extern "C" void emb_forest_destroy(emb_forest f)
{
    if (!f) return;
    cudaDeviceSynchronize();
    for (int L = 0; L < EMB_MAX_LEVELS; ++L) free_level(f->lv[L]);
    if (f->cand) cudaFree(f->cand);
    if (f->blk_off) cudaFree(f->blk_off);
    if (f->work) cudaFree(f->work);
    emb_readback_release(f->rb_slot);
    delete f;
}

// Refinement in two enqueue-only halves (buffers supplied by the caller):
//  (1) ranks of the flagged blocks of P: rank holds P.n + 1 uint32; the number of
//      flagged blocks F ends at rank[P.n]; tmp is scan scratch for P.n entries;
//  (2) level C: its first min(8 F, Cn) keys in (z, y, x) order and its index (rank bitmap,
//      or the hash over C.n keys where it has none); tmp is scan scratch for its bitmap.
//      `zeroed`: the caller has cleared the bitmap and tmp.  planned: see k_make_children.
emb_status emb_enq_flag_ranks(const EmbLevel &P, const uint8_t *d_flags, uint32_t *rank, uint64_t *tmp, bool zeroed,
                              cudaStream_t s, uint64_t expect)
{
    return emb_scan_flags(d_flags, rank, P.n, tmp, expect, zeroed, s);
}

emb_status emb_enq_child_level(const EmbLevel &P, const uint8_t *d_flags, const uint32_t *rank, EmbLevel &C, int64_t Cn,
                               bool planned, uint32_t *d_n, uint64_t *tmp, bool zeroed, cudaStream_t s)
{
    int *st = emb_status_word();
    if (!st) return EMB_ERR_CUDA;
    const int64_t nw = C.bits ? emb_bitmap_words(C.nb_axis) : 0;
    if (nw > 0 && !zeroed) EMB_CUDA_TRY(cudaMemsetAsync(C.bits, 0, nw * sizeof(uint64_t), s));
    if (P.n > 0 && (Cn > 0 || d_n))
        EMB_LAUNCH((k_make_children), emb_grid(P.n, 256), 256, 0, s)(P, d_flags, rank, C.key, Cn,
                                                                     (unsigned long long *)(nw > 0 ? C.bits : nullptr),
                                                                     planned, d_n, st);
    EMB_CUDA_TRY(cudaGetLastError());
    if (nw > 0) return emb_scan_popc(C.bits, C.wpre, nw, tmp, zeroed, s);
    return emb_enq_level_index(C, tmp, s);
}

emb_status emb_enq_root(EmbLevel &lv, cudaStream_t s)
{
    const int64_t R = lv.nb_axis, nw = emb_bitmap_words(R), n = R * R * R;
    EMB_LAUNCH((k_root), emb_grid(n > nw + 1 ? n : nw + 1, 256), 256, 0, s)(R, lv.key, lv.bits, lv.wpre, nw);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}

emb_status emb_forest_settle(emb_forest f)
{
    if (!f || f->n_pending < 0) return EMB_OK;
    EMB_CUDA_TRY(cudaEventSynchronize(f->rb_ev));
    f->lv[f->n_pending].n = 8 * (int64_t)(*(volatile uint32_t *)f->rb_h);
    f->n_pending = -1;
    return EMB_OK;
}

extern "C" emb_status emb_forest_refine(emb_forest f, int32_t level, const uint8_t *d_flags, void *stream)
{
    if (!f) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    if (level < 0 || level != f->top || level >= f->max_level) return EMB_ERR_STATE;
    if (!d_flags && f->lv[level].n > 0) return EMB_ERR_BAD_INPUT;
    cudaStream_t s = emb_stream(stream);
    EmbLevel &P = f->lv[level];
    EmbLevel &C = f->lv[level + 1];
    free_level(C);
    uint32_t *rank = nullptr;
    EMB_CUDA_TRY(emb_malloc_async(&rank, (P.n + 1) * sizeof(uint32_t), s));
    C.nb_axis = P.nb_axis * 2;
    const int64_t nw = emb_bitmap_words(C.nb_axis), sp = emb_scan_tmp_words(P.n);
    emb_status rc = EMB_OK;
    if (f->rb_slot < 0) f->rb_slot = emb_readback_acquire(&f->rb_h, &f->rb_ev);
    if (nw > 0 && f->rb_slot >= 0) {
        // The child level takes the rank bitmap: its keys (room for 8 per parent) and
        // index are built from the flagged count on the device while that count comes
        // back to the host, so the GPU is not left idle during the read-back.  The two
        // scans' states lie behind the bitmap, cleared with it.
        const int64_t cap = 8 * P.n, zw = nw + sp + emb_scan_tmp_words(nw);
        EMB_CUDA_TRY(emb_malloc_async(&C.bits, zw * sizeof(uint64_t), s));
        EMB_CUDA_TRY(emb_malloc_async(&C.wpre, (nw + 1) * sizeof(uint32_t), s));
        EMB_CUDA_TRY(emb_malloc_async(&C.key, (cap + 1) * sizeof(uint64_t), s));
        EMB_CUDA_TRY(cudaMemsetAsync(C.bits, 0, zw * sizeof(uint64_t), s));
        rc = emb_enq_flag_ranks(P, d_flags, rank, C.bits + nw, true, s);
        if (rc != EMB_OK) return rc;
        EMB_CUDA_TRY(cudaMemcpyAsync(f->rb_h, rank + P.n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
        EMB_CUDA_TRY(cudaEventRecord(f->rb_ev, s));
        rc = emb_enq_child_level(P, d_flags, rank, C, cap, false, nullptr, C.bits + nw + sp, true, s);
        EMB_CUDA_TRY(cudaFreeAsync(rank, s));
        if (rc != EMB_OK) return rc;
        // the count is stored when a call first needs it (emb_forest_settle): work that
        // does not need it, such as the next level's x-line filter, is queued first, so
        // that the GPU has it while the count travels
        C.n = 0;
        f->n_pending = level + 1;
    } else {
        uint64_t *tmp = nullptr;
        const int64_t sc = nw > 0 ? emb_scan_tmp_words(nw) : 1;
        EMB_CUDA_TRY(emb_malloc_async(&tmp, (sp > sc ? sp : sc) * sizeof(uint64_t), s));
        rc = emb_enq_flag_ranks(P, d_flags, rank, tmp, false, s);
        if (rc != EMB_OK) return rc;
        uint32_t F = 0;
        EMB_CUDA_TRY(cudaMemcpyAsync(&F, rank + P.n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
        EMB_CUDA_TRY(cudaStreamSynchronize(s));
        C.n = 8 * (int64_t)F;
        EMB_CUDA_TRY(emb_malloc_async(&C.key, (C.n + 1) * sizeof(uint64_t), s));
        if (nw > 0) {
            EMB_CUDA_TRY(emb_malloc_async(&C.bits, nw * sizeof(uint64_t), s));
            EMB_CUDA_TRY(emb_malloc_async(&C.wpre, (nw + 1) * sizeof(uint32_t), s));
        } else {
            C.hcap = emb_hash_capacity(C.n);
            EMB_CUDA_TRY(emb_malloc_async(&C.hkey, C.hcap * sizeof(uint64_t), s));
            EMB_CUDA_TRY(emb_malloc_async(&C.hval, C.hcap * sizeof(int32_t), s));
        }
        rc = emb_enq_child_level(P, d_flags, rank, C, C.n, false, nullptr, tmp, false, s);
        EMB_CUDA_TRY(cudaFreeAsync(rank, s));
        EMB_CUDA_TRY(cudaFreeAsync(tmp, s));
        if (rc != EMB_OK) return rc;
    }
    f->top = level + 1;
    // a new finest level invalidates cached link candidates
    if (f->cand) {
        cudaFreeAsync(f->cand, s);
        f->cand = nullptr;
    }
    if (f->blk_off) {
        cudaFreeAsync(f->blk_off, s);
        f->blk_off = nullptr;
    }
    if (f->work) {
        cudaFreeAsync(f->work, s);
        f->work = nullptr;
    }
    f->work_n = nullptr;
    f->n_links = -1;
    return EMB_OK;
}

extern "C" emb_status emb_forest_num_blocks(emb_forest f, int32_t level, int64_t *h_out)
{
    if (!f || !h_out || level < 0 || level >= EMB_MAX_LEVELS) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    *h_out = level <= f->top ? f->lv[level].n : 0;
    return EMB_OK;
}

extern "C" emb_status emb_forest_blocks(emb_forest f, int32_t level, int32_t *d_out, void *stream)
{
    EMB_SETTLE(f);
    if (!f || level < 0 || level > f->top) return EMB_ERR_STATE;
    const EmbLevel &lv = f->lv[level];
    if (lv.n == 0) return EMB_OK;
    if (!d_out) return EMB_ERR_BAD_INPUT;
    EMB_LAUNCH((k_unpack_keys), emb_grid(lv.n, 256), 256, 0, emb_stream(stream))(lv.key, lv.n, d_out);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}

extern "C" emb_status emb_forest_neighbors(emb_forest f, int32_t level, int32_t *d_out, void *stream)
{
    EMB_SETTLE(f);
    if (!f || level < 0 || level > f->top) return EMB_ERR_STATE;
    EmbLevel &lv = f->lv[level];
    if (lv.n == 0) return EMB_OK;
    if (!d_out) return EMB_ERR_BAD_INPUT;
    cudaStream_t s = emb_stream(stream);
    emb_status rc = emb_build_neighbors(lv, s);
    if (rc != EMB_OK) return rc;
    EMB_CUDA_TRY(cudaMemcpyAsync(d_out, lv.nbr, lv.n * 26 * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    return EMB_OK;
}

extern "C" emb_status emb_forest_masks(emb_forest f, int32_t level, uint64_t *d_out, void *stream)
{
    EMB_SETTLE(f);
    if (!f || level < 0 || level > f->top || !f->lv[level].mask_valid) return EMB_ERR_STATE;
    const EmbLevel &lv = f->lv[level];
    if (lv.n == 0) return EMB_OK;
    if (!d_out) return EMB_ERR_BAD_INPUT;
    EMB_CUDA_TRY(cudaMemcpyAsync(d_out, lv.mask, lv.n * sizeof(uint64_t), cudaMemcpyDeviceToDevice, emb_stream(stream)));
    return EMB_OK;
}
