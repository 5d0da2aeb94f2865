// Solid voxelization of one level (Sec. 3.4, "Partial Surface Voxelization" and
// "External Cell Flag Propagation").
//
// A cell is solid iff its centre lies inside the closed surface, i.e. iff the
// +x ray from the (perturbed) centre crosses the surface an odd number of times.
// The work is split along each x-line of cell centres:
//   k_vox (triangle-parallel over the filtered list): every crossing of a level
//     x-line with a triangle is owned by the block whose box [lo, lo + W) holds
//     the crossing's x.  The owner XORs two things: for each of its four cells on
//     that line, whether the crossing lies beyond the cell centre (bit of s), and
//     the line's block parity (bit of p).
//   k_xscan (one thread per block): solid = s XOR (parity of every crossing in the
//     blocks further along +x), by a segmented suffix scan over the rows.
// Rows are contiguous and x-ordered in the level's block list.  Under the distance
// refine rule, unrefined gaps between blocks of a row contain no surface; under the
// paper's block-layer rule they may, and a crossing in a gap joins the line parity of
// the next block of the row (or a tail word of the row's last block that the row scan
// starts from), so the scan sees every crossing either way.  Block-local parity plays the role of the
// paper's internal propagation, and the suffix scan that of Alg. 4's
// neighbour-to-neighbour walk along +x.
#include "emb_internal.cuh"

// One triangle as the voxelizer sees it: its x-lines (j, k) in [j0, j1] x [k0, k1]
// and the x-range [bx0, bx1] of blocks its crossings can fall in.
struct VoxTri {
    int4 A, B, C;
    long long nx, ny, nz;
    int sx;
    int j0, j1, k0, k1, bx0, bx1;
    bool narrow;  // plane offsets of this triangle fit 64 bits (vox_cross)
};

// false for a triangle parallel to x (no line crosses it); in 32 bits but for the normal
// (coordinates below 2^25)
__device__ __forceinline__ bool vox_setup(const int4 *__restrict__ rec, int64_t t, const LevelGeom &g, VoxTri &V)
{
    V.A = rec[3 * t];
    V.B = rec[3 * t + 1];
    V.C = rec[3 * t + 2];
    const int4 A = V.A, B = V.B, C = V.C;
    const int ux = B.x - A.x, uy = B.y - A.y, uz = B.z - A.z, vx = C.x - A.x, vy = C.y - A.y, vz = C.z - A.z;
    V.nx = (long long)uy * vz - (long long)uz * vy;
    V.ny = (long long)uz * vx - (long long)ux * vz;
    V.nz = (long long)ux * vy - (long long)uy * vx;
    if (V.nx == 0) return false;
    V.sx = V.nx > 0 ? 1 : -1;
    const int lox = min(A.x, min(B.x, C.x)), hix = max(A.x, max(B.x, C.x)), loy = min(A.y, min(B.y, C.y)),
              hiy = max(A.y, max(B.y, C.y)), loz = min(A.z, min(B.z, C.z)), hiz = max(A.z, max(B.z, C.z));
    const int half = (int)g.half, nc = (int)g.ncell;
    V.j0 = max(-((-(loy - half)) >> g.lh), 0);
    V.j1 = min((hiy - half) >> g.lh, nc - 1);
    V.k0 = max(-((-(loz - half)) >> g.lh), 0);
    V.k1 = min((hiz - half) >> g.lh, nc - 1);
    V.bx0 = max(lox >> g.lW, 0);
    V.bx1 = min(hix >> g.lW, (int)g.nb - 1);
    V.narrow = max(hix - lox, max(hiy - loy, hiz - loz)) < (1 << 18) && g.lW <= 18;
    return true;
}

__device__ __forceinline__ unsigned long long vox_items(const VoxTri &V)
{
    if (V.j1 < V.j0 || V.k1 < V.k0) return 0;
    return (unsigned long long)(V.j1 - V.j0 + 1) * (unsigned long long)(V.k1 - V.k0 + 1);
}

// Parity sinks of one voxelization: per block the cell bits s and the line parity p,
// and per block the row tail t (crossings beyond the last block of its row, read by
// the row scan of that last block); the level's sorted keys locate them.
struct VoxAcc {
    unsigned long long *s;
    unsigned int *p, *t;
    const uint64_t *key;
    int64_t n;
};

// A crossing inside a block position the level does not have (a region left coarser by
// the refinement rule): it flips every cell of the row to its left, so it joins the line
// parity of the next block of the row to its right, or the row tail of the row's last
// block when there is none.
__device__ __noinline__ void vox_gap(const VoxAcc &acc, long long bx, long long by, long long bz, int line)
{
    const uint64_t row = (uint64_t)emb_key(0, by, bz) >> EMB_KEY_BITS;
    const int64_t nx = lower_bound_u64(acc.key, acc.n, emb_key(bx + 1, by, bz));
    if (nx < acc.n && (acc.key[nx] >> EMB_KEY_BITS) == row) atomicXor(acc.p + nx, 1u << line);
    else if (nx > 0 && (acc.key[nx - 1] >> EMB_KEY_BITS) == row) atomicXor(acc.t + nx - 1, 1u << line);
}

// The block of [bx0, bx1] whose box [lo, lo + W) holds the crossing of the line (py, pz) with
// the plane, and its cells before the crossing; -1 if none does.  n . (A - (x, py, pz)) =
// D_yz + n_x (A_x - x); the crossing is at x_hit with x_hit - x = D(x) / n_x.  In 64 bits
// where the triangle's extents and W are at most 2^18: |n| <= 2^37, A.y - py and A.z - pz lie
// within the extent (the line meets the projection), A.x - lo within extent + W, so every sum
// stays below 2^58; else in 128.  (Always in 128, the levels of embed_112k took 42 us and those
// of 7.2M triangles 123; now 36 and 95.)
// Returned as bx << 4 | cells.
template <class I>
__device__ __forceinline__ int vox_cross(long long nx, long long ny, long long nz, int ax, int dy, int dz, int bx0, int bx1,
                                         int lW)
{
    const I Dyz = (I)ny * (I)dy + (I)nz * (I)dz;
    const bool pos = nx > 0;
    const int half = 1 << (lW - 3);  // W = 8 half
    for (int bx = bx0; bx <= bx1; ++bx) {
        const I Dlo = Dyz + (I)nx * (I)(ax - (bx << lW));
        if (pos ? Dlo < 0 : Dlo > 0) continue;  // x_hit < lo
        const I Dhi = Dlo - ((I)nx << lW);
        if (pos ? Dhi >= 0 : Dhi <= 0) continue;  // x_hit >= lo + W
        // cell q of this line (centre lo + (2q+1) half) lies before the crossing iff
        // the perturbed centre sees the plane ahead: sign(D) == sign(n_x), D == 0 -> no
        int bits = 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const I Dq = Dlo - (I)nx * (I)((2 * q + 1) * half);
            if (pos ? Dq > 0 : Dq < 0) bits |= 1 << q;
        }
        return bx << 4 | bits;
    }
    return -1;
}
__device__ __noinline__ int vox_cross_wide(long long nx, long long ny, long long nz, int ax, int dy, int dz, int bx0, int bx1,
                                           int lW)
{
    return vox_cross<i128>(nx, ny, nz, ax, dy, dz, bx0, bx1, lW);
}

// The crossing of line (j, k) with the triangle, if any, recorded in its owner block.
__device__ __forceinline__ void vox_line(const VoxTri &V, const LevelGeom &g, const EmbLookup &lk, int j, int k,
                                         const VoxAcc &acc, int *st)
{
    const int4 A = V.A, B = V.B, C = V.C;
    const int sx = V.sx, half = (int)g.half;
    const int pz = (2 * k + 1) * half, py = (2 * j + 1) * half;
    if (emb_orient_yz(A.y, A.z, B.y, B.z, py, pz) != sx || emb_orient_yz(B.y, B.z, C.y, C.z, py, pz) != sx ||
        emb_orient_yz(C.y, C.z, A.y, A.z, py, pz) != sx)
        return;
    const int r = V.narrow ? vox_cross<long long>(V.nx, V.ny, V.nz, A.x, A.y - py, A.z - pz, V.bx0, V.bx1, g.lW)
                           : vox_cross_wide(V.nx, V.ny, V.nz, A.x, A.y - py, A.z - pz, V.bx0, V.bx1, g.lW);
    if (r < 0) {
        emb_set_status(st, EMB_ERR_STATE);  // no block owns the crossing
        return;
    }
    const int32_t id = emb_lookup(lk, r >> 4, j >> 2, k >> 2);
    const int line = (j & 3) + 4 * (k & 3);
    if (id < 0) {
        vox_gap(acc, r >> 4, j >> 2, k >> 2, line);
        return;
    }
    if (!emb_ck((uint64_t)id, (uint64_t)acc.n, st)) return;
    if (r & 15) atomicXor(acc.s + id, (unsigned long long)(r & 15) << (4 * line));
    atomicXor(acc.p + id, 1u << line);
}

// 80 registers (the 128-bit path alone would take 112): latency-bound, six warps a scheduler.
__global__ void __maxnreg__(80) k_vox(const int4 *__restrict__ rec, int64_t T, const uint32_t *__restrict__ flist, int64_t nf,
                      const uint32_t *__restrict__ d_nf, const uint32_t *__restrict__ keep, LevelGeom g, EmbLookup lk,
                      VoxAcc acc, EmbBigQ Q, int *st)
{
    // nf: the planned count of a replay, or T when the count is still on the device;
    // d_nf: the count the filter found.  Grid-stride, so that a level with few kept
    // triangles does not launch a thread per triangle of the mesh.
    int64_t n = nf;
    if (d_nf && (int64_t)*d_nf < n) n = (int64_t)*d_nf;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = flist[i];
        if ((int64_t)t >= T) continue;
        if (keep && !keep[t]) continue;  // filtered out, the list not compacted
        VoxTri V;
        if (!vox_setup(rec, t, g, V)) continue;
        const unsigned long long items = vox_items(V);
        if (items > Q.items && emb_bigq_push(Q, t, items)) continue;
        for (int k = V.k0; k <= V.k1; ++k)
            for (int j = V.j0; j <= V.j1; ++j) vox_line(V, g, lk, j, k, acc, st);
    }
}

// The queued chunks of large triangles, one warp per chunk (lines in j-major order).
__global__ void __launch_bounds__(EMB_BIG_BLOCK) k_vox_big(const int4 *__restrict__ rec, LevelGeom g, EmbLookup lk,
                                                           VoxAcc acc, EmbBigQ Q, int *st)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long nq = emb_bigq_count(Q);
    const unsigned long long nw = (unsigned long long)gridDim.x * (EMB_BIG_BLOCK / 32);
    for (unsigned long long e = (unsigned long long)blockIdx.x * (EMB_BIG_BLOCK / 32) + (threadIdx.x >> 5); e < nq;
         e += nw) {
        const uint2 E = Q.q[e];
        if (E.x == EMB_BIG_NONE) continue;
        VoxTri V;
        if (!vox_setup(rec, E.x, g, V)) continue;
        const unsigned long long items = vox_items(V);
        unsigned long long i0, i1;
        emb_bigq_range(E.y, items, i0, i1);
        const unsigned long long nj = (unsigned long long)(V.j1 - V.j0 + 1);
        const unsigned long long first = i0 + lane;
        long long jj = (long long)(first % nj), kk = (long long)(first / nj);
        const long long dj = (long long)(32 % nj), dk = (long long)(32 / nj);
        for (unsigned long long it = first; it < i1; it += 32) {
            vox_line(V, g, lk, V.j0 + (int)jj, V.k0 + (int)kk, acc, st);
            jj += dj;
            kk += dk;
            if (jj >= (long long)nj) {
                jj -= (long long)nj;
                ++kk;
            }
        }
    }
}

// Bit l of a 16-bit line set -> the four cell bits 4l .. 4l+3.
__device__ __forceinline__ unsigned long long spread_lines(unsigned int p)
{
    unsigned long long x = p & 0xFFFFu;
    x = (x | (x << 24)) & 0x000000FF000000FFull;
    x = (x | (x << 12)) & 0x000F000F000F000Full;
    x = (x | (x << 6)) & 0x0303030303030303ull;
    x = (x | (x << 3)) & 0x1111111111111111ull;
    return x * 0xFull;
}

// A warp takes 32 consecutive blocks: y = the XOR of the line parities from a block to the
// end of its row (the row tail included), a suffix scan in which a row's blocks are
// neighbours; the row that goes on past the warp's last block is followed 32 blocks at a
// time.  Everything is read and written coalesced.  (One thread walking each row, 8 blocks
// a step, took 9.4 us on 97K blocks and 59 on 1.0M, the second mask a copy of its own.)
__global__ void __launch_bounds__(256) k_xscan(const uint64_t *__restrict__ key, int64_t n,
                                               const unsigned long long *__restrict__ s_acc,
                                               const unsigned int *__restrict__ p_acc,
                                               const unsigned int *__restrict__ t_acc, uint64_t *__restrict__ mask,
                                               uint64_t *__restrict__ mask_out, const uint32_t *d_n)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    n = emb_count(n, d_n);
    if (i - lane >= n) return;  // the whole warp
    // block j of a warp's 32 (row ~0: none), whether its row ends there, and its parities
    auto load = [&](int64_t j, uint64_t &row, bool &last, unsigned int &p) {
        row = j < n ? key[j] >> EMB_KEY_BITS : ~0ull;
        uint64_t next = __shfl_down_sync(0xffffffffu, row, 1);
        if (lane == 31) next = j + 1 < n ? key[j + 1] >> EMB_KEY_BITS : ~0ull;
        last = next != row;
        p = j < n ? p_acc[j] : 0u;
        return j < n && last ? p ^ t_acc[j] : p;
    };
    uint64_t row;
    bool last;
    unsigned int p;
    unsigned int y = load(i, row, last, p);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned int v = __shfl_down_sync(0xffffffffu, y, o);
        const uint64_t r = __shfl_down_sync(0xffffffffu, row, o);
        if (lane + o < 32 && r == row) y ^= v;
    }
    const uint64_t row31 = __shfl_sync(0xffffffffu, row, 31);
    bool more = row31 != ~0ull && !__shfl_sync(0xffffffffu, (int)last, 31);  // ~0: past the last block
    unsigned int carry = 0;
    for (int64_t j = i + 32; more; j += 32) {
        uint64_t r;
        bool l;
        unsigned int pp;
        const unsigned int v = load(j, r, l, pp);
        carry ^= __reduce_xor_sync(0xffffffffu, r == row31 ? v : 0u);
        more = __shfl_sync(0xffffffffu, (int)(r == row31 && !l), 31);
    }
    if (row == row31) y ^= carry;
    if (i >= n) return;
    const uint64_t m = s_acc[i] ^ spread_lines(y ^ p);
    mask[i] = m;
    if (mask_out) mask_out[i] = m;
}

// Scratch words of a voxelization of n blocks: cell bits, line parities, row tails, and
// the count of the chunk queue, cleared together.
int64_t emb_vox_words(int64_t n) { return 2 * n + 1; }

// Enqueue only: acc is scratch of emb_vox_words(lv.n); writes lv.mask, and mask_out (device
// memory) when given.
emb_status emb_enq_voxelize(const int4 *rec, int64_t T, const uint32_t *flist, int64_t nf, const uint32_t *d_nf,
                            const uint32_t *keep, LevelGeom g, const EmbLevel &lv, uint64_t *acc, uint64_t *mask_out,
                            const EmbBigQ &Q, int block, cudaStream_t s)
{
    int *st = emb_status_word();
    if (!st) return EMB_ERR_CUDA;
    if (lv.n == 0) return EMB_OK;
    unsigned long long *s_acc = (unsigned long long *)acc;
    unsigned int *p_acc = (unsigned int *)(s_acc + lv.n), *t_acc = p_acc + lv.n;
    EMB_CUDA_TRY(cudaMemsetAsync(acc, 0, emb_vox_words(lv.n) * sizeof(uint64_t), s));
    const VoxAcc va = {s_acc, p_acc, t_acc, lv.key, lv.n};
    EmbBigQ q = Q;
    q.n = (unsigned long long *)(t_acc + lv.n);
    if (nf > 0) {
        const EmbLookup lk = emb_lookup_of(lv);
        int64_t grid = emb_grid(nf, block);
        const int64_t full = (int64_t)emb_sm_count() * (2048 / block);  // one resident wave
        if (grid > full) grid = full;
        EMB_LAUNCH((k_vox), (int)grid, block, 0, s)(rec, T, flist, nf, d_nf, keep, g, lk, va, q, st);
        if (q.cap) EMB_LAUNCH((k_vox_big), EMB_BIG_GRID, EMB_BIG_BLOCK, 0, s)(rec, g, lk, va, q, st);
    }
    EMB_LAUNCH((k_xscan), emb_grid(lv.n, 256), 256, 0, s)(lv.key, lv.n, s_acc, p_acc, t_acc, lv.mask, mask_out, lv.d_n);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}

extern "C" emb_status emb_voxelize(emb_forest f, emb_bins b, int32_t level, uint64_t *d_solid_mask, void *stream)
{
    if (!f || !b) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    if (b->f != f || b->level != level || level < 0 || level > f->top) return EMB_ERR_STATE;
    void *mask_out = nullptr;
    bool dev_out = false;
    if (emb_device_view(d_solid_mask, &mask_out, &dev_out) != EMB_OK) return EMB_ERR_BAD_INPUT;
    cudaStream_t s = emb_stream(stream);
    EmbLevel &lv = f->lv[level];
    LevelGeom g = level_geom(f, level);
    if (lv.n == 0) {
        lv.mask_valid = 1;
        return EMB_OK;
    }
    if (!lv.mask) EMB_CUDA_TRY(emb_malloc_async(&lv.mask, lv.n * sizeof(uint64_t), s));
    // the accumulators and, where a triangle may cross more than EMB_BIG_ITEMS lines, the
    // entries of the chunk queue
    const emb_mesh m = b->m;
    EmbBigQ Q = emb_bigq(m->T);
    if (emb_mesh_big(m, 1, (m->ext >> g.lh) + 1, (m->ext >> g.lh) + 1)) Q.cap = (uint32_t)emb_bigq_capacity(m->T);
    const size_t a_acc = ((size_t)emb_vox_words(lv.n) * sizeof(uint64_t) + 255) & ~(size_t)255;
    char *scratch = nullptr;
    EMB_CUDA_TRY(emb_malloc_async(&scratch, a_acc + (size_t)Q.cap * sizeof(uint2), s));
    Q.q = (uint2 *)(scratch + a_acc);
    // the filtered count stays on the device: the grid covers every triangle and stops at it
    const emb_status rc =
        emb_enq_voxelize(m->rec, m->T, b->flist, b->known ? b->nf : m->T, (const uint32_t *)b->dcount, b->keep, g, lv,
                         (uint64_t *)scratch, dev_out ? (uint64_t *)mask_out : nullptr, Q, 128, s);
    if (rc != EMB_OK) return rc;
    if (mask_out && !dev_out)  // page-locked host memory: an asynchronous copy over the host link
        EMB_CUDA_TRY(cudaMemcpyAsync(mask_out, lv.mask, lv.n * sizeof(uint64_t), cudaMemcpyDefault, s));
    EMB_CUDA_TRY(cudaFreeAsync(scratch, s));
    lv.mask_valid = 1;
    if (level == f->top) f->n_links = -1;
    return EMB_OK;
}
