// Near-wall refinement flags (Sec. 3.4, "Refinement Flagging and Propagation").
//
// The paper marks solid-boundary blocks and propagates flags block by block a
// number of layers set by the near-wall distance (Eq. N_prop).  Here the
// criterion is evaluated directly and exactly: block B of level L is flagged iff
// some triangle overlaps B's closed box dilated by (rho_L - 1/2) h_L, i.e. iff a
// cell centre of B lies within L-infinity distance rho_L h_L of the surface.
// rho equals `band` one level above the finest and grows towards the root as
// rho_L = max(band, rho_{L+1}/2 + 5/2), which keeps all 26 neighbours of every
// refined block present (2:1 balance) and leaves unrefined blocks surface-free.
//
// Warps over tiles of 32 consecutive triangles (details at k_refine); a triangle with very
// many candidates goes in queued chunks to whole warps.  Flags are idempotent byte stores.
#include <math.h>

#include <atomic>

#include "emb_internal.cuh"

#define REFINE_WARPS 8
#ifndef REFINE_MINB
#define REFINE_MINB 4
#endif
// Largest bitmap (words) that a CTA of k_refine keeps a copy of: up to 64 blocks an axis.
#define REFINE_SM_WORDS 4096

__device__ __forceinline__ void refine_setup(const int4 *__restrict__ rec, int64_t t, const LevelGeom &g, long long dil,
                                             int4 &A, int4 &B, int4 &C, long long b0[3], long long b1[3])
{
    A = rec[3 * t];
    B = rec[3 * t + 1];
    C = rec[3 * t + 2];
    emb_block_range(min(A.x, min(B.x, C.x)), max(A.x, max(B.x, C.x)), g.lW, dil, g.nb, b0[0], b1[0]);
    emb_block_range(min(A.y, min(B.y, C.y)), max(A.y, max(B.y, C.y)), g.lW, dil, g.nb, b0[1], b1[1]);
    emb_block_range(min(A.z, min(B.z, C.z)), max(A.z, max(B.z, C.z)), g.lW, dil, g.nb, b0[2], b1[2]);
}

__device__ __forceinline__ unsigned long long refine_items(const long long b0[3], const long long b1[3])
{
    if (b1[0] < b0[0] || b1[1] < b0[1] || b1[2] < b0[2]) return 0;
    return (unsigned long long)(b1[0] - b0[0] + 1) * (unsigned long long)(b1[1] - b0[1] + 1) *
           (unsigned long long)(b1[2] - b0[2] + 1);
}

// Blocks of the level that are not flagged yet as one bit per dense position (bx + nb (by +
// nb bz)), when the level has a rank bitmap: a copy of it, from which flagging clears bits.
// One load tells a candidate that is missing or flagged from one that is left, and flagging
// is one atomic that nothing waits for; k_refine_flags turns the bits into the flag bytes
// afterwards.  w is in global memory, or for a small level in shared memory: a copy that the
// CTA keeps and merges at its end, since every warp of the grid reads and clears the few
// words of a coarse level (111K triangles on 16^3 blocks: 139 us through the L2).  A word
// read before another warp cleared a bit only sends the candidate through the full test,
// which decides exactly and flags once more.
// Words of 32 bits: those have native atomics in shared memory, 64-bit ones a
// compare-and-swap loop.
struct TodoBits {
    uint32_t *w;  // null: no dense bits, look the block up and test the flag bytes
    long long nb;
    int *st;
    // bounds mode: position p is one of the level's
    __device__ __forceinline__ bool in(unsigned long long p) const { return emb_ck(p, (uint64_t)nb * nb * nb, st); }
    __device__ __forceinline__ unsigned long long pos(long long bx, long long by, long long bz) const
    {
        return (unsigned long long)((bz * nb + by) * nb + bx);
    }
    __device__ __forceinline__ bool test(long long bx, long long by, long long bz) const
    {
        const unsigned long long p = pos(bx, by, bz);
        return in(p) && ((w[p >> 5] >> (p & 31)) & 1u);
    }
    __device__ __forceinline__ void clear(long long bx, long long by, long long bz) const
    {
        const unsigned long long p = pos(bx, by, bz);
        if (in(p)) atomicAnd(w + (p >> 5), ~(1u << (p & 31)));
    }
    // bits [0, nx) of the row segment from (bx, by, bz), nx <= 32
    __device__ __forceinline__ uint32_t row(int bx, int by, int bz, int nx) const
    {
        const unsigned long long p = pos(bx, by, bz);
        if (!in(p + (unsigned)(nx - 1))) return 0u;
        const int sh = (int)(p & 31);
        const uint32_t lo = w[p >> 5], hi = sh + nx > 32 ? w[(p >> 5) + 1] : 0u;
        return __funnelshift_r(lo, hi, sh) & (0xffffffffu >> (32 - nx));
    }
};

// Block (bx, by, bz) is left to flag.
__device__ __forceinline__ bool refine_left(const EmbLookup &lk, const TodoBits &td, const uint8_t *__restrict__ flags,
                                            long long bx, long long by, long long bz)
{
    if (td.w) return td.test(bx, by, bz);
    const int32_t id = emb_lookup(lk, bx, by, bz);
    return id >= 0 && !*((volatile const uint8_t *)flags + id);
}

__device__ __forceinline__ void refine_flag(const EmbLookup &lk, const TodoBits &td, uint8_t *__restrict__ flags,
                                            long long bx, long long by, long long bz)
{
    if (td.w) {
        td.clear(bx, by, bz);
        return;
    }
    const int32_t id = emb_lookup(lk, bx, by, bz);
    if (id >= 0) flags[id] = 1;
}

// The flag bytes of a level with the bitmap: the blocks whose bit was cleared (none of the
// entries past a replay's count).
__global__ void k_refine_flags(const uint64_t *__restrict__ key, int64_t n, const uint32_t *d_n,
                               const uint32_t *__restrict__ todo, int64_t nb, uint8_t *__restrict__ flags)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint8_t f = 0;
    if (i < emb_count(n, d_n)) {
        const uint64_t k = key[i];
        const int64_t bx = (int64_t)(k & EMB_KEY_MASK), by = (int64_t)((k >> EMB_KEY_BITS) & EMB_KEY_MASK),
                      bz = (int64_t)(k >> (2 * EMB_KEY_BITS));
        if (bx < nb && by < nb && bz < nb) {
            const int64_t pos = (bz * nb + by) * nb + bx;
            f = (uint8_t)(((todo[pos >> 5] >> (pos & 31)) & 1u) ^ 1u);
        }
    }
    flags[i] = f;
}

// 32-bit forms of the per-block arithmetic: coordinates, block origins, widths and
// dilations all lie below 2^25 in magnitude, block indices below 2^21.
__device__ __forceinline__ void ref_range(int mn, int mx, int lW, int dil, int nb, int &b0, int &b1)
{
    b0 = -((-(mn - dil - (1 << lW))) >> lW);  // ceil
    b1 = (mx + dil) >> lW;                    // floor
    if (b0 < 0) b0 = 0;
    if (b1 > nb - 1) b1 = nb - 1;
}
__device__ __forceinline__ bool ref_pt(const int4 &P, int lx, int ly, int lz, int hx, int hy, int hz)
{
    return P.x >= lx && P.x <= hx && P.y >= ly && P.y <= hy && P.z >= lz && P.z <= hz;
}
// (triangle lane, bx, by, bz) of candidates none of whose vertices lies in the dilated block,
// waiting for the separating-axis test.
struct RefWarp {
    int4 A[32], B[32], C[32];
    int4 q[64];
};

// The separating-axis test of the last n queued candidates, one a lane; a block flagged in
// the meantime is passed over.
__device__ __forceinline__ void ref_drain(RefWarp &S, int &qn, int n, int lane, int W, int dil, const EmbLookup &lk,
                                          const TodoBits &td, uint8_t *__restrict__ flags)
{
    __syncwarp();
    if (lane < n) {
        const int4 e = S.q[qn - n + lane];
        if (refine_left(lk, td, flags, e.y, e.z, e.w)) {
            const int lx = e.y * W - dil, ly = e.z * W - dil, lz = e.w * W - dil, w = W + 2 * dil;
            if (emb_tri_box(S.A[e.x], S.B[e.x], S.C[e.x], lx, ly, lz, lx + w, ly + w, lz + w))
                refine_flag(lk, td, flags, e.y, e.z, e.w);
        }
    }
    qn -= n;
    __syncwarp();
}

// Persistent CTAs, each over consecutive tiles of 32 consecutive triangles (so that the
// blocks it meets are few and soon flagged); each warp loads the records of its next tile
// before it works on the current one.  A tile is screened first: the rows of the union of its
// candidate blocks, one a lane, show in one load each which of them are left to flag; in a
// large mesh there is none for most tiles, or only where no lane's own candidates reach (the
// union is a box).  Otherwise every lane goes through the blocks left
// among its own triangle's candidates: a vertex in the dilated block flags it, else the
// pair waits for the separating-axis test, which the warp runs 32 at a time.
// Latency-bound; four CTAs an SM (64 registers, which spill 188 bytes of stores and 84 of loads
// a thread) over three: 5 % on 7.2M triangles.  Time over the levels, before (the union's or
// the spread pairs' blocks looked up and tested at once, global flag bits) and now: 7.2M
// triangles 1311 -> 860 us, 1.0M 311 -> 231, 111K 118 -> 91.  Triangles and vertices in any
// order: an embedding of 7.2M shuffled ones 10.4 -> 7.2 ms, of 1.0M 2.26 -> 1.80.
// Taking the union's blocks left one at a time for the whole warp is slower on most levels
// (986 us, 111K: 154).
template <bool SM>
__global__ void __launch_bounds__(REFINE_WARPS * 32, REFINE_MINB) k_refine(const int4 *__restrict__ rec, int64_t T, LevelGeom g,
                                                              long long dil, EmbLookup lk, uint8_t *__restrict__ flags,
                                                              uint32_t *todo, int nw, int64_t chunk, EmbBigQ Q)
{
    extern __shared__ __align__(16) unsigned char ref_smem[];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    RefWarp &S = reinterpret_cast<RefWarp *>(ref_smem)[w];
    uint32_t *const s_todo = (uint32_t *)(ref_smem + REFINE_WARPS * sizeof(RefWarp));
    if (SM) {
        for (int i = threadIdx.x; i < nw; i += REFINE_WARPS * 32) s_todo[i] = __ldcg(todo + i);
        __syncthreads();
    }
    const TodoBits td = {SM ? s_todo : todo, g.nb, lk.st};
    const int64_t first = (int64_t)blockIdx.x * chunk, all = (T + 31) / 32;
    const int64_t ntiles = first + chunk < all ? first + chunk : all, stride = REFINE_WARPS;
    int64_t tile = first + w;
    const int dil32 = (int)dil, W32 = (int)g.W, nb32 = (int)g.nb;
    int4 nA = make_int4(0, 0, 0, 0), nB = nA, nC = nA;
    if (tile < ntiles && tile * 32 + lane < T) {
        const int64_t t = tile * 32 + lane;
        nA = rec[3 * t];
        nB = rec[3 * t + 1];
        nC = rec[3 * t + 2];
    }
    for (; tile < ntiles; tile += stride) {
        const int64_t t = tile * 32 + lane;
        const int4 A = nA, B = nB, C = nC;
        {
            const int64_t tn = (tile + stride) * 32 + lane;
            if (tile + stride < ntiles && tn < T) {
                nA = rec[3 * tn];
                nB = rec[3 * tn + 1];
                nC = rec[3 * tn + 2];
            }
        }
        int b0[3] = {0x7fffffff, 0x7fffffff, 0x7fffffff}, b1[3] = {-1, -1, -1};
        if (t < T) {
            ref_range(min(A.x, min(B.x, C.x)), max(A.x, max(B.x, C.x)), g.lW, dil32, nb32, b0[0], b1[0]);
            ref_range(min(A.y, min(B.y, C.y)), max(A.y, max(B.y, C.y)), g.lW, dil32, nb32, b0[1], b1[1]);
            ref_range(min(A.z, min(B.z, C.z)), max(A.z, max(B.z, C.z)), g.lW, dil32, nb32, b0[2], b1[2]);
        }
        int u0[3], un[3];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            u0[d] = __reduce_min_sync(0xffffffffu, b0[d]);
            un[d] = __reduce_max_sync(0xffffffffu, b1[d]) - u0[d] + 1;
        }
        if (un[0] <= 0 || un[1] <= 0 || un[2] <= 0) continue;
        bool may = true;  // a block left may be among the lane's candidates
        if (td.w && un[0] <= 32 && un[1] <= 32 && un[2] <= 32) {
            const unsigned ny = (unsigned)un[1], rows = ny * (unsigned)un[2], my = emb_recip(ny);
            uint32_t xs = 0, ys = 0, zs = 0;  // where on the axes of the union there are any
            for (unsigned r = lane; r < rows; r += 32) {
                const unsigned rz = emb_div_recip(r, ny, my), ry = r - rz * ny;
                const uint32_t m = td.row(u0[0], u0[1] + (int)ry, u0[2] + (int)rz, un[0]);
                if (m) {
                    xs |= m;
                    ys |= 1u << ry;
                    zs |= 1u << rz;
                }
            }
            xs = __reduce_or_sync(0xffffffffu, xs);
            if (xs == 0u) continue;
            ys = __reduce_or_sync(0xffffffffu, ys);
            zs = __reduce_or_sync(0xffffffffu, zs);
            auto in = [&](int d) {  // b0 <= b1 within the union: shifts of 0 .. 31
                return b0[d] <= b1[d] ? (0xffffffffu >> (31 - (b1[d] - u0[d]))) & (0xffffffffu << (b0[d] - u0[d])) : 0u;
            };
            may = (xs & in(0)) && (ys & in(1)) && (zs & in(2));
            if (!__any_sync(0xffffffffu, may)) continue;
        }
        const int onx = b1[0] - b0[0] + 1, ony = b1[1] - b0[1] + 1, onz = b1[2] - b0[2] + 1;
        const unsigned long long own = t < T && onx > 0 && ony > 0 && onz > 0
                                           ? (unsigned long long)onx * (unsigned long long)ony * (unsigned long long)onz
                                           : 0ull;
        const bool mine = may && own > 0 && !(own > Q.items && emb_bigq_push(Q, (uint32_t)t, own));
        S.A[lane] = A;  // the previous tile's queue was drained behind a warp barrier
        S.B[lane] = B;
        S.C[lane] = C;
        int qn = 0;
        // the lane's place in its candidates: a row (y, z) and, in it, the blocks from x on
        int x = 0x7fffffff, y = b0[1] - 1, z = b0[2];
        uint32_t m = 0;  // blocks left in the row segment from x (with the bitmap)
        bool more = mine;
        while (__any_sync(0xffffffffu, more)) {
            bool need = false;
            int bx = 0, by = 0, bz = 0;
            while (more && !need) {
                // the next candidate that is left to flag
                bool have = false;
                if (td.w) {
                    if (m == 0) {
                        // the next 32 blocks of the row, or the next row
                        if (y >= b0[1] && x + 32 <= b1[0]) {
                            x += 32;
                        } else {
                            x = b0[0];
                            if (++y > b1[1]) {
                                y = b0[1];
                                ++z;
                            }
                        }
                        if (z > b1[2]) {
                            more = false;
                            break;
                        }
                        m = td.row(x, y, z, min(32, b1[0] - x + 1));
                    }
                    if (m) {
                        const int i = __ffs(m) - 1;
                        m &= m - 1;
                        bx = x + i;
                        have = true;
                    }
                } else {
                    if (y < b0[1] || ++x > b1[0]) {
                        x = b0[0];
                        if (++y > b1[1]) {
                            y = b0[1];
                            ++z;
                        }
                    }
                    if (z > b1[2]) {
                        more = false;
                        break;
                    }
                    bx = x;
                    have = refine_left(lk, td, flags, x, y, z);
                }
                if (!have) continue;
                by = y;
                bz = z;
                const int lx = bx * W32 - dil32, ly = by * W32 - dil32, lz = bz * W32 - dil32, wd = W32 + 2 * dil32;
                if (ref_pt(A, lx, ly, lz, lx + wd, ly + wd, lz + wd) || ref_pt(B, lx, ly, lz, lx + wd, ly + wd, lz + wd) ||
                    ref_pt(C, lx, ly, lz, lx + wd, ly + wd, lz + wd))
                    refine_flag(lk, td, flags, bx, by, bz);
                else
                    need = true;
            }
            const unsigned nm = __ballot_sync(0xffffffffu, need);
            if (need) S.q[qn + __popc(nm & ((1u << lane) - 1u))] = make_int4(lane, bx, by, bz);
            qn += __popc(nm);
            if (qn >= 32) ref_drain(S, qn, 32, lane, W32, dil32, lk, td, flags);
        }
        if (qn > 0) ref_drain(S, qn, qn, lane, W32, dil32, lk, td, flags);
        __syncwarp();
    }
    if (SM) {
        __syncthreads();
        for (int i = threadIdx.x; i < nw; i += REFINE_WARPS * 32) {
            const uint32_t v = s_todo[i];
            if (__ldcg(todo + i) & ~v) atomicAnd(todo + i, v);
        }
    }
}

// The queued chunks of large triangles, one warp per chunk (candidates x fastest).
__global__ void __launch_bounds__(EMB_BIG_BLOCK) k_refine_big(const int4 *__restrict__ rec, LevelGeom g, long long dil,
                                                              EmbLookup lk, uint8_t *__restrict__ flags, TodoBits td,
                                                              EmbBigQ Q)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long nq = emb_bigq_count(Q);
    const unsigned long long nw = (unsigned long long)gridDim.x * (EMB_BIG_BLOCK / 32);
    for (unsigned long long e = (unsigned long long)blockIdx.x * (EMB_BIG_BLOCK / 32) + (threadIdx.x >> 5); e < nq;
         e += nw) {
        const uint2 E = Q.q[e];
        if (E.x == EMB_BIG_NONE) continue;
        int4 A, B, C;
        long long b0[3], b1[3];
        refine_setup(rec, E.x, g, dil, A, B, C, b0, b1);
        unsigned long long i0, i1;
        emb_bigq_range(E.y, refine_items(b0, b1), i0, i1);
        const long long nx = b1[0] - b0[0] + 1, ny = b1[1] - b0[1] + 1;
        const unsigned long long first = i0 + lane;
        long long x = (long long)(first % (unsigned long long)nx);
        long long y = (long long)((first / (unsigned long long)nx) % (unsigned long long)ny);
        long long z = (long long)((first / (unsigned long long)nx) / (unsigned long long)ny);
        const long long dx = 32 % nx, dy = (32 / nx) % ny, dz = (32 / nx) / ny;
        for (unsigned long long it = first; it < i1; it += 32) {
            const long long bx = b0[0] + x, by = b0[1] + y, bz = b0[2] + z;
            if (refine_left(lk, td, flags, bx, by, bz)) {
                const long long lx = bx * g.W - dil, ly = by * g.W - dil, lz = bz * g.W - dil, wd = g.W + 2 * dil;
                if (emb_point_in_box(A, lx, ly, lz, lx + wd, ly + wd, lz + wd) ||
                    emb_point_in_box(B, lx, ly, lz, lx + wd, ly + wd, lz + wd) ||
                    emb_point_in_box(C, lx, ly, lz, lx + wd, ly + wd, lz + wd) ||
                    emb_tri_box(A, B, C, lx, ly, lz, lx + wd, ly + wd, lz + wd))
                    refine_flag(lk, td, flags, bx, by, bz);
            }
            x += dx;
            y += dy;
            z += dz;
            if (x >= nx) {
                x -= nx;
                ++y;
            }
            if (y >= ny) {
                y -= ny;
                ++z;
            }
        }
    }
}

// (rho_L - 1/2) h_L in frame units, or -1 if it is not an integer.  At most the width of the
// domain (below 2^25): from there on every block's dilated box holds the whole of it, and
// box corners stay within the 32 bits that the tests form them in.
long long emb_refine_dilation(const emb_forest_s *f, int L, int band)
{
    const int sh = 16;  // rho is kept as an integer multiple of 2^-16
    long long rho = (long long)band << sh;
    for (int l = f->max_level - 1; l > L; --l) {
        long long cand = rho / 2 + (5ll << (sh - 1));
        rho = cand > ((long long)band << sh) ? cand : ((long long)band << sh);
    }
    long long h = 1ll << (18 - f->k - L);
    long long num = (rho - (1ll << (sh - 1))) * h;
    if (num % (1ll << sh) != 0) return -1;
    const long long width = (long long)f->r_o << 20;
    return (num >> sh) < width ? num >> sh : width;
}

// The shared memory of the largest copied bitmap is above the default limit; set once a
// device, before any capture (a batch plans, and so launches, outside of one).
static emb_status refine_init()
{
    static std::atomic<bool> done[64];
    int dev = 0;
    EMB_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return EMB_ERR_CUDA;
    if (done[dev].load(std::memory_order_acquire)) return EMB_OK;
    EMB_CUDA_TRY(cudaFuncSetAttribute(k_refine<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(REFINE_WARPS * sizeof(RefWarp) + REFINE_SM_WORDS * sizeof(uint64_t))));
    done[dev].store(true, std::memory_order_release);
    return EMB_OK;
}

// Enqueue only: flags (lv.n bytes) are written; fbits (NULL for a level without a
// bitmap) is scratch of the size of the level's bitmap.
emb_status emb_enq_refine(const int4 *rec, int64_t T, LevelGeom g, long long dil, const EmbLevel &lv, uint8_t *flags,
                          unsigned long long *fbits, const EmbBigQ &Q, cudaStream_t s)
{
    if (lv.n == 0) return EMB_OK;
    const emb_status ri = refine_init();
    if (ri != EMB_OK) return ri;
    const EmbLookup lk = emb_lookup_of(lv);
    TodoBits td = {nullptr, g.nb, lk.st};
    const int64_t nw = emb_bitmap_words(lv.nb_axis);
    if (fbits && lv.bits && nw > 0) {
        EMB_CUDA_TRY(cudaMemcpyAsync(fbits, lv.bits, nw * sizeof(unsigned long long), cudaMemcpyDeviceToDevice, s));
        td.w = (uint32_t *)fbits;
    } else {
        EMB_CUDA_TRY(cudaMemsetAsync(flags, 0, lv.n, s));
    }
    if (Q.cap) EMB_CUDA_TRY(cudaMemsetAsync(Q.n, 0, sizeof(unsigned long long), s));
    // consecutive tiles for each CTA, a whole number of its warps
    const int64_t tiles = (T + 31) / 32, resident = (int64_t)emb_sm_count() * REFINE_MINB;
    int64_t chunk = (tiles + resident - 1) / resident;
    chunk = (chunk + REFINE_WARPS - 1) / REFINE_WARPS * REFINE_WARPS;
    const int grid = emb_grid(tiles, (int)(chunk > 0 ? chunk : REFINE_WARPS));
    if (chunk < REFINE_WARPS) chunk = REFINE_WARPS;
    const size_t smem = REFINE_WARPS * sizeof(RefWarp);
    if (td.w && nw <= REFINE_SM_WORDS) {
        EMB_LAUNCH((k_refine<true>), grid, 32 * REFINE_WARPS, smem + (size_t)nw * sizeof(uint64_t), s)
        (rec, T, g, dil, lk, flags, td.w, (int)(2 * nw), chunk, Q);
    } else {
        EMB_LAUNCH((k_refine<false>), grid, 32 * REFINE_WARPS, smem, s)(rec, T, g, dil, lk, flags, td.w, 0, chunk, Q);
    }
    if (Q.cap) EMB_LAUNCH((k_refine_big), EMB_BIG_GRID, EMB_BIG_BLOCK, 0, s)(rec, g, dil, lk, flags, td, Q);
    if (td.w)
        EMB_LAUNCH((k_refine_flags), emb_grid(lv.n, 256), 256, 0, s)(lv.key, lv.n, lv.d_n, td.w, g.nb, flags);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}

extern "C" emb_status emb_refine_flags(emb_forest f, emb_bins b, int32_t level, int32_t band, uint8_t *d_flags,
                                       void *stream)
{
    if (!f || !b || band < 1 || band > (1 << 20)) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    if (b->f != f || level < 0 || level > f->top || level >= f->max_level) return EMB_ERR_STATE;
    const EmbLevel &lv = f->lv[level];
    if (lv.n == 0) return EMB_OK;
    if (!d_flags) return EMB_ERR_BAD_INPUT;
    long long dil = emb_refine_dilation(f, level, band);
    if (dil < 0) return EMB_ERR_RANGE;
    cudaStream_t s = emb_stream(stream);
    // the flagged bits, and the chunk queue where a triangle may meet more than
    // EMB_BIG_ITEMS dilated blocks: [-dil, extent + dil] spans at most this many an axis, and the level has nb
    const emb_mesh m = b->m;
    const LevelGeom g = level_geom(f, level);
    const long long most = ((m->ext + 2 * dil) >> g.lW) + 2, span = most < g.nb ? most : g.nb;
    EmbBigQ Q = emb_bigq(m->T);
    if (emb_mesh_big(m, span, span, span)) Q.cap = (uint32_t)emb_bigq_capacity(m->T);
    const int64_t nw = emb_bitmap_words(lv.nb_axis);
    const size_t a_bits = ((size_t)(nw + 1) * sizeof(unsigned long long) + 255) & ~(size_t)255;
    char *scratch = nullptr;
    EMB_CUDA_TRY(emb_malloc_async(&scratch, a_bits + (size_t)Q.cap * sizeof(uint2), s));
    Q.n = (unsigned long long *)scratch + nw;
    Q.q = (uint2 *)(scratch + a_bits);
    const emb_status rc = emb_enq_refine(m->rec, m->T, g, dil, lv, d_flags,
                                         nw > 0 ? (unsigned long long *)scratch : nullptr, Q, s);
    cudaFreeAsync(scratch, s);
    return rc;
}

// ---------------------------------------------------------------------------
// the paper's refinement rules (Sec. 3.4, "Refinement Flagging and Propagation")
// ---------------------------------------------------------------------------
// Block classes from the masks: solid (a solid cell), fully fluid (none).  cls bit 0:
// solid; bit 1: solid-boundary (solid with a fully fluid neighbour of the level);
// bit 2: eligible (every in-domain neighbour position holds a block of the level,
// always at the root: refining a block on the refinement interface breaks 2:1).
// The solid-boundary blocks are the first marks.
__global__ void k_pf_classify(const uint64_t *__restrict__ key, const uint64_t *__restrict__ mask,
                              const int32_t *__restrict__ nbr, int64_t n, int64_t nb, int root,
                              uint8_t *__restrict__ cls, uint8_t *__restrict__ marks)
{
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    const uint64_t k = key[b];
    const int64_t bx = (int64_t)(k & EMB_KEY_MASK), by = (int64_t)((k >> EMB_KEY_BITS) & EMB_KEY_MASK),
                  bz = (int64_t)(k >> (2 * EMB_KEY_BITS));
    const bool solid = mask[b] != 0;
    bool eligible = true, fluid_nbr = false;
    for (int d = 1; d < 27; ++d) {
        int cx, cy, cz;
        emb_dir(d, cx, cy, cz);
        const int64_t x = bx + cx, y = by + cy, z = bz + cz;
        if (x < 0 || y < 0 || z < 0 || x >= nb || y >= nb || z >= nb) continue;
        const int32_t j = nbr[b * 26 + d - 1];
        if (j < 0) {
            if (!root) eligible = false;
        } else if (mask[j] == 0) {
            fluid_nbr = true;
        }
    }
    const bool sb = solid && fluid_nbr;
    cls[b] = (uint8_t)((solid ? 1 : 0) | (sb ? 2 : 0) | (eligible ? 4 : 0));
    marks[b] = (uint8_t)(sb && eligible);
}

// One propagation step: out = in, plus every eligible block in scope next to a block
// whose `want` bits are set in cls (the adjacency step: want = solid-boundary, every
// class in scope) or that is marked in `in` (the propagation rounds: want = 0, scope =
// fully fluid blocks, and solid ones in the first round).
__global__ void k_pf_step(const int32_t *__restrict__ nbr, int64_t n, const uint8_t *__restrict__ cls, int want,
                          int solid_in_scope, const uint8_t *__restrict__ in, uint8_t *__restrict__ out)
{
    const int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= n) return;
    uint8_t m = in[b];
    const uint8_t c = cls[b];
    if (!m && (c & 4) && (!(c & 1) || solid_in_scope)) {
        for (int d = 0; d < 26 && !m; ++d) {
            const int32_t j = nbr[b * 26 + d];
            if (j >= 0 && (want ? (cls[j] & want) : in[j])) m = 1;
        }
    }
    out[b] = m;
}

extern "C" emb_status emb_refine_flags_paper(emb_forest f, int32_t level, double d_spec, uint8_t *d_flags, void *stream)
{
    if (!f || !(d_spec >= 0.0) || d_spec > 1e6) return EMB_ERR_BAD_INPUT;
    EMB_SETTLE(f);
    if (level < 0 || level != f->top || level >= f->max_level) return EMB_ERR_STATE;
    EmbLevel &lv = f->lv[level];
    if (!lv.mask_valid) return EMB_ERR_STATE;
    if (lv.n == 0) return EMB_OK;
    if (!d_flags) return EMB_ERR_BAD_INPUT;
    cudaStream_t s = emb_stream(stream);
    // Eq. N_prop: 1 + floor(2^-L d_spec / (sqrt(2) Dx_{b,L})), Dx_{b,L} = 4 Dx_L = 1 / (R 2^L)
    // for d_spec in units of the unit domain: the 2^L factors cancel
    const double np_d = floor((d_spec * (double)f->R) / sqrt(2.0));
    if (np_d > 1e6) return EMB_ERR_BAD_INPUT;
    const int nprop = 1 + (int)np_d;
    emb_status rc = emb_build_neighbors(lv, s);
    if (rc != EMB_OK) return rc;
    uint8_t *cls = nullptr, *tmp = nullptr;
    EMB_CUDA_TRY(emb_malloc_async(&cls, lv.n, s));
    EMB_CUDA_TRY(emb_malloc_async(&tmp, lv.n, s));
    const int grid = emb_grid(lv.n, 256);
    EMB_LAUNCH((k_pf_classify), grid, 256, 0, s)(lv.key, lv.mask, lv.nbr, lv.n, lv.nb_axis, level == 0 ? 1 : 0, cls,
                                                 d_flags);
    // blocks next to the solid boundary (both classes), then the rounds, ping-pong
    EMB_LAUNCH((k_pf_step), grid, 256, 0, s)(lv.nbr, lv.n, cls, 2, 1, d_flags, tmp);
    uint8_t *a = tmp, *b = d_flags;
    for (int r = 0; r < nprop; ++r) {
        EMB_LAUNCH((k_pf_step), grid, 256, 0, s)(lv.nbr, lv.n, cls, 0, r == 0 ? 1 : 0, a, b);
        uint8_t *t = a;
        a = b;
        b = t;
    }
    if (a != d_flags) EMB_CUDA_TRY(cudaMemcpyAsync(d_flags, a, lv.n, cudaMemcpyDeviceToDevice, s));
    EMB_CUDA_TRY(cudaGetLastError());
    EMB_CUDA_TRY(cudaFreeAsync(cls, s));
    EMB_CUDA_TRY(cudaFreeAsync(tmp, s));
    return EMB_OK;
}
