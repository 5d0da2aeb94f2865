// Geometry input (Sec. 3.1): snapped vertex check, integer frame, 48-byte
// triangle records, and the watertightness check on the GPU.
#include <limits.h>
#include <stdlib.h>

#include "emb_edges.cuh"
#include "emb_internal.cuh"

#define MESH_ERR_ID 1         // vertex id out of range
#define MESH_ERR_SNAP 2       // coordinate not a multiple of 2^-20 inside (0,1)
#define MESH_ERR_DUP_EDGE 4   // a directed edge occurs twice
#define MESH_ERR_OPEN_EDGE 8  // a directed edge has no reverse
#define MESH_ERR_DEG_EDGE 16  // an edge joins a vertex to itself
#define MESH_ERR_TABLE 32     // the overflow table of edges is full: once more with a larger one

// Edge table of the watertight check.  An undirected edge {lo, hi} is the word
// lo << 33 | hi << 2 | directions seen (1: lo -> hi, 2: hi -> lo); 0 is a free slot.  It
// lives in one of the EDGE_SLOTS slots of one of its vertices (which of the two, a hash
// decides: 3 edges a vertex on average), and when those are taken by other edges, in an
// overflow table probed by hash.  Neighbouring triangles have neighbouring vertex ids in
// most meshes, so the slots they touch are neighbours too; a table addressed by hash alone
// missed the L2 on every access and held every directed edge twice as sparsely (7.2M
// triangles: records 100 us, clear + insert + look-up of the reverse 1150 us; now 434 us
// for all, and 25 for the clear; with triangles and vertices shuffled a mesh of 7.2M takes 790
// us in all instead of 1380, of 1.0M 160 instead of 161).  Sizes: emb_edges.cuh.  The mesh is
// closed and
// oriented iff no direction is seen twice and every edge is completed by its other one:
// 3T/2 completions.
#define EDGE_SLOTS 4
#define EDGE_COUNTERS 64  // completions, spread over the CTAs
struct EdgeTable {
    unsigned long long *slot, *over;  // V x EDGE_SLOTS (NULL: overflow only); cap (a power of two)
    uint64_t cap, probes;             // probes of the overflow table before it counts as full
    uint32_t *done;                   // EDGE_COUNTERS; NULL: no check
    int *err;                         // the error word: nobody goes on probing a table that is full
};

// 0: p holds another edge; 1: entered or repeated; 2: completed
__device__ __forceinline__ int edge_try(unsigned long long *p, unsigned long long have, unsigned long long key,
                                        unsigned long long bit, int &bad)
{
    if (have == 0) {
        have = atomicCAS(p, 0ull, key | bit);
        if (have == 0) return 1;
    }
    if ((have ^ key) >> 2) return 0;
    const unsigned long long old = atomicOr(p, bit);
    if (old & bit) {
        bad |= MESH_ERR_DUP_EDGE;
        return 1;
    }
    return 2;
}

__device__ __forceinline__ bool edge_enter(const EdgeTable &E, uint32_t a, uint32_t b, int &bad)
{
    const uint32_t lo = min(a, b), hi = max(a, b);
    const unsigned long long key = (unsigned long long)lo << 33 | (unsigned long long)hi << 2, bit = a < b ? 1 : 2;
    if (E.slot) {
        unsigned long long *s = E.slot + (int64_t)EDGE_SLOTS * (((lo ^ hi) * 2654435761u) >> 31 ? lo : hi);
        // the whole bucket with two loads from the L2 (slots only ever gain bits)
        const ulonglong2 v0 = __ldcg((const ulonglong2 *)s), v1 = __ldcg((const ulonglong2 *)s + 1);
        const unsigned long long v[EDGE_SLOTS] = {v0.x, v0.y, v1.x, v1.y};
#pragma unroll
        for (int i = 0; i < EDGE_SLOTS; ++i) {
            const int r = edge_try(s + i, v[i], key, bit, bad);
            if (r) return r == 2;
        }
    }
    const uint64_t m = E.cap - 1;
    uint64_t p = emb_hash_mix(key) & m;
    for (uint64_t it = 0; it < E.probes; ++it) {
        const int r = edge_try(E.over + p, __ldcg(E.over + p), key, bit, bad);
        if (r) return r == 2;
        p = (p + 1) & m;
        if ((it & 15) == 15 && (*(volatile int *)E.err & MESH_ERR_TABLE)) return false;
    }
    atomicOr(E.err, MESH_ERR_TABLE);
    return false;
}

// Records, the largest extent, and with E.done the edges (a thread per triangle).
__global__ void k_mesh_records(const float *__restrict__ verts, const int32_t *__restrict__ tris, int64_t V, int64_t T,
                               int32_t r_o, int4 *__restrict__ rec, EdgeTable E, int *ext, int *err)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    int bad = 0;
    uint32_t done = 0;
    // few warps raise the extent: what it was on entry, read while the vertices are fetched
    const int seen = *(volatile int *)ext;
    int lo[3] = {INT_MAX, INT_MAX, INT_MAX}, hi[3] = {0, 0, 0};
    if (t < T) {
        int32_t vid[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int32_t id = vid[k] = tris[3 * t + k];
            if (id < 0 || (int64_t)id >= V) {
                bad |= MESH_ERR_ID;
                rec[3 * t + k] = make_int4(0, 0, 0, -1);
                continue;
            }
            int c[3];
#pragma unroll
            for (int d = 0; d < 3; ++d) {
                float m = verts[3 * (int64_t)id + d] * 1048576.0f;  // exact: power-of-two scaling
                if (!(m > 0.0f && m < 1048576.0f && m == truncf(m))) bad |= MESH_ERR_SNAP;
                c[d] = (int)m * r_o;
                lo[d] = min(lo[d], c[d]);
                hi[d] = max(hi[d], c[d]);
            }
            rec[3 * t + k] = make_int4(c[0], c[1], c[2], id);
        }
        if (E.done && !(bad & MESH_ERR_ID)) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const uint32_t a = (uint32_t)vid[k], b = (uint32_t)vid[(k + 1) % 3];
                if (a == b) bad |= MESH_ERR_DEG_EDGE;
                else if (edge_enter(E, a, b, bad)) ++done;
            }
        }
        if (bad) atomicOr(err, bad);
    }
    int e = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) e = max(e, hi[d] - lo[d]);
    e = __reduce_max_sync(0xffffffffu, t < T && !(bad & MESH_ERR_ID) ? e : 0);
    if ((threadIdx.x & 31) == 0 && e > seen) atomicMax(ext, e);
    if (E.done) {
        done = __reduce_add_sync(0xffffffffu, done);
        if ((threadIdx.x & 31) == 0 && done) atomicAdd(E.done + blockIdx.x % EDGE_COUNTERS, done);
    }
}

// New vertex positions for the same triangles: corner j of triangle t takes the
// coordinates of its vertex id (kept in the record's fourth word).  A coordinate
// that is not a multiple of 2^-20 inside (0,1) leaves the record unchanged and
// raises EMB_ERR_BAD_INPUT in the device status word.
__global__ void k_mesh_move(const float *__restrict__ verts, int64_t V, int64_t T, int32_t r_o, int4 *__restrict__ rec,
                            int *st)
{
    const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 3 * T) return;
    const int4 r = rec[e];
    if (r.w < 0 || (int64_t)r.w >= V) {
        emb_set_status(st, EMB_ERR_BAD_INPUT);
        return;
    }
    int c[3];
    bool ok = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const float m = verts[3 * (int64_t)r.w + d] * 1048576.0f;  // exact: power-of-two scaling
        if (!(m > 0.0f && m < 1048576.0f && m == truncf(m))) ok = false;
        c[d] = ok ? (int)m * r_o : 0;
    }
    if (!ok) {
        emb_set_status(st, EMB_ERR_BAD_INPUT);
        return;
    }
    rec[e] = make_int4(c[0], c[1], c[2], r.w);
}

extern "C" emb_status emb_mesh_create(const float *d_verts, const int32_t *d_tris, int64_t V, int64_t T, int32_t R,
                                      int32_t check_watertight, void *stream, emb_mesh *out)
{
    if (!out || !d_verts || !d_tris || V < 3 || T < 1 || R < 1 || V > 2147483647ll || T > (1ll << 30))
        return EMB_ERR_BAD_INPUT;
    *out = nullptr;
    int32_t r_o = R, k = 0;
    while ((r_o & 1) == 0) {
        r_o >>= 1;
        ++k;
    }
    if (k > 17 || (int64_t)r_o * (1 << 20) >= (1ll << 25)) return EMB_ERR_RANGE;
    cudaStream_t s = emb_stream(stream);
    emb_mesh m = (emb_mesh)calloc(1, sizeof(emb_mesh_s));
    if (!m) return EMB_ERR_CUDA;
    m->R = R;
    m->r_o = r_o;
    m->k = k;
    m->V = V;
    m->T = T;
    cudaGetDevice(&m->device);
    // error word, completion counters and extent, then the edge table: cleared together
    char *scratch = nullptr;
    emb_status rc = EMB_OK;
    // its copy on the host, in page-locked memory where a slot is free
    uint32_t here[1 + EDGE_COUNTERS + 1] = {0}, *head = here;
    static_assert(sizeof(here) <= EMB_RB_WORDS * sizeof(uint64_t), "a read-back slot holds the head");
    uint64_t *rb = nullptr;
    cudaEvent_t rb_ev;
    const int slot = emb_readback_acquire(&rb, &rb_ev);
    if (slot >= 0) head = (uint32_t *)rb;
    const size_t a_head = 512;
    // records and scratch from the library's pool (stream-ordered on s; the
    // synchronisation below completes them before the mesh is used on any stream)
    if (emb_malloc_async(&m->rec, (size_t)T * 3 * sizeof(int4), s) != cudaSuccess) {
        rc = EMB_ERR_CUDA;
        goto done;
    }
    for (int attempt = 0;; ++attempt) {
        const EdgePlan plan = emb_edge_plan(V, T, attempt);
        const bool slots = check_watertight && plan.slots;
        const uint64_t cap = plan.cap;
        const size_t a_slot = slots ? (size_t)V * EDGE_SLOTS * sizeof(unsigned long long) : 0,
                     a_all = a_head + a_slot + (check_watertight ? cap * sizeof(unsigned long long) : 0);
        if (emb_malloc_async(&scratch, a_all, s) != cudaSuccess) {
            rc = EMB_ERR_CUDA;
            goto done;
        }
        cudaMemsetAsync(scratch, 0, a_all, s);
        const EdgeTable E = {slots ? (unsigned long long *)(scratch + a_head) : nullptr,
                             (unsigned long long *)(scratch + a_head + a_slot), cap, plan.all ? cap : EDGE_PROBES,
                             check_watertight ? (uint32_t *)scratch + 1 : nullptr, (int *)scratch};
        EMB_LAUNCH((k_mesh_records), emb_grid(T, 256), 256, 0, s)(d_verts, d_tris, V, T, r_o, m->rec, E,
                                                                      (int *)scratch + 1 + EDGE_COUNTERS, (int *)scratch);
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(head, scratch, sizeof(here), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            (slot >= 0 && cudaEventRecord(rb_ev, s) != cudaSuccess) ||
            cudaStreamSynchronize(s) != cudaSuccess) {
            rc = EMB_ERR_CUDA;
            goto done;
        }
        if (!(head[0] & MESH_ERR_TABLE) || plan.all) break;
        cudaFreeAsync(scratch, s);
        scratch = nullptr;
    }
    if (check_watertight) {
        int64_t closed = 0;
        for (int i = 0; i < EDGE_COUNTERS; ++i) closed += head[1 + i];
        if (2 * closed != 3 * T) head[0] |= MESH_ERR_OPEN_EDGE;
    }
    m->ext = (int32_t)head[1 + EDGE_COUNTERS];
    m->ext_known = true;
    if (head[0] & (MESH_ERR_ID | MESH_ERR_SNAP)) rc = EMB_ERR_BAD_INPUT;
    else if (head[0]) rc = EMB_ERR_NOT_WATERTIGHT;
done:
    emb_readback_release(slot);
    if (scratch) cudaFreeAsync(scratch, s);
    if (rc != EMB_OK) {
        emb_mesh_destroy(m);
        return rc;
    }
    *out = m;
    return EMB_OK;
}

extern "C" void emb_mesh_destroy(emb_mesh m)
{
    if (!m) return;
    if (m->rec) cudaFree(m->rec);
    free(m);
}

extern "C" emb_status emb_mesh_update(emb_mesh m, const float *d_verts, int64_t V, void *stream)
{
    if (!m || !d_verts || V != m->V) return EMB_ERR_BAD_INPUT;
    int *st = emb_status_word();
    if (!st) return EMB_ERR_CUDA;
    cudaStream_t s = emb_stream(stream);
    m->ext_known = false;
    EMB_LAUNCH((k_mesh_move), emb_grid(3 * m->T, 256), 256, 0, s)(d_verts, V, m->T, m->r_o, m->rec, st);
    EMB_CUDA_TRY(cudaGetLastError());
    return EMB_OK;
}
