// Numbering of the indexed mesh output's vertices: one vertex per crossing
// lattice edge (the optional vert_xyz / tri_idx outputs of gh_mesh).  Marching
// Cubes, which runs next and holds its cells' corner entries, writes the
// triangles' indices from it.
//
// A lattice edge leaves its lower end point A along +x, +y or +z and crosses
// the surface when f(A) and f(B) differ in sign (inside <=> f < 0, the tie
// rule of the Marching Cubes pass).  The four cells around a crossing edge
// are sign-change cells, which the hopper marks (Algorithm 1 polygonizes
// every cell the surface passes through), so both end points are in the
// vertex list the pipeline already holds (vkey: grouped by vertical lattice
// line, c ascending) together with their final values (vval).
//
// Numbering: vertex-list order of the lower end point, then axis order x, y,
// z.  It depends only on the set of crossing edges, not on the order in which
// the Marching Cubes kernel emits its triangles.  Vertex positions use the
// Marching Cubes interpolation t = f(A) / (f(A) - f(B)) from A with the same
// operations, so they are bit-identical to the triangle soup's.
#include "gh_internal.cuh"
#include "lookback.cuh"

namespace gh {

namespace {

// index of lattice point c of vertical line `line` in the vertex list, or -1
__device__ __forceinline__ long long find_point(const Scratch &s, uint32_t line, uint32_t c) {
    uint32_t lo = s.lineoff[line], hi = s.lineoff[line + 1];
    if (lo >= hi) return -1;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if ((uint32_t)(s.vkey[mid] >> 32) <= c) lo = mid; else hi = mid;
    }
    return (uint32_t)(s.vkey[lo] >> 32) == c ? (long long)lo : -1;
}

// A list entry: its lattice coordinates and value, the value fn[ax] of the
// upper end point of its edge along each axis, and the mask m of the axes whose
// edge crosses.  hint[ax]: where the upper end point along x and y is looked
// for first (one past the entry before's); returned for the next entry.
struct Edges {
    uint32_t a, b, c;
    float f, fn[3];
    int m;
};

__device__ __forceinline__ Edges edges_of(const GridP &g, const Scratch &s, unsigned long long v, unsigned long long V,
                                          long long (&hint)[2]) {
    const uint32_t N = (uint32_t)g.N, N1 = N + 1;
    const unsigned long long key = s.vkey[v];
    const uint32_t line = (uint32_t)(key & 0xFFFFFFFFull);
    Edges e;
    e.c = (uint32_t)(key >> 32);
    e.a = line / N1;
    e.b = line - e.a * N1;
    e.f = s.vval[v];
    e.fn[0] = e.fn[1] = e.fn[2] = 0.f;
    e.m = 0;
    const bool neg = e.f < 0.f;
#pragma unroll
    for (int ax = 0; ax < 2; ++ax) {
        if ((ax == 0 ? e.a : e.b) >= N) {
            hint[ax] = -1;
            continue;
        }
        const uint32_t nline = ax == 0 ? line + N1 : line + 1u;
        const unsigned long long want = (unsigned long long)nline | ((unsigned long long)e.c << 32);
        long long nb = hint[ax];
        if (nb < 0 || (unsigned long long)nb >= V || s.vkey[nb] != want) nb = find_point(s, nline, e.c);
        hint[ax] = nb >= 0 ? nb + 1 : -1;
        if (nb >= 0) {
            e.fn[ax] = s.vval[nb];
            if ((e.fn[ax] < 0.f) != neg) e.m |= 1 << ax;
        }
    }
    if (v + 1 < V && s.vkey[v + 1] == key + (1ull << 32)) {  // the next entry: the upper neighbour along z, if it is one
        e.fn[2] = s.vval[v + 1];
        if ((e.fn[2] < 0.f) != neg) e.m |= 4;
    }
    return e;
}

// The positions of an entry's vertices, numbered from id on.
__device__ __forceinline__ void put_vertices(const GridP &g, const gh_mesh &out, const Edges &e, unsigned long long id) {
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        if (!(e.m & (1 << ax))) continue;
        const float tt = e.f / (e.f - e.fn[ax]);
        float px = fmaf((float)e.a, g.h, g.lo[0]);
        float py = fmaf((float)e.b, g.h, g.lo[1]);
        float pz = fmaf((float)e.c, g.h, g.lo[2]);
        if (ax == 0) px = fmaf(tt, g.h, px);
        else if (ax == 1) py = fmaf(tt, g.h, py);
        else pz = fmaf(tt, g.h, pz);
        if (id < (unsigned long long)out.capacity_verts) {
            out.vert_xyz[3 * id] = px;
            out.vert_xyz[3 * id + 1] = py;
            out.vert_xyz[3 * id + 2] = pz;
        }
        ++id;
    }
}

// One call: count, number and emit in one pass.  Blocks take tiles of 1,024
// entries; a thread has four consecutive ones, whose neighbours mostly follow
// each other too, so that only the first is searched for.  (A counting pass, a
// two-pass scan and an emitting pass took 61 us for 1.6 M entries, this 55, and
// at 10 k entries three launches less count more.)
constexpr int EDGE_T = 256, EDGE_E = 4, EDGE_TILE = EDGE_T * EDGE_E;

__global__ void __launch_bounds__(EDGE_T) k_edges(GridP g, Scratch s, gh_mesh out) {
    __shared__ uint32_t wsum[EDGE_T / 32], base_s;
    __shared__ unsigned long long tile_s;
    // one decision for the block: another block's wait may run out at any time (which
    // leaves the list as readable as it was)
    if (__syncthreads_or((s.ctr->flags & STOP_FLAGS) != 0ull)) return;
    const unsigned long long V = s.ctr->verts;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (;;) {
        if (threadIdx.x == 0) tile_s = atomicAdd(&s.ctr->tick[2], 1ull);
        __syncthreads();
        const unsigned long long tile = tile_s, v0 = tile * EDGE_TILE + (unsigned long long)threadIdx.x * EDGE_E;
        if (tile * EDGE_TILE >= V) return;
        Edges e[EDGE_E];
        long long hint[2] = {-1, -1};
        uint32_t cnt = 0;
#pragma unroll
        for (int k = 0; k < EDGE_E; ++k) {
            e[k].m = 0;
            if (v0 + k < V) {
                e[k] = edges_of(g, s, v0 + k, V, hint);
                s.vflag[v0 + k] = (uint8_t)e[k].m;
                cnt += (uint32_t)__popc(e[k].m);
            }
        }
        uint32_t x = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[wid] = x;
        __syncthreads();
        uint32_t tot = 0, wb = 0;
        for (int q = 0; q < EDGE_T / 32; ++q) {
            if (q < wid) wb += wsum[q];
            tot += wsum[q];
        }
        if (wid == 0) {
            const uint32_t p = lb_prefix(s.lbe, s.lb[0], (long long)tile, tot, s.ctr, false);
            if (lane == 0) base_s = p;
        }
        __syncthreads();
        uint32_t id = base_s + wb + x - cnt;
#pragma unroll
        for (int k = 0; k < EDGE_E; ++k) {
            if (v0 + k >= V) break;
            s.ebase[v0 + k] = id;
            if (out.vert_xyz && e[k].m) put_vertices(g, out, e[k], id);
            id += (uint32_t)__popc(e[k].m);
            if (v0 + k == V - 1) s.ctr->mesh_verts = id;
        }
        __syncthreads();  // tile_s and the sums are rewritten
    }
}

// Batches: counted, scanned (two passes) and emitted over all items, grid
// strides without tickets.  Per entry the crossing mask goes into vflag and its
// population into rlist, whose refinement list is no longer needed.
__global__ void __launch_bounds__(256) k_edge_count_b(const Item *__restrict__ items, int n) {
    const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    for (int b = 0; b < n; ++b) {
        const Item &it = items[b];
        if (!wants_index(it.out) || (it.s.ctr->flags & STOP_FLAGS)) continue;
        const unsigned long long V = it.s.ctr->verts;
        for (unsigned long long v = t; v < V; v += (unsigned long long)gridDim.x * blockDim.x) {
            long long hint[2] = {-1, -1};
            const Edges e = edges_of(it.g, it.s, v, V, hint);
            it.s.vflag[v] = (uint8_t)e.m;
            it.s.rlist[v] = (uint32_t)__popc(e.m);
        }
    }
}

__global__ void __launch_bounds__(256) k_emit_vertices_b(const Item *__restrict__ items, int n) {
    const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    for (int b = 0; b < n; ++b) {
        const Item &it = items[b];
        if (!it.out.vert_xyz || (it.s.ctr->flags & STOP_FLAGS)) continue;
        const unsigned long long V = it.s.ctr->verts;
        for (unsigned long long v = t; v < V; v += (unsigned long long)gridDim.x * blockDim.x) {
            if (!it.s.vflag[v]) continue;
            long long hint[2] = {-1, -1};
            put_vertices(it.g, it.out, edges_of(it.g, it.s, v, V, hint), it.s.ebase[v]);
        }
    }
}

}  // namespace

long long lbe_words(long long nverts) { return nverts / EDGE_TILE + 1; }

void launch_index_mesh(const GridP &g, Scratch &s, const gh_mesh &out, int nsm, cudaStream_t st) {
    k_edges<<<nsm * 4, EDGE_T, 0, st>>>(g, s, out);
}

void launch_index_mesh_b(const Item *items, int n, int nsm, cudaStream_t st) {
    k_edge_count_b<<<nsm * 8, 256, 0, st>>>(items, n);
    launch_index_scan_b(items, n, nsm, st);
    k_emit_vertices_b<<<nsm * 8, 256, 0, st>>>(items, n);
}

}  // namespace gh
