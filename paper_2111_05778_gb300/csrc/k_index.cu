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

namespace gh {

namespace {

constexpr unsigned long long STOPF = FLAG_MARK_OVERFLOW | FLAG_VERT_OVERFLOW;

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

// Walks the list: visit(v, a, b, c, f, fn, m) for each entry v: its lattice
// coordinates and value, the value fn[ax] of the upper end point of its edge
// along each axis, and the mask m of the axes whose edge crosses.
template <typename F>
__device__ __forceinline__ void walk_edges(const GridP &g, const Scratch &s, unsigned long long t0,
                                           unsigned long long stride, F visit) {
    const unsigned long long V = s.ctr->verts;
    const uint32_t N = (uint32_t)g.N, N1 = N + 1;
    for (unsigned long long v = t0; v < V; v += stride) {
        const unsigned long long key = s.vkey[v];
        const uint32_t line = (uint32_t)(key & 0xFFFFFFFFull), c = (uint32_t)(key >> 32);
        const uint32_t a = line / N1, b = line - a * N1;
        const float f = s.vval[v];
        const bool neg = f < 0.f;
        const long long nx = a < N ? find_point(s, line + N1, c) : -1;
        const long long ny = b < N ? find_point(s, line + 1, c) : -1;
        const unsigned long long kz = v + 1 < V ? s.vkey[v + 1] : ~0ull;  // upper neighbour along z, if it is one
        const long long nz = (uint32_t)(kz & 0xFFFFFFFFull) == line && (uint32_t)(kz >> 32) == c + 1u ? (long long)v + 1 : -1;
        const long long nb[3] = {nx, ny, nz};
        float fn[3] = {0.f, 0.f, 0.f};
        int m = 0;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax)
            if (nb[ax] >= 0) {
                fn[ax] = s.vval[nb[ax]];
                if ((fn[ax] < 0.f) != neg) m |= 1 << ax;
            }
        visit(v, a, b, c, f, fn, m);
    }
}

// per list entry: the crossing mask (into vflag) and its population (into
// rlist, whose refinement list is no longer needed)
__device__ __forceinline__ void edge_count(const GridP &g, const Scratch &s, unsigned long long t0,
                                           unsigned long long stride) {
    walk_edges(g, s, t0, stride, [&](unsigned long long v, uint32_t, uint32_t, uint32_t, float, const float(&)[3], int m) {
        s.vflag[v] = (uint8_t)m;
        s.rlist[v] = (uint32_t)__popc(m);
    });
}

__device__ __forceinline__ void emit_vertices(const GridP &g, const Scratch &s, const gh_mesh &out,
                                              unsigned long long t0, unsigned long long stride) {
    walk_edges(g, s, t0, stride, [&](unsigned long long v, uint32_t a, uint32_t b, uint32_t c, float fa,
                                     const float(&fn)[3], int m) {
        if (!m) return;
        unsigned long long id = s.ebase[v];
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
            if (!(m & (1 << ax))) continue;
            const float tt = fa / (fa - fn[ax]);
            float px = fmaf((float)a, g.h, g.lo[0]);
            float py = fmaf((float)b, g.h, g.lo[1]);
            float pz = fmaf((float)c, g.h, g.lo[2]);
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
    });
}

__global__ void __launch_bounds__(256) k_emit_vertices(GridP g, Scratch s, gh_mesh out) {
    if (s.ctr->flags & STOPF) return;
    const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    emit_vertices(g, s, out, t, (unsigned long long)gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(256) k_emit_vertices_b(const Item *__restrict__ items, int n) {
    const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    for (int b = 0; b < n; ++b) {
        const Item &it = items[b];
        if (!it.out.vert_xyz || (it.s.ctr->flags & STOPF)) continue;
        emit_vertices(it.g, it.s, it.out, t, (unsigned long long)gridDim.x * blockDim.x);
    }
}

__global__ void __launch_bounds__(256) k_edge_count(GridP g, Scratch s) {
    if (s.ctr->flags & STOPF) return;
    const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    edge_count(g, s, t, (unsigned long long)gridDim.x * blockDim.x);
}

__global__ void __launch_bounds__(256) k_edge_count_b(const Item *__restrict__ items, int n) {
    const unsigned long long t = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x;
    for (int b = 0; b < n; ++b) {
        const Item &it = items[b];
        if (!wants_index(it.out) || (it.s.ctr->flags & STOPF)) continue;
        edge_count(it.g, it.s, t, (unsigned long long)gridDim.x * blockDim.x);
    }
}

}  // namespace

void launch_index_mesh(const GridP &g, Scratch &s, const gh_mesh &out, int nsm, cudaStream_t st) {
    const long long n = s.cap_verts;
    long long nb = (n + 255) / 256;
    if (nb > nsm * 8) nb = nsm * 8;
    k_edge_count<<<(int)nb, 256, 0, st>>>(g, s);
    scan_u32_dev(s.rlist, n, &s.ctr->verts, s.ebase, s.ebsum, &s.ctr->mesh_verts, s.ctr, st);
    if (out.vert_xyz) k_emit_vertices<<<(int)nb, 256, 0, st>>>(g, s, out);
}

void launch_index_mesh_b(const Item *items, int n, int nsm, cudaStream_t st) {
    k_edge_count_b<<<nsm * 8, 256, 0, st>>>(items, n);
    launch_index_scan_b(items, n, nsm, st);
    k_emit_vertices_b<<<nsm * 8, 256, 0, st>>>(items, n);
}

}  // namespace gh
