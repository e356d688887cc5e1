// stream_node.cuh -- per-node and per-chunk pieces shared by the two
// stream-collide kernels (register-pipelined k_stream.cu, staged k_staged.cu):
// domain geometry loads, flag-word loads, the moments of nodes that change
// side, and the parts of one V-node chunk (pulled vectors, bounce-back, Zou-He
// and corner patches, collision, stores).  arXiv:2006.12910 Sec. 2 Eqs. e.LB1 /
// e.LB2, Sec. 3 (halfway bounce-back, Zou-He), Sec. 4 (noise), Sec. 5 (tau*).
#pragma once
#include <cstddef>

#include "kernels.h"
#include "collide_fix.cuh"
#include "lbm_dev.cuh"

namespace lbmk {

// Geometry of one domain for a work item, read with 16-byte loads.
struct Geo {
    int nx, ny, pitch, flags;
    int64_t off, plane, node_off, mask_off, item_off;
    int spr;  // warp segments per row
    uint32_t magic;  // multiply-high reciprocal of spr, or 0
};
static_assert(offsetof(DomDev, ny) == offsetof(DomDev, nx) + 4 && offsetof(DomDev, flags) == offsetof(DomDev, nx) + 12 &&
                  offsetof(DomDev, nx) % 16 == 0, "nx..flags must form one 16-byte block");
static_assert(offsetof(DomDev, plane) == offsetof(DomDev, off) + 8 && offsetof(DomDev, off) % 16 == 0 &&
                  offsetof(DomDev, mask_off) == offsetof(DomDev, node_off) + 8 && offsetof(DomDev, node_off) % 16 == 0 &&
                  offsetof(DomDev, seg_per_row) == offsetof(DomDev, item_off) + 8 && offsetof(DomDev, item_off) % 16 == 0,
              "64-bit offsets must pair into 16-byte blocks");
__device__ __forceinline__ Geo load_geo(const DomDev& D) {
    const int4 a = __ldg(reinterpret_cast<const int4*>(&D.nx));
    const longlong2 b = __ldg(reinterpret_cast<const longlong2*>(&D.off));
    const longlong2 c = __ldg(reinterpret_cast<const longlong2*>(&D.node_off));
    const longlong2 e = __ldg(reinterpret_cast<const longlong2*>(&D.item_off));
    Geo G;
    G.nx = a.x; G.ny = a.y; G.pitch = a.z; G.flags = a.w;
    G.off = b.x; G.plane = b.y; G.node_off = c.x; G.mask_off = c.y; G.item_off = e.x;
    G.spr = (int)(uint32_t)(uint64_t)e.y;
    G.magic = 0u;
    return G;
}
// The same from a descriptor held in the launch parameters (no memory loads).
__device__ __forceinline__ Geo param_geo(const DomDev& D) {
    Geo G;
    G.nx = D.nx; G.ny = D.ny; G.pitch = D.pitch; G.flags = D.flags;
    G.off = D.off; G.plane = D.plane; G.node_off = D.node_off; G.mask_off = D.mask_off; G.item_off = D.item_off;
    G.spr = D.seg_per_row;
    G.magic = D.spr_magic;
    return G;
}
// Row of a domain-local work item.
__device__ __forceinline__ int item_row(const Geo& G, int local) {
    return G.magic ? (int)__umulhi((uint32_t)local, G.magic) : local / G.spr;
}

// Rows that row y pulls from: y -/+ 1, wrapped when periodic in y; with y
// walls y = -1 and y = ny are ghost rows, whose values bounce-back replaces.
__device__ __forceinline__ void pull_rows(const Geo& G, int y, int& ym, int& yp) {
    ym = y - 1;
    yp = y + 1;
    if (G.flags & FLAG_PY) {
        if (ym < 0) ym = G.ny - 1;
        if (yp >= G.ny) yp = 0;
    }
}

// V per-node flag words of one chunk (V*2 bytes, aligned).
template <int V>
__device__ __forceinline__ void load_flags(const uint16_t* p, uint16_t (&fl)[V]) {
    if constexpr (V == 1) {
        fl[0] = __ldg(p);
    } else if constexpr (V == 2) {
        const uint32_t w = __ldg(reinterpret_cast<const uint32_t*>(p));
        fl[0] = (uint16_t)w; fl[1] = (uint16_t)(w >> 16);
    } else if constexpr (V == 4) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(p));
        fl[0] = (uint16_t)w.x; fl[1] = (uint16_t)(w.x >> 16); fl[2] = (uint16_t)w.y; fl[3] = (uint16_t)(w.y >> 16);
    } else {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(p));
        const uint32_t a[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int k = 0; k < 4; ++k) { fl[2 * k] = (uint16_t)a[k]; fl[2 * k + 1] = (uint16_t)(a[k] >> 16); }
    }
}

// The nine pulled populations of a chunk from its row vectors v and the edge
// elements e (x - 1 of the first node for the directions with e_x = 1, x + 1 of
// the last one for those with e_x = -1).  last: the index of the row's last
// node in the chunk; in a ragged last chunk (last < V - 1) that node takes the
// edge element, and the nodes beyond it are padding, whose values reach nobody.
template <class S>
__device__ __forceinline__ void form_chunk(const Chunk<S> (&v)[9], const typename S::T (&e)[9],
                                           typename ChunkOf<S>::W (&f)[9][ChunkOf<S>::N], int last) {
    typedef typename S::A A;
    typedef Vec<typename ChunkOf<S>::W> K;
    constexpr int V = S::V, N = K::N, NP = ChunkOf<S>::N;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        typename ChunkOf<S>::W u[NP];
        v[i].get(u);
        if (cx(i) == 0) {
#pragma unroll
            for (int q = 0; q < NP; ++q) f[i][q] = u[q];
        } else if (cx(i) == 1) {  // source x-1
            K::set(f[i][0], 0, to_a(e[i], (A)1));
#pragma unroll
            for (int k = 1; k < V; ++k) K::set(f[i][k / N], k % N, K::get(u[(k - 1) / N], (k - 1) % N));
        } else {  // source x+1
#pragma unroll
            for (int k = 0; k < V - 1; ++k) K::set(f[i][k / N], k % N, K::get(u[(k + 1) / N], (k + 1) % N));
            K::set(f[i][NP - 1], N - 1, to_a(e[i], (A)1));
        }
    }
    if (last < V - 1) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
            if (cx(i) == -1) {
#pragma unroll
                for (int k = 0; k < V - 1; ++k)
                    if (k == last) K::set(f[i][k / N], k % N, to_a(e[i], (A)1));
            }
    }
}
// Bits of a chunk's solid nodes and, in a ragged last chunk (left nodes of the
// row from its first one on), of the padding beyond the row.
template <int V>
__device__ __forceinline__ uint32_t solid_nodes(const uint16_t (&fl)[V], int left) {
    uint32_t m = left < V ? (((1u << V) - 1u) << left) & ((1u << V) - 1u) : 0u;
#pragma unroll
    for (int k = 0; k < V; ++k) m |= (uint32_t)(fl[k] & NF_SOLID) << k;
    return m;
}

// Moments of a node that changes side this step (tag stamped step + 1): rho
// and sum f* e of the populations just stored, read back in the storage
// format so they equal what a later read of the arena would give.
template <class S>
__device__ __noinline__ void flip_moments(const StreamArgs& a, const DomDev& D, int y, int x,
                                          const typename S::T* obase, int32_t stamp) {
    const int64_t ni = (int64_t)y * D.pitch + x;
    const int64_t tag = a.fliptag[(int64_t)(stamp & 1) * a.fliptag_stride + D.node_off + ni];
    if ((int32_t)(tag >> 32) != stamp) return;
    double r = 0.0, jx = 0.0, jy = 0.0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        double v = (double)to_a(obase[(int64_t)i * D.plane + ni], (typename S::A)D.inv_scale);
        if (S::SHIFT) v += wgt(i) * D.rho0;
        r += v;
        jx += v * cx(i);
        jy += v * cy(i);
    }
#pragma unroll 1
    for (uint32_t slot = (uint32_t)tag; slot != NO_SLOT; slot = a.fliplink[slot]) {
        a.flipmom[3 * (int64_t)slot + 0] = r;
        a.flipmom[3 * (int64_t)slot + 1] = jx;
        a.flipmom[3 * (int64_t)slot + 2] = jy;
    }
}

// Boundary nodes of a special chunk (fl: its flag words), before the collision:
// halfway bounce-back (flag bit j: the neighbour x + e_j is solid or beyond a y
// wall, so the population coming from there, opp(j), is the node's own f*_j),
// then the wall-corner and Zou-He patches of the open columns.  Straight-line
// selects: a row of disks puts flagged chunks into most warps, and branches per
// node and direction cost more than the selects they would skip.
template <class S>
__device__ __forceinline__ void patch_chunk(const DomDev& D, const Geo& G, typename S::A scale,
                                            typename ChunkOf<S>::W (&f)[9][ChunkOf<S>::N], const uint16_t (&fl)[S::V],
                                            int y, int x0, const typename S::T* base) {
    typedef typename S::A A;
    typedef Vec<typename ChunkOf<S>::W> K;
    constexpr int V = S::V, N = K::N;
    constexpr bool SC = S::SCALED;
    const int64_t pitch = G.pitch, plane = G.plane;
    const typename S::T* own = base + y * pitch + x0;
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < V; ++k) any |= (fl[k] & NF_SOLID) ? 0u : fl[k];
    if (any & 0x1FEu) {
#pragma unroll
        for (int j = 1; j < 9; ++j) {
            if (!(any & (1u << j))) continue;
            Chunk<S> o;
            typename ChunkOf<S>::W u[ChunkOf<S>::N];
            o.load(own + j * plane);
            o.get(u);
#pragma unroll
            for (int k = 0; k < V; ++k)
                if (fl[k] & (1u << j)) K::set(f[opp(j)][k / N], k % N, K::get(u[k / N], k % N));
        }
    }
    if (any & (NF_ZH_IN | NF_ZH_OUT | NF_CORNER)) {
#pragma unroll
        for (int k = 0; k < V; ++k) {
            if (fl[k] & NF_CORNER) {  // sources beyond the x range: the node's own opposite slot
                const int x = x0 + k;
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    if ((x == 0 && cx(i) == 1) || (x == G.nx - 1 && cx(i) == -1))
                        K::set(f[i][k / N], k % N, load_one<S>(own + (int64_t)opp(i) * plane + k, (A)1));
            }
            if (fl[k] & (NF_ZH_IN | NF_ZH_OUT)) {
                A n9[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) n9[i] = K::get(f[i][k / N], k % N);
                const int side = (fl[k] & NF_ZH_IN) ? 0 : 1;
                zou_he<A>(n9, side, SC ? zou_he_excess<A>(D, side) * scale : zou_he_excess<A>(D, side));
#pragma unroll
                for (int i = 0; i < 9; ++i) K::set(f[i][k / N], k % N, n9[i]);
            }
        }
    }
}

// Normals of a chunk's nodes.  They need no population, so the kernels draw them
// while the loads are in flight.
template <class S, bool NOISE, bool PL>
__device__ __forceinline__ void chunk_thetas(const ExtPrm<typename S::A>& X, uint32_t node, uint32_t step,
                                             typename ChunkOf<S>::W (&th)[ChunkOf<S>::N][6]) {
    typedef Vec<typename ChunkOf<S>::W> K;
    if (NOISE) {
        if (X.kT > (typename S::A)0) {
#pragma unroll
            for (int p = 0; p < ChunkOf<S>::N; ++p) thetas(node + p * K::N, step, X.dom_id, X.seed, th[p]);
            return;
        }
    }
#pragma unroll
    for (int p = 0; p < ChunkOf<S>::N; ++p)
#pragma unroll
        for (int m = 0; m < 6; ++m) th[p][m] = K::all(0);
}

// Collision and stores of one chunk, f[i] its pulled populations i as vectors
// W of the collision (scaled half-precision kinds in their scaled units), th
// the normals of its nodes, solid
// the bits of its solid and padding nodes: they compute on values that mean
// nothing, their slots are stored with the vectors and read by nobody, and a
// chunk of them alone stores nothing.  orow: the store row's start, xo: the
// chunk's byte offset in it.  Then the moments of nodes that change side (near
// items only).  False when a density is not a positive finite number.
template <class S, bool NOISE, bool PL, bool FLIPS>
__device__ __forceinline__ bool finish_chunk(const StreamArgs& a, const DomDev& D, const Geo& G,
                                             const HotPrm<typename S::A>& H, const ExtPrm<typename S::A>& X,
                                             typename ChunkOf<S>::W (&f)[9][ChunkOf<S>::N],
                                             const typename ChunkOf<S>::W (&th)[ChunkOf<S>::N][6], uint32_t solid, int y,
                                             int x0, typename S::T* obase, char* orow, uint32_t xo, bool near_item,
                                             int32_t next_stamp) {
    typedef typename ChunkOf<S>::W W;
    typedef Vec<W> K;
    constexpr int V = S::V, N = K::N;
    uint32_t good = solid;
    bool fix = false;
    if constexpr (S::KIND == 0 && !NOISE && !PL) {
        const FixPrm F = a.ndom == 1 ? a.dom0.fix : load_fix(D);
        fix = F.on != 0;
        if (fix) {
#pragma unroll
            for (int p = 0; p < V; ++p) {
                double n9[9], out[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) n9[i] = f[i][p];
                bool ok = collide_fix(n9, out, F);
                if (!ok && !((solid >> p) & 1u)) {
                    ok = collide_f64(D, n9);
#pragma unroll
                    for (int i = 0; i < 9; ++i) out[i] = n9[i];
                }
                if (ok) good |= 1u << p;
#pragma unroll
                for (int i = 0; i < 9; ++i) f[i][p] = out[i];
            }
        }
    }
    W tau[ChunkOf<S>::N];
    if constexpr (PL) {
        typename S::A as[V], ts[V];
#pragma unroll
        for (int p = 0; p < ChunkOf<S>::N; ++p) {
            W n9[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) n9[i] = f[i][p];
            const W r = strain<W, S::SHIFT, S::SCALED>(n9, H);
#pragma unroll
            for (int k = 0; k < N; ++k) as[p * N + k] = K::get(r, k);
        }
        solve_taus(as, X, ts);
#pragma unroll
        for (int k = 0; k < V; ++k) K::set(tau[k / N], k % N, ts[k]);
    } else {
#pragma unroll
        for (int p = 0; p < ChunkOf<S>::N; ++p) tau[p] = K::all(0);
    }
    if (!fix)
#pragma unroll
    for (int p = 0; p < ChunkOf<S>::N; ++p) {
        W n9[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) n9[i] = f[i][p];
        const W rho = collide_nodes<W, S::SHIFT, NOISE, PL, S::SCALED>(n9, H, X, th[p], tau[p]);
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (rho_ok(K::get(rho, k))) good |= 1u << (p * N + k);
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i][p] = n9[i];
    }
    if (solid != (1u << V) - 1u) {
#pragma unroll
        for (int i = 0; i < 9; ++i)
            store_chunk<S>(orow + (int64_t)i * G.plane * (int64_t)sizeof(typename S::T) + xo, f[i]);
    }
    if (FLIPS && near_item) {
#pragma unroll 1
        for (int k = 0; k < V && x0 + k < G.nx; ++k) flip_moments<S>(a, D, y, x0 + k, obase, next_stamp);
    }
    return good == (1u << V) - 1u;
}

}  // namespace lbmk
