// k_stream.cu -- fused pull-stream + collide kernel of the D2Q9 hot path
// (arXiv:2006.12910 Sec. 2 Eq. e.LB1 with the collision of Eq. e.LB2, the
// noise of Sec. 4 and the local tau* of Sec. 5; halfway bounce-back of Sec. 3).
//
// Layout: structure of arrays, plane i of domain d at arena[off + i*plane],
// rows of `pitch` elements, x fastest.  The stored values are the
// post-collision populations f*(t).  Each lane owns V consecutive nodes of
// one row (V*sizeof(T) = 8 or 16 bytes), a warp owns 32 such chunks; a work
// item is one (domain, row, warp segment).  For every direction the lane loads
// the vector of the source row and, for the two x-shifted families, one
// extra element at the chunk edge (served by L1 from the neighbour lane's
// sector), then collides in registers -- FP32 kinds two nodes at a time in the
// packed instructions -- and writes vectors.
//
// The per-node flag words are loaded for every chunk together with the
// populations, and a chunk with any flag replaces the populations that no
// fluid node sent (patch_chunk): halfway bounce-back takes the node's own
// opposite population, so every chunk stores whole vectors and nothing is
// written outside it.  (Bounced populations written into the solid
// neighbours' slots instead needed conditional stores per node and plane and a
// flag look-up before the loads: 765 instructions an item against 596.)  A
// ragged last chunk treats the padding beyond the row as solid nodes.
//
// Bounds: FP32 stores by HBM and L2 (2048x1024 porous geometry, one graph:
// 27.5 -> 26.4 us a step; 4096x2048 103.6 -> 101.9, 5.9 TB/s); half-precision
// stores by latency and issue (18.7 -> 14.7 us); noise and tau* by arithmetic.
#include "stream_node.cuh"

namespace lbmk {

// At most 128 threads per CTA, and the storage kind's resident CTAs per SM
// (MINB / MINB_EXT): the register cap they imply keeps the common variants
// from spilling while leaving room for as many warps as possible (plain FP32
// and half-precision kinds: 96 registers, 20 warps per SM).
template <class S, bool NOISE, bool PL>
constexpr int k1_min_blocks() { return (!NOISE && !PL) ? S::MINB : S::MINB_EXT; }

template <class S, bool NOISE, bool PL, bool FLIPS>
__global__ void __launch_bounds__(REG_K1_MAX_BLOCK, (k1_min_blocks<S, NOISE, PL>()))
    k_stream_collide(const __grid_constant__ StreamArgs a) {
    // A programmatic dependent launch waits here for the kernels before it
    // (completion and memory flush); otherwise this returns at once.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    typedef typename S::T T;
    typedef typename S::A A;
    typedef typename ChunkOf<S>::W W;
    constexpr int V = S::V, NP = ChunkOf<S>::N, EB = sizeof(T);
    const int lane = threadIdx.x & 31;
    // the same for all lanes (a broadcast, so that the compiler knows it)
    const uint32_t warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
    const uint32_t wpb = blockDim.x >> 5;
    const uint32_t nwarps = gridDim.x * wpb;
    const int64_t step64 = *a.ctr_in;
    // every pass writes the (same) counter of the next state, so whichever
    // pass a later kernel waits for has published it
    if (blockIdx.x == 0 && threadIdx.x == 0) *a.ctr_out = step64 + 1;
    const uint32_t step = (uint32_t)step64;
    const int par = (int)(step64 % 3);
    const T* src = static_cast<const T*>(a.src);
    T* dst = static_cast<T*>(a.dst);
    bool ok = true;
    const uint32_t count = a.mode == STREAM_NEAR ? (uint32_t)__ldg(a.near_cnt + par) : (uint32_t)a.total_items;
    const int32_t next_stamp = (int32_t)(step64 + 1);
    const int32_t* mark = a.mark + (int64_t)par * a.total_items;
    const bool one = a.ndom == 1, far = a.mode == STREAM_FAR;

    uint32_t w = blockIdx.x * wpb + warp;
    int32_t mk_next = far && w < count ? __ldg(mark + w) : 0;
    for (; w < count; w += nwarps) {
        uint32_t g = w;
        int32_t mk = (int32_t)step64;
        if (a.mode == STREAM_NEAR) {
            g = __shfl_sync(0xffffffffu, (uint32_t)__ldg(a.near_list + (int64_t)par * a.total_items + w), 0);
        } else if (far) {
            // The force launch beside a FAR pass rewrites slots of near items
            // (the link exchange), so nothing of a near item may be read here.
            // Its mark is taken an item ahead, which keeps that load's latency
            // off all items but a warp's first.
            mk = mk_next;
            if (w + nwarps < count) mk_next = __ldg(mark + w + nwarps);
            if (__shfl_sync(0xffffffffu, mk, 0) == (int32_t)step64) continue;
        } else if (FLIPS) {
            mk = __ldg(mark + w);
        }
        const int d = one ? 0 : (int)__ldg(a.item_dom + g);
        const DomDev& D = a.doms[d];
        const Geo G = one ? param_geo(a.dom0) : load_geo(D);
        const int nx = G.nx;
        const int64_t pitch = G.pitch, plane = G.plane;
        const int local = (int)(g - (uint32_t)G.item_off);
        const int y = item_row(G, local);
        const int seg = local - y * G.spr;
        const T* base = src + G.off;
        T* obase = dst + G.off;
        int ym, yp;
        pull_rows(G, y, ym, yp);
        const char* rows[3] = {reinterpret_cast<const char*>(base + y * pitch), reinterpret_cast<const char*>(base + ym * pitch),
                               reinterpret_cast<const char*>(base + yp * pitch)};
        // x-1 / x+V across a seam: wrapped when periodic; at open ends any
        // in-range element stands in until the Zou-He or corner patch.  Lanes
        // beyond the row read the segment's first chunk and store nothing.
        const int x0 = (seg * 32 + lane) * V, xs = seg * 32 * V;
        const bool in_row = x0 < nx;
        int xl = x0 - 1, xr = x0 + V;
        if (xl < 0) xl = (G.flags & FLAG_PX) ? nx - 1 : 0;
        if (xr >= nx) xr = (G.flags & FLAG_PX) ? 0 : nx - 1;
        const uint32_t xo = (uint32_t)(in_row ? x0 : xs) * EB, xlo = (uint32_t)(in_row ? xl : xs) * EB,
                       xro = (uint32_t)(in_row ? xr : xs) * EB;
        // The flag words are loaded for every chunk, with the populations: a load
        // that waits for a bit of the row's mask first costs more than the 2 bytes
        // a node.
        uint16_t fl[V];
        load_flags<V>(a.nflags + G.node_off + y * pitch + (in_row ? x0 : xs), fl);
        // The parameters before the loads, but after them in the plain power-law
        // variant (FP64 89.5 -> 84 us a step at 2048x1024 by the former, 4096x256 at
        // n = 0.75 15.79 -> 15.67 by the latter).
        HotPrm<A> H;
        ExtPrm<A> X;
        if (!PL || NOISE) {
            H = one ? param_hot<A>(a.dom0) : load_hot<A>(D);
            X = load_ext<A, NOISE, PL>(one ? a.dom0 : D);
        }
        // The normals are drawn while the loads are in flight; with the power law
        // before them, for want of registers (ensemble 169 us a step, 191 before
        // the loads; noise and tau* 56.6, 57.9 behind them).
        W th[NP][6];
        if (PL && NOISE) chunk_thetas<S, NOISE, PL>(X, (uint32_t)(y * nx + x0), step, th);
        Chunk<S> v[9];
        T e[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const char* p = rows[cy(i) == 0 ? 0 : (cy(i) == 1 ? 1 : 2)] + (int64_t)i * plane * EB;
            v[i].load(p + xo);
            if (cx(i)) {
                // with noise alone a plain dereference (3000x41 channel 5.41 -> 5.32 us a
                // step of three contexts, 512x512 alone 14.7 -> 14.1)
                const char* q = p + (cx(i) == 1 ? xlo : xro);
                if (NOISE && !PL) e[i] = *reinterpret_cast<const T*>(q);
                else load_pop(e[i], q);
            }
        }
        if (PL && !NOISE) {
            H = one ? param_hot<A>(a.dom0) : load_hot<A>(D);
            X = load_ext<A, NOISE, PL>(one ? a.dom0 : D);
        }
        if (!(PL && NOISE)) chunk_thetas<S, NOISE, PL>(X, (uint32_t)(y * nx + x0), step, th);
        const bool near_item = FLIPS && __shfl_sync(0xffffffffu, mk, 0) == (int32_t)step64;
        if (in_row) {
            W f[9][NP];
            form_chunk<S>(v, e, f, nx - 1 - x0);
            uint32_t any = 0;
#pragma unroll
            for (int k = 0; k < V; ++k) any |= fl[k];
            if (any) patch_chunk<S>(D, G, H.scale, f, fl, y, x0, base);
            ok &= finish_chunk<S, NOISE, PL, FLIPS>(a, D, G, H, X, f, th, solid_nodes<V>(fl, nx - x0), y, x0, obase,
                                                    reinterpret_cast<char*>(obase + y * pitch), xo, near_item,
                                                    next_stamp);
        }
        __syncwarp();
    }
    // The next pass may be placed on the SMs while the last CTAs finish (it
    // waits for their completion).
    asm volatile("griddepcontrol.launch_dependents;");
    if (!ok) atomicOr(a.err, ERR_UNSTABLE);
}

template <class S, bool NOISE, bool PL, bool FLIPS>
static cudaError_t launch_one(const StreamArgs& a, int block, int64_t grid, cudaStream_t s, bool pdl) {
    if (!pdl) {
        k_stream_collide<S, NOISE, PL, FLIPS><<<(unsigned)grid, block, 0, s>>>(a);
        return cudaGetLastError();
    }
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_stream_collide<S, NOISE, PL, FLIPS>, a);
}

template <class S, bool FLIPS>
static cudaError_t launch_kind_f(bool noise, bool pl, const StreamArgs& a, int block, int64_t grid, cudaStream_t s,
                                 bool pdl) {
    if (noise && pl) return launch_one<S, true, true, FLIPS>(a, block, grid, s, pdl);
    if (noise) return launch_one<S, true, false, FLIPS>(a, block, grid, s, pdl);
    if (pl) return launch_one<S, false, true, FLIPS>(a, block, grid, s, pdl);
    return launch_one<S, false, false, FLIPS>(a, block, grid, s, pdl);
}

// The variant that writes the moments of nodes changing side runs the items
// near particles (mode STREAM_NEAR, or STREAM_ALL when particles exist).
template <class S>
static cudaError_t launch_kind(bool noise, bool pl, const StreamArgs& a, int block, int64_t grid, cudaStream_t s,
                               bool pdl) {
    if (a.flips) return launch_kind_f<S, true>(noise, pl, a, block, grid, s, pdl);
    return launch_kind_f<S, false>(noise, pl, a, block, grid, s, pdl);
}

cudaError_t launch_stream_staged(int kind, bool noise, bool pl, const StreamArgs& a, int block, int64_t grid,
                                 int stages, cudaStream_t s);

cudaError_t launch_stream_collide(int kind, bool noise, bool pl, const StreamArgs& a, int block, int64_t grid,
                                  int stages, cudaStream_t s, bool pdl) {
    if (stages > 0 && a.mode != STREAM_NEAR) return launch_stream_staged(kind, noise, pl, a, block, grid, stages, s);
    switch (kind) {
        case 0: return launch_kind<StF64>(noise, pl, a, block, grid, s, pdl);
        case 1: return launch_kind<StF32>(noise, pl, a, block, grid, s, pdl);
        case 2: return launch_kind<StF32S>(noise, pl, a, block, grid, s, pdl);
        case 3: return launch_kind<StF16S>(noise, pl, a, block, grid, s, pdl);
        case 4: return launch_kind<StBF16S>(noise, pl, a, block, grid, s, pdl);
        default: return cudaErrorInvalidValue;
    }
}

template <class S>
static int reg_bps(bool noise, bool pl, int block) {
    int n = 0;
    cudaError_t e;
    if (noise && pl) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_stream_collide<S, true, true, false>, block, 0);
    else if (noise) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_stream_collide<S, true, false, false>, block, 0);
    else if (pl) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_stream_collide<S, false, true, false>, block, 0);
    else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_stream_collide<S, false, false, false>, block, 0);
    return e == cudaSuccess ? n : 0;
}

int reg_blocks_per_sm(int kind, bool noise, bool pl, int block) {
    if (block < 32 || block > REG_K1_MAX_BLOCK) return 0;
    switch (kind) {
        case 0: return reg_bps<StF64>(noise, pl, block);
        case 1: return reg_bps<StF32>(noise, pl, block);
        case 2: return reg_bps<StF32S>(noise, pl, block);
        case 3: return reg_bps<StF16S>(noise, pl, block);
        case 4: return reg_bps<StBF16S>(noise, pl, block);
        default: return 0;
    }
}

int store_vector_width(int kind) {
    switch (kind) {
        case 0: return StF64::V;
        case 1: return StF32::V;
        case 2: return StF32S::V;
        case 3: return StF16S::V;
        case 4: return StBF16S::V;
        default: return 0;
    }
}

}  // namespace lbmk
