// Modified Hauser-Verhey (HV) model kernels, arXiv 2309.08068 Section III.
//
// One thread updates one cell: 6 directions, each an electric vector e_i and a magnetic vector h_i
// (36 scalars), pulled as a 4-vector (e_x, e_y, e_z, h_x) and a 2-vector (h_y, h_z) from cell
// x - v_i (float4 + float2, or 8 + 4 bytes with 16-bit storage); arithmetic is FP32.
// Velocities in the Section III order: v1 = +x, v2 = +y, v3 = -x, v4 = -y, v5 = -z, v6 = +z.
//
// With tau = 1/2 the collision (eqs. equilibriumHV, CollisionHV, CollisionmodifiedHV) is
//   e_i' = 2 e_i^eq - e_i + T_i = D/3 - v_i x H - e_i - (J . v_i) v_i / 2
//   h_i' = 2 h_i^eq - h_i       = B/3 + v_i x E - h_i
// with D = sum e_i, B = sum h_i (eq. MacroscopicFieldsHV), E = D / eps, H = B / mu, eps = eps0 eps_r,
// mu = mu0 mu_r, and J = sigma E + J_ext. For v_i = s a (a a unit axis, s = +-1) the source term is
// -(J_a / 2) a whatever the sign s.
#include "hv_core.cuh"

namespace lbm {
namespace {

// Two steps per pass (see FusedArgs): phase A streams the A/B buffers in once and writes the
// intermediate plane, phase B pulls from the intermediate planes (L2 loads) and streams the other
// A/B buffers out. The arithmetic is hv_update's, so the results equal two single steps bit for bit.
template <int S>
struct HVToRing : FusedStash {
    using T4 = typename Pack4<S>::T;
    using T2 = typename Pack2<S>::T;
    T4* plane;
    T2* plane2;
    int base, nxy;
    template <int S2>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&e)[6], float2 (&hy)[6]) const {
        const T4* ein = static_cast<const T4*>(a.fin);
        const T2* hin = static_cast<const T2*>(a.fin2);
        static_for<0, 6>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            const int src = pull_index<k>(h);
            e[k] = Pack4<S>::unpack(__ldcs(ein + (size_t)k * a.g.n + src), a.inv_scale);
            hy[k] = Pack2<S>::unpack(__ldcs(hin + (size_t)k * a.g.n + src), a.inv_scale);
        });
    }
    template <int S2>
    __device__ void put(const StepArgs& a, int k, int i, float4 e, float2 hy) const {
        __stcg(plane + (size_t)k * nxy + (i - base), Pack4<S>::pack(e, a.scale));
        __stcg(plane2 + (size_t)k * nxy + (i - base), Pack2<S>::pack(hy, a.scale));
    }
};

template <int S>
struct HVFromRing : FusedStash {
    using T4 = typename Pack4<S>::T;
    using T2 = typename Pack2<S>::T;
    const T4* plane[3];  // slots of planes z - 1, z, z + 1
    const T2* plane2[3];
    int nxy;
    template <int S2>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&e)[6], float2 (&hy)[6]) const {
        static_for<0, 6>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            constexpr int ax = kHVAxis[k], sg = kHVSign[k];
            constexpr int sx = ax == 0 ? -sg : 0, sy = ax == 1 ? -sg : 0, sz = ax == 2 ? -sg : 0;
            const int off = (int)((size_t)k * nxy) + h.xo[sx + 1] + h.yo[sy + 1];
            e[k] = Pack4<S>::unpack(__ldcg(plane[sz + 1] + off), a.inv_scale);
            hy[k] = Pack2<S>::unpack(__ldcg(plane2[sz + 1] + off), a.inv_scale);
        });
    }
    template <int S2>
    __device__ void put(const StepArgs& a, int k, int i, float4 e, float2 hy) const {
        T4* __restrict__ eout = static_cast<T4*>(a.fout);
        T2* __restrict__ hout = static_cast<T2*>(a.fout2);
        __stcs(eout + (size_t)k * a.g.n + i, Pack4<S>::pack(e, a.scale));
        __stcs(hout + (size_t)k * a.g.n + i, Pack2<S>::pack(hy, a.scale));
    }
};

template <int S, int M>
__global__ void __launch_bounds__(kFusedThreads, 3) hv_fused2_kernel(StepArgs aA, StepArgs aB, FusedArgs F) {
    using T4 = typename Pack4<S>::T;
    using T2 = typename Pack2<S>::T;
    __shared__ float2 s_stash[12 * kBlock];  // the h components, [slot][compute thread]
    const unsigned stash = fused_stash_slot(s_stash);
    const int nz = aA.g.nz, nxy = aA.g.nx * aA.g.ny;
    auto slot = [&](int p) -> T4* {
        if (p == 0) return static_cast<T4*>(F.lo);
        if (p == nz - 1) return static_cast<T4*>(F.hi);
        return static_cast<T4*>(F.ring) + (size_t)(p % F.R) * 6 * nxy;
    };
    auto slot2 = [&](int p) -> T2* {
        if (p == 0) return static_cast<T2*>(F.lo2);
        if (p == nz - 1) return static_cast<T2*>(F.hi2);
        return static_cast<T2*>(F.ring2) + (size_t)(p % F.R) * 6 * nxy;
    };
    auto describe = [&](const FusedItem& it, FusedDesc& d) {
        if (it.type == kPhaseA) {
            d.ptr[0] = slot(it.plane);
            d.ptr[1] = slot2(it.plane);
        } else {
            const int pm = (it.plane + nz - 1) % nz, pp = (it.plane + 1) % nz;
            d.ptr[0] = slot(pm);
            d.ptr[1] = slot(it.plane);
            d.ptr[2] = slot(pp);
            d.ptr[3] = slot2(pm);
            d.ptr[4] = slot2(it.plane);
            d.ptr[5] = slot2(pp);
        }
    };
    fused_loop(F, aA.g.nx, nxy, nz, describe, [&](const FusedDesc& d) {
        const int j = d.j, base = d.plane * nxy;
        if (d.type == kPhaseA) {
            const HVToRing<S> io{{stash}, static_cast<T4*>(d.ptr[0]), static_cast<T2*>(d.ptr[1]), base, nxy};
            const int end = min(base + (j + 1) * F.tile_cells, base + nxy);
            for (int i = base + j * F.tile_cells + threadIdx.x; i < end; i += kBlock)
                hv_update<S, M, false, false>(aA, i, 0, io);
            if (d.s_hi > d.s_lo) {  // the tile's source cells replace their ordinary update
                named_sync(kComputeBarrier, kBlock);
                for (int m = d.s_lo + threadIdx.x; m < d.s_hi; m += kBlock)
                    hv_update<S, M, true, false>(aA, aA.sv.cell[m], m, io);
            }
        } else {
            const HVFromRing<S> io{{stash},
                                   {static_cast<const T4*>(d.ptr[0]), static_cast<const T4*>(d.ptr[1]),
                                    static_cast<const T4*>(d.ptr[2])},
                                   {static_cast<const T2*>(d.ptr[3]), static_cast<const T2*>(d.ptr[4]),
                                    static_cast<const T2*>(d.ptr[5])},
                                   nxy};
            const int end = min(base + (j + 1) * F.tile_cells, base + nxy);
            for (int i = base + j * F.tile_cells + threadIdx.x; i < end; i += kBlock)
                hv_update<S, M, false, false>(aB, i, 0, io);
            if (d.s_hi > d.s_lo) {  // the tile's source cells replace their ordinary update
                named_sync(kComputeBarrier, kBlock);
                for (int m = d.s_lo + threadIdx.x; m < d.s_hi; m += kBlock)
                    hv_update<S, M, true, false>(aB, aB.sv.cell[m], m, io);
            }
        }
    });
}

// Two steps per pass over shared-memory tiles (see TileArgs). HV's two z directions lead to the cell's
// own column, so phase B of a thread's cell takes them from the thread itself: -z of plane q + 1 from
// registers, +z of plane q - 1 from a ring of three slots that only this thread uses. The four in-plane
// directions pass between threads through two planes of shared memory: while phase A writes plane p,
// phase B reads plane p - 1, which the barrier at the end of the previous plane has completed, so a
// plane takes one barrier.
//
// Two steps cannot move less than 288 B per cell: 0.711 ms on 256^3 at the copy rate. This kernel takes
// 0.806 ms (0.403 ms per step; 300 B of DRAM traffic per cell, at chunks of 19 planes). With 16 x 16
// cells and an L2 prefetch of the next plane instead of its loads, three blocks per SM and everything in
// shared memory it was 1.08 ms: the prefetches doubled the load instructions, whose queue was what the
// warps waited for. 128^3 with a medium per cell: 58 us per step, was 94.
template <int S>
struct HVTile {
    using T4 = typename Pack4<S>::T;
    using T2 = typename Pack2<S>::T;
    // direction planes of Tile::kCells cells: 0-3 and 4-7 in-plane directions of even and odd planes,
    // 8-10 +z of the last three planes; the 4-vectors, then the 2-vectors
    static constexpr int kPlanes = 11;
    static constexpr size_t kBytes = kPlanes * Tile::kCells * (sizeof(T4) + sizeof(T2));
};

template <int S, int M>
__global__ void __launch_bounds__(Tile::kCells, 2) hv_tile2_kernel(StepArgs aA,
                                                                     StepArgs aB, TileArgs T) {
    using T4 = typename Pack4<S>::T;
    using T2 = typename Pack2<S>::T;
    extern __shared__ __align__(16) unsigned char hv_tile_smem[];
    __shared__ TileSources<Tile>::Shared s_sources;
    after_predecessor();
    T4* const base4 = reinterpret_cast<T4*>(hv_tile_smem);
    T2* const base2 = reinterpret_cast<T2*>(hv_tile_smem + HVTile<S>::kPlanes * Tile::kCells * sizeof(T4));
    const int tid = threadIdx.x, nz = aA.g.nz, nxy = aA.g.nx * aA.g.ny;
    const size_t n = (size_t)aA.g.n;
    const TileCell c = tile_cell<Tile>(aA.g, T, tid);
    const int cxy = c.row + c.x;
    TileSources<Tile> src{&s_sources, T.entries, aA.sv.first, c.z0 - 1};
    const TilePull t = tile_pull(aA.g, c, 0);
    const int from[4] = {t.x[0] + c.row, c.x + t.row[0], t.x[2] + c.row, c.x + t.row[2]};  // x - v of +x, +y, -x, -y
    // Phase A's inputs of the next plane, loaded while phase B of the plane before runs: they are
    // the block's only loads from memory, and two blocks per SM hide no round trip on their own.
    T4 pe[6];
    T2 ph[6];
    RawMedium<M> raw;
    auto fetch = [&](int p) {
        const T4* ein = static_cast<const T4*>(aA.fin);
        const T2* hin = static_cast<const T2*>(aA.fin2);
        static_for<0, 6>([&](auto kc) {
            constexpr int k = decltype(kc)::value;
            constexpr int vz = kHVAxis[k] == 2 ? kHVSign[k] : 0;
            const int at = tile_wrap(p - vz, nz) * nxy + (vz != 0 ? cxy : from[k & 3]);
            pe[k] = ein[k * n + at];
            ph[k] = hin[k * n + at];
        });
        raw.load(aA.media, tile_wrap(p, nz) * nxy + cxy);
    };
    fetch(c.z0 - 1);
    src.start(T, c, nz);
    MatCoef mat_b;           // medium and source cell of phase B's plane: phase A's one plane before
    int m_b = -1, ring = 0;  // ring slot of +z of plane p
    for (int p = c.z0 - 1; p <= c.z1; ++p) {
        const MatCoef mat = coef_of<kModelHV, M>(aA.media, raw, aA.eps0, aA.mu0);
        const int m = src.take(p);
        T4 down4;  // -z of plane p, for phase B
        T2 down2;
        auto half = [](auto, float&, float&, float&) {};
        {  // phase A: step t of the extended tile's cells of plane p
            float4 e[6];
            float2 hy[6];
            static_for<0, 6>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                e[k] = Pack4<S>::unpack(pe[k], aA.inv_scale);
                hy[k] = Pack2<S>::unpack(ph[k], aA.inv_scale);
            });
            const int plane = 4 * (p & 1);
            auto put = [&](auto kc, float4 ev, float2 hv) {
                constexpr int k = decltype(kc)::value;
                const T4 v4 = Pack4<S>::pack(ev, aA.scale);
                const T2 v2 = Pack2<S>::pack(hv, aA.scale);
                if constexpr (k == 4) {
                    down4 = v4;
                    down2 = v2;
                } else {
                    const int at = (k < 4 ? plane + k : 8 + ring) * Tile::kCells + tid;
                    base4[at] = v4;
                    base2[at] = v2;
                }
            };
            const CellSource cs = tile_source(aA, m);
            hv_collide(hv_fields<true>(e, hy, mat, cs.J), e, hy, half, put);
            if (cs.imposed) hv_impose(mat, cs, put);
        }
        if (p < c.z1) {
            fetch(p + 1);
            src.prepare(p + 1);
        }
        if (p > c.z0 && c.core) {  // phase B: step t + 1 of the tile's own cells of plane q = p - 1
            const int plane = 4 * ((p - 1) & 1), below = ring == 2 ? 0 : ring + 1;  // +z of plane q - 1
            float4 e[6];
            float2 hy[6];
            static_for<0, 6>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                constexpr int vx = kHVAxis[k] == 0 ? kHVSign[k] : 0, vy = kHVAxis[k] == 1 ? kHVSign[k] : 0;
                if constexpr (k == 4) {
                    e[k] = Pack4<S>::unpack(down4, aB.inv_scale);
                    hy[k] = Pack2<S>::unpack(down2, aB.inv_scale);
                } else {
                    const int at = (k < 4 ? plane + k : 8 + below) * Tile::kCells + tid - (vx + vy * Tile::EX);
                    e[k] = Pack4<S>::unpack(base4[at], aB.inv_scale);
                    hy[k] = Pack2<S>::unpack(base2[at], aB.inv_scale);
                }
            });
            const int out = (p - 1) * nxy + cxy;
            auto put = [&](auto kc, float4 ev, float2 hv) {
                constexpr int k = decltype(kc)::value;
                __stcs(static_cast<T4*>(aB.fout) + k * n + out, Pack4<S>::pack(ev, aB.scale));
                __stcs(static_cast<T2*>(aB.fout2) + k * n + out, Pack2<S>::pack(hv, aB.scale));
            };
            const CellSource cs = tile_source(aB, m_b);
            hv_collide(hv_fields<true>(e, hy, mat_b, cs.J), e, hy, half, put);
            if (cs.imposed) hv_impose(mat_b, cs, put);
        }
        mat_b = mat;
        m_b = m;
        ring = ring == 2 ? 0 : ring + 1;
        __syncthreads();
    }
}

// The block's source cells are recomputed at the end (block_source_cells). 4 resident blocks (64
// registers); 3 for 24-bit storage, whose decoding would spill at 64.
template <int S, int M>
__global__ void __launch_bounds__(kBlock, S == kF24 ? 3 : 4) hv_step_kernel(StepArgs a) {
    wait_predecessor();
    const int i = a.cell_begin + blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.cell_end) hv_update<S, M, false>(a, i, 0);
    block_source_cells(a.sv, blockIdx.x, [&](int c, int m) { hv_update<S, M, true>(a, c, m); });
}

// The same on a lattice of few waves of blocks, with its sources known early (early_source, which has the
// figures).
template <int S, int M>
__global__ void __launch_bounds__(kBlock, S == kF24 ? 3 : 4) hv_step_early_kernel(StepArgs a) {
    const int i = a.cell_begin + blockIdx.x * blockDim.x + threadIdx.x;
    CellSource cs;
    const bool sources = early_source(a, blockIdx.x, i, &cs);
    wait_predecessor();
    if (i >= a.cell_end) return;
    if (sources) hv_update_sourced<S, M>(a, i, cs);
    else hv_update<S, M, false>(a, i, 0);
}

// Equilibria for fields E, B and J = 0 (Appendix B initialisation), stored so that cell x pulls
// them at the next step: direction i at y holds the equilibrium of cell y + v_i.
template <int S, int M>
__global__ void __launch_bounds__(kBlock) hv_init_kernel(StepArgs a, const float* E, const float* B) {
    after_predecessor_by_size();
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= a.g.n) return;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, y);
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        constexpr int A = kHVAxis[k], G = kHVSign[k];
        const int x = push_index<k>(h);
        const MatCoef mat = load_coef<kModelHV, M>(a.media, x, a.eps0, a.mu0);
        const float3 Ex = make_float3(E[x], E[n + x], E[2 * n + x]);
        const float3 Bx = make_float3(B[x], B[n + x], B[2 * n + x]);
        const float3 cH = axis_cross<A, G>(hv_h(Bx, mat));
        const float3 cE = axis_cross<A, G>(Ex);
        const float3 d6 = hv_sixth_of_d(Ex, mat), b6 = sixth(Bx);
        // e^eq = (D - 3 v x B / mu) / 6 = D/6 - (v x H)/2;  h^eq = (B + 3 v x D / eps) / 6 = B/6 + (v x E)/2
        hv_put<S>(a, k, y,
                  make_float4(d6.x - 0.5f * cH.x, d6.y - 0.5f * cH.y, d6.z - 0.5f * cH.z, b6.x + 0.5f * cE.x),
                  make_float2(b6.y + 0.5f * cE.y, b6.z + 0.5f * cE.z));
    });
}

// Fields of cell i; m is its index in the special-cell list when kSpecial.
template <int S, int M, bool kSpecial>
__device__ __forceinline__ void hv_fields_cell(const StepArgs& a, const FieldsOut& out, int i, int m) {
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, i);
    float4 e[6];
    float2 hy[6];
    hv_pull<S>(a, h, e, hy);
    const MatCoef mat = load_coef<kModelHV, M>(a.media, i, a.eps0, a.mu0);
    float3 jext = make_float3(0.f, 0.f, 0.f);
    if constexpr (kSpecial) jext = cell_source(a.sv, a.sc, m).J;
    const HVFields F = hv_fields(e, hy, mat, jext);
    auto put = [&](float* p, float3 v) {
        if (p) {
            p[i] = v.x;
            p[n + i] = v.y;
            p[2 * n + i] = v.z;
        }
    };
    put(out.E, F.E);
    put(out.B, F.B);
    put(out.D, F.D);
    put(out.H, F.H);
    put(out.J, F.J);
}

// Every cell, and, where the blocks' source-cell offsets cover the whole lattice (not a z-slab, whose
// offsets cover the stepped planes), the block's source cells after them.
template <int S, int M>
__global__ void __launch_bounds__(kBlock) hv_fields_kernel(StepArgs a, FieldsOut out) {
    after_predecessor();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.g.n) hv_fields_cell<S, M, false>(a, out, i, 0);
    if (a.cell_begin == 0)
        block_source_cells(a.sv, blockIdx.x, [&](int c, int m) { hv_fields_cell<S, M, true>(a, out, c, m); });
}

template <int S, int M>
__global__ void __launch_bounds__(kBlock) hv_fields_special_kernel(StepArgs a, FieldsOut out) {
    after_predecessor();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < a.sv.n_special) hv_fields_cell<S, M, true>(a, out, a.sv.cell[m], m);
}

// Canonical layout out[k * n + x], k = r*18 + (i-1)*3 + c.
template <int S>
__global__ void __launch_bounds__(kBlock) hv_get_kernel(StepArgs a, float* __restrict__ out) {
    after_predecessor();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= a.g.n) return;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, x);
    float4 e[6];
    float2 hy[6];
    hv_pull<S>(a, h, e, hy);
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        out[(size_t)(3 * k + 0) * n + x] = e[k].x;
        out[(size_t)(3 * k + 1) * n + x] = e[k].y;
        out[(size_t)(3 * k + 2) * n + x] = e[k].z;
        out[(size_t)(18 + 3 * k + 0) * n + x] = e[k].w;
        out[(size_t)(18 + 3 * k + 1) * n + x] = hy[k].x;
        out[(size_t)(18 + 3 * k + 2) * n + x] = hy[k].y;
    });
}

template <int S>
__global__ void __launch_bounds__(kBlock) hv_set_kernel(StepArgs a, const float* in) {
    after_predecessor_by_size();
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= a.g.n) return;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, y);
    float4 e[6];  // every load before the first store, which the loads could not be moved across
    float2 hy[6];
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        const int x = push_index<k>(h);
        e[k] = make_float4(in[(size_t)(3 * k) * n + x], in[(size_t)(3 * k + 1) * n + x],
                           in[(size_t)(3 * k + 2) * n + x], in[(size_t)(18 + 3 * k) * n + x]);
        hy[k] = make_float2(in[(size_t)(19 + 3 * k) * n + x], in[(size_t)(20 + 3 * k) * n + x]);
    });
    static_for<0, 6>([&](auto ic) { hv_put<S>(a, decltype(ic)::value, y, e[decltype(ic)::value], hy[decltype(ic)::value]); });
}

// Per-block partial sums of (1/2)(E.D + B.H) and sum f^2 (E does not depend on J_ext in HV, so no
// source-cell correction is needed).
template <int S, int M>
__global__ void __launch_bounds__(kBlock) hv_reduce_kernel(StepArgs a, double* __restrict__ partials) {
    after_predecessor();
    double w = 0.0, f2 = 0.0;
    for (int i = a.cell_begin + blockIdx.x * blockDim.x + threadIdx.x; i < a.cell_end; i += gridDim.x * blockDim.x) {
        const Neighbourhood h = neighbourhood(a.g, i);
        float4 e[6];
        float2 hy[6];
        hv_pull<S>(a, h, e, hy);
        const MatCoef mat = load_coef<kModelHV, M>(a.media, i, a.eps0, a.mu0);
        const HVFields F = hv_fields(e, hy, mat, make_float3(0.f, 0.f, 0.f));
        w += 0.5 * ((double)F.E.x * F.D.x + (double)F.E.y * F.D.y + (double)F.E.z * F.D.z +
                    (double)F.B.x * F.H.x + (double)F.B.y * F.H.y + (double)F.B.z * F.H.z);
        double s = 0.0;
#pragma unroll
        for (int k = 0; k < 6; ++k)
            s += (double)e[k].x * e[k].x + (double)e[k].y * e[k].y + (double)e[k].z * e[k].z +
                 (double)e[k].w * e[k].w + (double)hy[k].x * hy[k].x + (double)hy[k].y * hy[k].y;
        f2 += s;
    }
    block_sum3_store(w, f2, 0.0, partials + 3 * blockIdx.x);
}

// Batched step j of several lattices (see mm_batch_kernel).
template <int S, int BLOCK>
__global__ void __launch_bounds__(BLOCK) hv_batch_kernel(const BatchLattice* __restrict__ lat,
                                                         const BatchTile* __restrict__ tiles, int n_tiles, int j) {
    wait_predecessor();
    for (int b = blockIdx.x; b < n_tiles; b += gridDim.x) {
        const BatchTile tile = tiles[b];
        const BatchLattice* L = &lat[tile.lattice];
        const int i = tile.begin + threadIdx.x;
        if (j >= L->steps || i >= L->base.g.n) continue;
        const StepArgs a = batch_args(L, j);
        switch (a.media_mode) {
            case kUniform: hv_update<S, kUniform, false>(a, i, 0); break;
            case kTable: hv_update<S, kTable, false>(a, i, 0); break;
            default: hv_update<S, kPerCell, false>(a, i, 0); break;
        }
    }
}

template <int S>
__global__ void __launch_bounds__(kBlock) hv_batch_special_kernel(const BatchLattice* __restrict__ lat,
                                                                  const BatchTile* __restrict__ tiles, int j) {
    wait_predecessor();
    const BatchTile tile = tiles[blockIdx.x];
    const BatchLattice* L = &lat[tile.lattice];
    const int m = tile.begin + threadIdx.x;
    if (j >= L->steps || m >= L->base.sv.n_special) return;
    StepArgs a = batch_args(L, j);
    batch_sources(L, j, a);
    const int i = a.sv.cell[m];
    switch (a.media_mode) {
        case kUniform: hv_update<S, kUniform, true>(a, i, m); break;
        case kTable: hv_update<S, kTable, true>(a, i, m); break;
        default: hv_update<S, kPerCell, true>(a, i, m); break;
    }
}

template <int M>
__global__ void __launch_bounds__(kBlock) hv_record_kernel(StepArgs a) {
    wait_predecessor();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.g.n) hv_update<kF32, M, false, true>(a, i, 0);
    block_source_cells(a.sv, blockIdx.x, [&](int c, int m) { hv_update<kF32, M, true, true>(a, c, m); });
}

// ---------------------------------------------------------------------------------------------
// Adjoint of one HV step. With adjoints e_i^, h_i^ of the post-collision vectors, the transpose of
// e_i' = D/3 - v_i x H - e_i - (J . v_i) v_i / 2 and h_i' = B/3 + v_i x E - h_i is
//   gH = sum_i v_i x e_i^,   gE = sum_i h_i^ x v_i + sigma gJ,   gJ_a = -(1/2) sum_{i on axis a} e_i^_a,
//   gD = sum_i e_i^ / 3 + gE / eps,   gB = sum_i h_i^ / 3 + gH / mu,
//   nu(e_i) = gD - e_i^,   nu(h_i) = gB - h_i^,
//   dL/d eps_r += -gE . E / eps_r   (E = D / (eps0 eps_r)),   dL/d sigma += gJ . E.
// Imposed cells output f_eq(E_imp, B_imp, 0), where D_imp = eps0 eps_r E_imp: nothing flows back
// to f, and d e_i' / d eps_r = eps0 E_imp / 6. The plane loss |E|^2 adds 2E to gE.
template <int M, bool kSpecial, bool kTerminal>
__device__ __forceinline__ void hv_adjoint_cell(const AdjointArgs& A, int i, int m) {
    const StepArgs& a = A.a;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, i);
    const MatCoef mat = load_coef<kModelHV, M>(a.media, i, a.eps0, a.mu0);
    CellSource cs;
    bool imposed = false;
    if constexpr (kSpecial) {
        cs = cell_source(a.sv, a.sc, m);
        imposed = cs.imposed;
    }
    // Every load is issued up front: the source-cell mask of the main launch only gates the stores,
    // so it adds no round trip before the others.
    const bool skip = !kSpecial && !kTerminal && A.special_mask[i] != 0;
    const float geps_old = A.grad_eps[i], gsig_old = A.grad_sigma ? A.grad_sigma[i] : 0.f;
    // E of f^n: from the forward step's record, or (terminal) from the final state
    float3 E;
    if constexpr (kTerminal) {
        float4 e[6];
        float2 hy[6];
        hv_pull<kF32>(a, h, e, hy);
        E = hv_fields(e, hy, mat, make_float3(0.f, 0.f, 0.f)).E;
    } else {
        E = make_float3(a.rec[i], a.rec[n + i], a.rec[2 * n + i]);
    }
    struct {
        float3 E;
    } F{E};
    const float inv_eps = mat.c0.y, inv_mu = mat.c0.w, sigma = mat.c1.x, er = mat.c1.y;
    float4 le[6];
    float2 lh[6];
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        if constexpr (kTerminal) {
            le[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            lh[k] = make_float2(0.f, 0.f);
        } else {
            const int dst = push_index<k>(h);
            le[k] = static_cast<const float4*>(A.nu_in)[(size_t)k * n + dst];
            lh[k] = static_cast<const float2*>(A.nu_in2)[(size_t)k * n + dst];
        }
    });
    float3 Se = make_float3(0.f, 0.f, 0.f), Sh = Se, gH = Se, gE = Se, gJ = Se;
    float geps_imposed = 0.f;
    if (!imposed) {
        static_for<0, 6>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            constexpr int AX = kHVAxis[k], G = kHVSign[k];
            const float3 ek = make_float3(le[k].x, le[k].y, le[k].z);
            const float3 hk = make_float3(le[k].w, lh[k].x, lh[k].y);
            Se = make_float3(Se.x + ek.x, Se.y + ek.y, Se.z + ek.z);
            Sh = make_float3(Sh.x + hk.x, Sh.y + hk.y, Sh.z + hk.z);
            const float3 ve = axis_cross<AX, G>(ek);  // v_k x e_k^
            const float3 vh = axis_cross<AX, G>(hk);  // v_k x h_k^ = -(h_k^ x v_k)
            gH = make_float3(gH.x + ve.x, gH.y + ve.y, gH.z + ve.z);
            gE = make_float3(gE.x - vh.x, gE.y - vh.y, gE.z - vh.z);
            if constexpr (AX == 0) gJ.x -= 0.5f * ek.x;
            else if constexpr (AX == 1) gJ.y -= 0.5f * ek.y;
            else gJ.z -= 0.5f * ek.z;
        });
        gE = make_float3(__fmaf_rn(sigma, gJ.x, gE.x), __fmaf_rn(sigma, gJ.y, gE.y), __fmaf_rn(sigma, gJ.z, gE.z));
    } else if constexpr (kSpecial) {
        const float3 dE = make_float3(div_rn(a.eps0 * cs.E.x, 6.f, kInv6), div_rn(a.eps0 * cs.E.y, 6.f, kInv6),
                                      div_rn(a.eps0 * cs.E.z, 6.f, kInv6));
        static_for<0, 6>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            geps_imposed += le[k].x * dE.x + le[k].y * dE.y + le[k].z * dE.z;
        });
    }
    if (A.loss_active && in_plane(h, a.g, A.plane_axis, A.plane_index)) {  // |E|^2 of time n
        gE = make_float3(__fmaf_rn(2.f, F.E.x, gE.x), __fmaf_rn(2.f, F.E.y, gE.y), __fmaf_rn(2.f, F.E.z, gE.z));
        add_plane_loss<kTerminal>(A, h, F.E);
    }
    const float3 gD = make_float3(__fmaf_rn(gE.x, inv_eps, div_rn(Se.x, 3.f, kInv3)),
                                  __fmaf_rn(gE.y, inv_eps, div_rn(Se.y, 3.f, kInv3)),
                                  __fmaf_rn(gE.z, inv_eps, div_rn(Se.z, 3.f, kInv3)));
    const float3 gB = make_float3(__fmaf_rn(gH.x, inv_mu, div_rn(Sh.x, 3.f, kInv3)),
                                  __fmaf_rn(gH.y, inv_mu, div_rn(Sh.y, 3.f, kInv3)),
                                  __fmaf_rn(gH.z, inv_mu, div_rn(Sh.z, 3.f, kInv3)));
    if (skip) return;  // a source cell: the second launch writes it
    float4* eout = static_cast<float4*>(A.nu_out);
    float2* hout = static_cast<float2*>(A.nu_out2);
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        float4 o;
        float2 p;
        if (imposed) {
            o = make_float4(gD.x, gD.y, gD.z, gB.x);
            p = make_float2(gB.y, gB.z);
        } else {
            o = make_float4(gD.x - le[k].x, gD.y - le[k].y, gD.z - le[k].z, gB.x - le[k].w);
            p = make_float2(gB.y - lh[k].x, gB.z - lh[k].y);
        }
        eout[(size_t)k * n + i] = o;
        hout[(size_t)k * n + i] = p;
    });
    // explicit fused multiply-adds wherever a product meets a sum (the same bits in every kernel)
    const float gEdotE = __fmaf_rn(gE.z, F.E.z, __fmaf_rn(gE.y, F.E.y, __fmul_rn(gE.x, F.E.x)));
    A.grad_eps[i] = geps_old + (geps_imposed - div_rn(gEdotE, er, 1.f / er));
    if (A.grad_sigma)
        A.grad_sigma[i] = gsig_old + __fmaf_rn(gJ.z, F.E.z, __fmaf_rn(gJ.y, F.E.y, __fmul_rn(gJ.x, F.E.x)));
}

// Source cells (skipped by the ordinary update through the mask) are stepped back at the end of
// their block (block_source_cells).
template <int M>
__global__ void __launch_bounds__(kBlock) hv_adjoint_kernel(AdjointArgs A) {
    wait_predecessor();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < A.a.g.n) hv_adjoint_cell<M, false, false>(A, i, 0);
    block_source_cells(A.a.sv, blockIdx.x, [&](int c, int m) { hv_adjoint_cell<M, true, false>(A, c, m); });
}

template <int M>
__global__ void __launch_bounds__(kBlock) hv_adjoint_terminal_kernel(AdjointArgs A, int n_plane) {
    after_predecessor();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_plane) return;
    hv_adjoint_cell<M, false, true>(A, plane_cell(A.a.g, A.plane_axis, A.plane_index, k), 0);
}

}  // namespace

int hv_launch_step(const StepArgs& a, cudaStream_t st) {
    int launched = 0;
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            const int nb = blocks_for(a.cell_end - a.cell_begin);
            if (a.sv.block_begin && nb <= kEarlySourceBlocks) launch_after(hv_step_early_kernel<S, M>, nb, kBlock, 0, st, a);
            else launch_after(hv_step_kernel<S, M>, nb, kBlock, 0, st, a);
            launched = 1;
        });
    });
    return launched;
}

int hv_launch_init(const StepArgs& a, const float* E, const float* B, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            launch_after(hv_init_kernel<S, M>, blocks_for(a.g.n), kBlock, 0, st, a, E, B);
        });
    });
    return 1;
}

int hv_launch_fields(const StepArgs& a, FieldsOut out, cudaStream_t st) {
    int launched = 0;
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            launch_after(hv_fields_kernel<S, M>, blocks_for(a.g.n), kBlock, 0, st, a, out);
            launched = 1;
            if (a.sv.n_special > 0 && a.cell_begin != 0) {
                launch_after(hv_fields_special_kernel<S, M>, blocks_for(a.sv.n_special), kBlock, 0, st, a, out);
                launched = 2;
            }
        });
    });
    return launched;
}

int hv_launch_get(const StepArgs& a, float* out, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        launch_after(hv_get_kernel<S>, blocks_for(a.g.n), kBlock, 0, st, a, out);
    });
    return 1;
}

int hv_launch_set(const StepArgs& a, const float* in, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        launch_after(hv_set_kernel<S>, blocks_for(a.g.n), kBlock, 0, st, a, in);
    });
    return 1;
}

int hv_launch_reduce(const StepArgs& a, double* partials, int n_blocks, double* result, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            launch_after(hv_reduce_kernel<S, M>, n_blocks, kBlock, 0, st, a, partials);
        });
    });
    return 1 + launch_reduce_partials(partials, n_blocks, result, st);
}

int hv_launch_batch_step(const BatchLaunch& b, int j, int n_tiles, int n_stiles, cudaStream_t st) {
    int launched = 0;
    with_storage(b.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        if (n_tiles > 0) {
            const int grid = b.grid_cap > 0 ? (n_tiles < b.grid_cap ? n_tiles : b.grid_cap) : n_tiles;
            if (b.block == 128) launch_after(hv_batch_kernel<S, 128>, grid, 128, 0, st, b.lat, b.tiles, n_tiles, j);
            else launch_after(hv_batch_kernel<S, 256>, grid, 256, 0, st, b.lat, b.tiles, n_tiles, j);
            ++launched;
        }
        if (n_stiles > 0) {
            launch_after(hv_batch_special_kernel<S>, n_stiles, kBlock, 0, st, b.lat, b.stiles, j);
            ++launched;
        }
    });
    return launched;
}

int hv_batch_occupancy(int storage, int block) {
    int blocks = 0;
    with_storage(storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        if (block == 128) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, hv_batch_kernel<S, 128>, 128, 0);
        else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, hv_batch_kernel<S, 256>, 256, 0);
    });
    return blocks;
}

int hv_launch_adjoint(const AdjointArgs& A, cudaStream_t st) {
    int launched = 0;
    with_media(A.a.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        launch_after(hv_adjoint_kernel<M>, blocks_for(A.a.g.n), kBlock, 0, st, A);
        launched = 1;
    });
    return launched;
}

int hv_launch_adjoint_terminal(const AdjointArgs& A, int n_plane, cudaStream_t st) {
    with_media(A.a.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        launch_after(hv_adjoint_terminal_kernel<M>, blocks_for(n_plane), kBlock, 0, st, A, n_plane);
    });
    return 1;
}

int hv_fused2_occupancy(int storage, int media_mode) {
    int blocks = 0;
    with_pass_storage(storage, [&](auto sc) {
        with_media(media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, hv_fused2_kernel<S, M>, kFusedThreads, 0);
        });
    });
    return blocks;
}

int hv_launch_fused2(const StepArgs& aA, const StepArgs& aB, const FusedArgs& F, cudaStream_t st) {
    if (aA.storage == kF24) return 0;  // no 24-bit form of the passes
    const int grid = fused_grid(hv_fused2_occupancy(aA.storage, aA.media_mode));
    with_pass_storage(aA.storage, [&](auto sc) {
        with_media(aA.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            hv_fused2_kernel<S, M><<<grid, kFusedThreads, 0, st>>>(aA, aB, F);
        });
    });
    return 1;
}

template <int S, int M>
bool hv_tile2_prepare() {
    static std::atomic<unsigned long long> done{0};
    return allow_shared(done, hv_tile2_kernel<S, M>, HVTile<S>::kBytes);
}

int hv_tile2_occupancy(int storage, int media_mode) {
    int blocks = 0;
    with_pass_storage(storage, [&](auto sc) {
        with_media(media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            if (!hv_tile2_prepare<S, M>() ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, hv_tile2_kernel<S, M>, Tile::kCells,
                                                              HVTile<S>::kBytes) != cudaSuccess) {
                cudaGetLastError();
                blocks = 0;
            }
        });
    });
    return blocks;
}

int hv_launch_tile2(const StepArgs& aA, const StepArgs& aB, const TileArgs& T, cudaStream_t st) {
    if (aA.storage == kF24) return 0;  // no 24-bit form of the passes
    const dim3 grid(T.tiles_x * T.tiles_y, (aA.g.nz + T.chunk - 1) / T.chunk);
    int launched = 0;
    with_pass_storage(aA.storage, [&](auto sc) {
        with_media(aA.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            if (!hv_tile2_prepare<S, M>()) return;  // the caller reads the error
            launch_after(hv_tile2_kernel<S, M>, grid, Tile::kCells, HVTile<S>::kBytes, st, aA, aB, T);
            launched = 1;
        });
    });
    return launched;
}

int hv_halo_dirs(int vz_sign, int* dirs) {
    int k = 0;
    for (int d = 0; d < 6; ++d)
        if (kHVAxis[d] == 2 && kHVSign[d] == vz_sign) dirs[k++] = d;
    return k;
}

int hv_launch_record_step(const StepArgs& a, cudaStream_t st) {
    int launched = 0;
    with_media(a.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        launch_after(hv_record_kernel<M>, blocks_for(a.g.n), kBlock, 0, st, a);
        launched = 1;
    });
    return launched;
}

}  // namespace lbm
