// Mendoza-Munoz (MM) model kernels, arXiv 2309.08068 Section II.
//
// One thread updates one cell. The 48 moving populations arrive as 12 vector pulls (one per D3Q13
// velocity; the four values of a velocity move together: a float4, or 8 bytes with 16-bit storage),
// the whole collision runs in FP32 registers, and the 12 results are stored at the cell (pull
// scheme). The ordinary update is branch-free; source and imposed cells are recomputed afterwards
// with their current and imposed fields, overwriting the ordinary result: at the end of their
// block in the single-step kernels (block_source_cells), in their tile in the two-step passes, and
// by a second small launch over the merged source-cell list in the batched kernels.
//
// Direction tables. Direction d = p*4 + (i-1) with the plane p and index i of eq.
// VelocitySetMiller: v_i^p = sqrt(2) (cos((2i-1) pi/4), sin((2i-1) pi/4)) in the xy (p = 0), xz
// (p = 1) and yz (p = 2) planes, which are the edge diagonals below. The electric vectors of eq.
// ElectromagneticVectorsMiller are e_{i0} = v_{[(i+2) mod 4]+1} / 2 and e_{i1} = v_{[i mod 4]+1} / 2
// = -e_{i0}; kMMEh holds 2 e_{i0}. The magnetic vectors b_{ij} = v_i x e_{ij} come out as -z for
// every direction of plane 0, +y for plane 1 and -x for plane 2, with b_{i1} = -b_{i0}.
//
// Because e_{i1} = -e_{i0} and b_{i1} = -b_{i0}, only the differences f_{d0} - f_{d1} enter the
// moments D' and B; the sums enter only rho_c. The collision below is written per velocity in
// terms of s = v.J/16, alpha = (eps_r/4) E.e0 + B.b0/(8 mu_r) and beta = E.e0/4 + B.b0/8:
//   f^(0)eq_{d0,d1} = s +- alpha,  f^(1)eq_{d0,d1} = s +- beta   (eq. equilibriumsMiller)
//   f' = 2 f^eq - f                                              (eq. CollisionMiller)
#include "mm_core.cuh"

namespace lbm {
namespace {

// 3 resident blocks for FP32 storage; 4 for 16-bit storage, whose halved bytes need more loads in
// flight per SM to reach the copy bandwidth (256^3 dipole on GB300, BF16: 0.475 against 0.497 ms
// per step at 3 blocks); 3 for 24-bit storage, whose decoding would spill at 64 registers.
// The block's source cells are recomputed at the end (block_source_cells).
template <int S, int M, bool kRho>
__global__ void __launch_bounds__(kBlock, S == kF32 || S == kF24 ? 3 : 4) mm_step_kernel(StepArgs a) {
    wait_predecessor();
    const int i = a.cell_begin + blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.cell_end) mm_update<S, M, false, kRho>(a, i, 0);
    block_source_cells(a.sv, blockIdx.x, [&](int c, int m) { mm_update<S, M, true, kRho>(a, c, m); });
}

// The same on a lattice of few waves of blocks, with its sources known early (early_source, which has the
// figures).
template <int S, int M>
__global__ void __launch_bounds__(kBlock, S == kF32 || S == kF24 ? 3 : 4) mm_step_early_kernel(StepArgs a) {
    const int i = a.cell_begin + blockIdx.x * blockDim.x + threadIdx.x;
    CellSource cs;
    const bool sources = early_source(a, blockIdx.x, i, &cs);
    wait_predecessor();
    if (i >= a.cell_end) return;
    if (sources) mm_update_sourced<S, M>(a, i, cs);
    else mm_update<S, M, false, false>(a, i, 0);
}

// Equilibrium populations of cell x for fields E, B and J = 0 (Appendix B initialisation).
template <int S, int M>
__global__ void __launch_bounds__(kBlock) mm_init_kernel(StepArgs a, const float* E, const float* B) {
    after_predecessor_by_size();
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= a.g.n) return;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, y);
    // Stored value at y for direction d is the population cell x = y + v_d pulls next step.
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        constexpr int e0 = kMMEh[d][0], e1 = kMMEh[d][1], e2 = kMMEh[d][2];
        constexpr int b0 = kMMB[d][0], b1 = kMMB[d][1], b2 = kMMB[d][2];
        const int x = shifted<kMMV[d][0], kMMV[d][1], kMMV[d][2]>(h);
        const MatCoef mat = load_coef<kModelMM, M>(a.media, x, a.eps0, a.mu0);
        const float ee = sdot<e0, e1, e2>(E[x], E[n + x], E[2 * n + x]);
        const float bb = sdot<b0, b1, b2>(B[x], B[n + x], B[2 * n + x]);
        const float alpha = __fmaf_rn(bb, 0.5f * mat.c0.w, 0.125f * __fmul_rn(mat.c0.x, ee));  // 0.5 / (4 mu_r)
        const float beta = 0.125f * ee + 0.125f * bb;
        mm_put<S>(a, d, y, make_float4(alpha, -alpha, beta, -beta));
    });
}

// Fields of cell i; m is its index in the special-cell list when kSpecial.
template <int S, int M, bool kSpecial>
__device__ __forceinline__ void mm_fields_cell(const StepArgs& a, const FieldsOut& out, int i, int m) {
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, i);
    float4 f[12];
    mm_pull<S>(a, h, f);
    const MatCoef mat = load_coef<kModelMM, M>(a.media, i, a.eps0, a.mu0);
    float3 jext = make_float3(0.f, 0.f, 0.f);
    if constexpr (kSpecial) jext = cell_source(a.sv, a.sc, m).J;
    const MMFields F = mm_fields<false>(f, 0.f, mat, jext);
    auto put = [&](float* p, float3 v) {
        if (p) {
            p[i] = v.x;
            p[n + i] = v.y;
            p[2 * n + i] = v.z;
        }
    };
    put(out.E, F.E);
    put(out.B, F.B);
    put(out.D, F.Dpp);  // D = eps0 eps_r E with eps0 = 1
    // H = B / (mu0 mu_r) with mu0 = 2; 1 / (2 mu_r) = 2 / (4 mu_r) exactly
    const float two_mu = 2.f * mat.c1.y, inv2mu = 2.f * mat.c0.w;
    put(out.H, make_float3(div_rn(F.B.x, two_mu, inv2mu), div_rn(F.B.y, two_mu, inv2mu),
                           div_rn(F.B.z, two_mu, inv2mu)));
    put(out.J, F.J);
}

// Every cell, and, where the blocks' source-cell offsets cover the whole lattice (not a z-slab, whose
// offsets cover the stepped planes), the block's source cells after them.
template <int S, int M>
__global__ void __launch_bounds__(kBlock) mm_fields_kernel(StepArgs a, FieldsOut out) {
    after_predecessor();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.g.n) mm_fields_cell<S, M, false>(a, out, i, 0);
    if (a.cell_begin == 0)
        block_source_cells(a.sv, blockIdx.x, [&](int c, int m) { mm_fields_cell<S, M, true>(a, out, c, m); });
}

template <int S, int M>
__global__ void __launch_bounds__(kBlock) mm_fields_special_kernel(StepArgs a, FieldsOut out) {
    after_predecessor();
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < a.sv.n_special) mm_fields_cell<S, M, true>(a, out, a.sv.cell[m], m);
}

// Canonical layout out[k * n + x]: k = r*24 + p*8 + (i-1)*2 + j = r*24 + 2d + j; 48, 49 rest.
template <int S>
__global__ void __launch_bounds__(kBlock) mm_get_kernel(StepArgs a, const float* rest1,
                                                        float* __restrict__ out) {
    after_predecessor();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= a.g.n) return;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, x);
    float4 f[12];
    mm_pull<S>(a, h, f);
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        out[(size_t)(2 * d) * n + x] = f[d].x;
        out[(size_t)(2 * d + 1) * n + x] = f[d].y;
        out[(size_t)(24 + 2 * d) * n + x] = f[d].z;
        out[(size_t)(25 + 2 * d) * n + x] = f[d].w;
    });
    out[(size_t)48 * n + x] = a.rho_in ? a.rho_in[x] : 0.f;
    out[(size_t)49 * n + x] = rest1 ? rest1[x] : 0.f;
}

template <int S>
__global__ void __launch_bounds__(kBlock) mm_set_kernel(StepArgs a, const float* in,
                                                        float* __restrict__ rest1) {
    after_predecessor_by_size();
    const int y = blockIdx.x * blockDim.x + threadIdx.x;
    if (y >= a.g.n) return;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, y);
    float4 f[12];  // every load before the first store, which the loads could not be moved across
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        const int x = shifted<kMMV[d][0], kMMV[d][1], kMMV[d][2]>(h);
        f[d] = make_float4(in[(size_t)(2 * d) * n + x], in[(size_t)(2 * d + 1) * n + x],
                           in[(size_t)(24 + 2 * d) * n + x], in[(size_t)(25 + 2 * d) * n + x]);
    });
    static_for<0, 12>([&](auto dc) { mm_put<S>(a, decltype(dc)::value, y, f[decltype(dc)::value]); });
    if (a.rho_out) a.rho_out[y] = in[(size_t)48 * n + y];
    if (rest1) rest1[y] = in[(size_t)49 * n + y];
}

// Per-block partial sums of (1/2)(E.D + B.H), sum f^2 and rho_c over a grid-stride range of cells
// (external current taken as zero here; the special-cell pass adds the correction).
template <int S, int M, bool kRho>
__global__ void __launch_bounds__(kBlock) mm_reduce_kernel(StepArgs a, const float* rest1,
                                                           double* __restrict__ partials) {
    after_predecessor();
    double w = 0.0, f2 = 0.0, q = 0.0;
    for (int i = a.cell_begin + blockIdx.x * blockDim.x + threadIdx.x; i < a.cell_end; i += gridDim.x * blockDim.x) {
        const Neighbourhood h = neighbourhood(a.g, i);
        float4 f[12];
        mm_pull<S>(a, h, f);
        const MatCoef mat = load_coef<kModelMM, M>(a.media, i, a.eps0, a.mu0);
        float rest0 = 0.f;
        if constexpr (kRho) rest0 = a.rho_in[i];
        const MMFields F = mm_fields<kRho>(f, rest0, mat, make_float3(0.f, 0.f, 0.f));
        const double inv2mu = 1.0 / (2.0 * (double)mat.c1.y);
        w += 0.5 * ((double)F.E.x * F.Dpp.x + (double)F.E.y * F.Dpp.y + (double)F.E.z * F.Dpp.z) +
             0.5 * inv2mu * ((double)F.B.x * F.B.x + (double)F.B.y * F.B.y + (double)F.B.z * F.B.z);
        double s = 0.0;
#pragma unroll
        for (int d = 0; d < 12; ++d)
            s += (double)f[d].x * f[d].x + (double)f[d].y * f[d].y + (double)f[d].z * f[d].z +
                 (double)f[d].w * f[d].w;
        if constexpr (kRho) {
            s += (double)rest0 * rest0;
            q += F.rho;
        }
        if (rest1) s += (double)rest1[i] * rest1[i];
        f2 += s;
    }
    block_sum3_store(w, f2, q, partials + 3 * blockIdx.x);
}

// Energy correction at source cells: (energy with J_ext) - (energy with J_ext = 0).
template <int S, int M>
__global__ void __launch_bounds__(kBlock) mm_reduce_special_kernel(StepArgs a, double* __restrict__ partials) {
    after_predecessor();
    double w = 0.0;
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m < a.sv.n_special) {
        const int i = a.sv.cell[m];
        const Neighbourhood h = neighbourhood(a.g, i);
        float4 f[12];
        mm_pull<S>(a, h, f);
        const MatCoef mat = load_coef<kModelMM, M>(a.media, i, a.eps0, a.mu0);
        const MMFields F1 = mm_fields<false>(f, 0.f, mat, cell_source(a.sv, a.sc, m).J);
        const MMFields F0 = mm_fields<false>(f, 0.f, mat, make_float3(0.f, 0.f, 0.f));
        w = 0.5 * ((double)F1.E.x * F1.Dpp.x + (double)F1.E.y * F1.Dpp.y + (double)F1.E.z * F1.Dpp.z) -
            0.5 * ((double)F0.E.x * F0.Dpp.x + (double)F0.E.y * F0.Dpp.y + (double)F0.E.z * F0.Dpp.z);
    }
    block_sum3_store(w, 0.0, 0.0, partials + 3 * blockIdx.x);
}

// Batched step j of several lattices: each block takes tiles (lattice, first cell) in turn; with a
// grid smaller than the tile count the blocks persist and stride over the tiles.
template <int S, int BLOCK, bool kRho>
__global__ void __launch_bounds__(BLOCK, 768 / BLOCK) mm_batch_kernel(const BatchLattice* __restrict__ lat,
                                                                        const BatchTile* __restrict__ tiles,
                                                                        int n_tiles, int j) {
    wait_predecessor();
    for (int b = blockIdx.x; b < n_tiles; b += gridDim.x) {
        const BatchTile tile = tiles[b];
        const BatchLattice* L = &lat[tile.lattice];
        const int i = tile.begin + threadIdx.x;
        if (j >= L->steps || i >= L->base.g.n) continue;
        const StepArgs a = batch_args(L, j);
        switch (a.media_mode) {
            case kUniform: mm_update<S, kUniform, false, kRho>(a, i, 0); break;
            case kTable: mm_update<S, kTable, false, kRho>(a, i, 0); break;
            default: mm_update<S, kPerCell, false, kRho>(a, i, 0); break;
        }
    }
}

template <int S, bool kRho>
__global__ void __launch_bounds__(kBlock) mm_batch_special_kernel(const BatchLattice* __restrict__ lat,
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
        case kUniform: mm_update<S, kUniform, true, kRho>(a, i, m); break;
        case kTable: mm_update<S, kTable, true, kRho>(a, i, m); break;
        default: mm_update<S, kPerCell, true, kRho>(a, i, m); break;
    }
}

template <int M, bool kRho>
__global__ void __launch_bounds__(kBlock, 3) mm_record_kernel(StepArgs a) {
    wait_predecessor();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < a.g.n) mm_update<kF32, M, false, kRho, true>(a, i, 0);
    block_source_cells(a.sv, blockIdx.x, [&](int c, int m) { mm_update<kF32, M, true, kRho, true>(a, c, m); });
}

// ---------------------------------------------------------------------------------------------
// Two steps per pass (see FusedArgs). Phase A reads the A/B buffer once (streaming loads that L2
// may evict first) and writes the intermediate plane; phase B pulls from the intermediate planes
// (L2 loads: they were written by other blocks of this launch) and writes the other A/B buffer
// once (streaming stores). The arithmetic is mm_update's, so the pair of steps gives the same
// bits as two single steps.
template <int S>
struct MMToRing : FusedStash {
    using T = typename Pack4<S>::T;
    T* plane;  // slot of this cell's plane
    int base;  // first cell of the plane
    int nxy;
    template <int S2>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&f)[12]) const {
        const T* fin = static_cast<const T*>(a.fin);
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            const int src = shifted<-kMMV[d][0], -kMMV[d][1], -kMMV[d][2]>(h);
            f[d] = Pack4<S>::unpack(__ldcs(fin + (size_t)d * a.g.n + src), a.inv_scale);
        });
    }
    template <int S2>
    __device__ void put(const StepArgs& a, int d, int i, float4 v) const {
        __stcg(plane + (size_t)d * nxy + (i - base), Pack4<S>::pack(v, a.scale));
    }
};

template <int S>
struct MMFromRing : FusedStash {
    using T = typename Pack4<S>::T;
    const T* plane[3];  // slots of planes z - 1, z, z + 1
    int nxy;
    template <int S2>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&f)[12]) const {
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            constexpr int sx = -kMMV[d][0], sy = -kMMV[d][1], sz = -kMMV[d][2];
            const T* src = plane[sz + 1] + (size_t)d * nxy + h.xo[sx + 1] + h.yo[sy + 1];
            f[d] = Pack4<S>::unpack(__ldcg(src), a.inv_scale);
        });
    }
    template <int S2>
    __device__ void put(const StepArgs& a, int d, int i, float4 v) const {
        T* __restrict__ fout = static_cast<T*>(a.fout);
        __stcs(fout + (size_t)d * a.g.n + i, Pack4<S>::pack(v, a.scale));
    }
};

template <int S, int M>
__global__ void __launch_bounds__(kFusedThreads, 3) mm_fused2_kernel(StepArgs aA, StepArgs aB, FusedArgs F) {
    using T = typename Pack4<S>::T;
    __shared__ float2 s_stash[12 * kBlock];  // the f^(1) halves, [velocity][compute thread]
    const unsigned stash = fused_stash_slot(s_stash);
    const int nz = aA.g.nz, nxy = aA.g.nx * aA.g.ny;
    auto slot = [&](int p) -> T* {
        if (p == 0) return static_cast<T*>(F.lo);
        if (p == nz - 1) return static_cast<T*>(F.hi);
        return static_cast<T*>(F.ring) + (size_t)(p % F.R) * 12 * nxy;
    };
    auto describe = [&](const FusedItem& it, FusedDesc& d) {
        if (it.type == kPhaseA) {
            d.ptr[0] = slot(it.plane);
        } else {
            d.ptr[0] = slot((it.plane + nz - 1) % nz);
            d.ptr[1] = slot(it.plane);
            d.ptr[2] = slot((it.plane + 1) % nz);
        }
    };
    fused_loop(F, aA.g.nx, nxy, nz, describe, [&](const FusedDesc& d) {
        const int j = d.j, base = d.plane * nxy;
        if (d.type == kPhaseA) {
            const MMToRing<S> io{{stash}, static_cast<T*>(d.ptr[0]), base, nxy};
            const int end = min(base + (j + 1) * F.tile_cells, base + nxy);
            for (int i = base + j * F.tile_cells + threadIdx.x; i < end; i += kBlock)
                mm_update<S, M, false, false, false>(aA, i, 0, io);
            if (d.s_hi > d.s_lo) {  // the tile's source cells replace their ordinary update
                named_sync(kComputeBarrier, kBlock);
                for (int m = d.s_lo + threadIdx.x; m < d.s_hi; m += kBlock)
                    mm_update<S, M, true, false, false>(aA, aA.sv.cell[m], m, io);
            }
        } else {
            const MMFromRing<S> io{{stash},
                                   {static_cast<const T*>(d.ptr[0]), static_cast<const T*>(d.ptr[1]),
                                    static_cast<const T*>(d.ptr[2])},
                                   nxy};
            const int end = min(base + (j + 1) * F.tile_cells, base + nxy);
            for (int i = base + j * F.tile_cells + threadIdx.x; i < end; i += kBlock)
                mm_update<S, M, false, false, false>(aB, i, 0, io);
            if (d.s_hi > d.s_lo) {  // the tile's source cells replace their ordinary update
                named_sync(kComputeBarrier, kBlock);
                for (int m = d.s_lo + threadIdx.x; m < d.s_hi; m += kBlock)
                    mm_update<S, M, true, false, false>(aB, aB.sv.cell[m], m, io);
            }
        }
    });
}

// ---------------------------------------------------------------------------------------------
// Two steps per pass over shared-memory tiles (see TileArgs). Directions by v_z: class 0 (in-plane,
// d = 0..3), class 1 (v_z = +1: d = 4, 5, 8, 9), class 2 (v_z = -1: d = 6, 7, 10, 11); four
// directions per class.
__host__ __device__ constexpr int mm_zclass(int d) { return d < 4 ? 0 : (((d >> 1) & 1) ? 2 : 1); }
__host__ __device__ constexpr int mm_zrank(int d) { return d < 4 ? d : (d & 1) + (d >= 8 ? 2 : 0); }
static_assert(mm_zclass(4) == 1 && mm_zclass(9) == 1 && mm_zclass(6) == 2 && mm_zclass(11) == 2 &&
                  mm_zrank(8) == 2 && mm_zrank(10) == 2 && mm_zrank(7) == 1,
              "v_z classes of the D3Q13 velocity table");

// Six slots of 4 directions x Tile::kCells cells: slot 0 the class-2 directions of the newest
// plane, slots 1-2 class 0 of the last two planes, slots 3-5 class 1 of the last three.
template <int S>
struct MMTile {
    using T = typename Pack4<S>::T;
    static constexpr size_t kBytes = 6 * 4 * Tile::kCells * sizeof(T);
    T* base;
    __device__ T* slot(int cls, int p) const {  // plane p >= -1
        const int s = cls == 2 ? 0 : (cls == 0 ? 1 + (p + 3) % 2 : 3 + (p + 3) % 3);
        return base + (size_t)s * 4 * Tile::kCells;
    }
};

// Phase A: pulls from the A/B buffer, results into the tile's slots of plane p.
template <int S>
struct MMToTile : NoStash {
    using T = typename Pack4<S>::T;
    T* dst[3];  // slots of plane p, by class
    int local;  // extended-tile position of the cell
    bool own;   // a cell of the block's own tile and planes: a recording pass writes its record
    __device__ bool keeps_record() const { return own; }
    template <int S2>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&f)[12]) const {
        mm_pull<S, true>(a, h, f);  // the kernel is launched plainly
    }
    template <int S2>
    __device__ void put(const StepArgs& a, int d, int, float4 v) const {
        dst[mm_zclass(d)][mm_zrank(d) * Tile::kCells + local] = Pack4<S>::pack(v, a.scale);
    }
};

// Phase B: pulls from the tile (class 0 from plane q, class 1 from q - 1, class 2 from q + 1),
// results into the other A/B buffer.
template <int S>
struct MMFromTile : NoStash {
    using T = typename Pack4<S>::T;
    const T* src[3];
    int local;
    template <int S2>
    __device__ void pull(const StepArgs& a, const Neighbourhood&, float4 (&f)[12]) const {
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            static_assert(kMMV[d][2] == (mm_zclass(d) == 0 ? 0 : (mm_zclass(d) == 1 ? 1 : -1)), "class of d");
            constexpr int off = mm_zrank(d) * Tile::kCells - (kMMV[d][0] + kMMV[d][1] * Tile::EX);
            f[d] = Pack4<S>::unpack(src[mm_zclass(d)][off + local], a.inv_scale);
        });
    }
    template <int S2>
    __device__ void put(const StepArgs& a, int d, int i, float4 v) const {
        T* __restrict__ fout = static_cast<T*>(a.fout);
        __stcs(fout + (size_t)d * a.g.n + i, Pack4<S>::pack(v, a.scale));
    }
};

// kRecord: both steps also write the adjoint's per-cell records (aA.rec, aB.rec), each cell's once,
// by the block that owns it.
// Launched plainly, not while its predecessor runs: the input buffer is then read-only for the kernel's
// lifetime, which lets the compiler move its loads across the barriers of a plane (read-only loads 592 us
// per step at 256^3, plain ones 637; the launch costs about 2 us per pass).
template <int S, int M, bool kRecord = false>
__global__ void __launch_bounds__(Tile::kCells, S == kF32 ? 2 : 3) mm_tile2_kernel(StepArgs aA, StepArgs aB,
                                                                                    TileArgs T) {
    let_successor();
    using TT = typename Pack4<S>::T;
    extern __shared__ __align__(16) unsigned char mm_tile_smem[];
    const MMTile<S> tile{reinterpret_cast<TT*>(mm_tile_smem)};
    const int nz = aA.g.nz, nxy = aA.g.nx * aA.g.ny;
    const TileCell c = tile_cell<Tile>(aA.g, T, threadIdx.x);
    const int cxy = c.row + c.x;
    const int* off = T.entry_off + (size_t)c.tile * nz;
    for (int p = c.z0 - 1; p <= c.z1; ++p) {
        const int pz = tile_wrap(p, nz);
        // The next plane's phase-A inputs, fetched into L2 while this plane is stepped: a plane's
        // loads are otherwise a DRAM round trip that two blocks per SM cannot hide.
        if (p < c.z1) mm_prefetch<S, M>(aA, tile_wrap(p + 1, nz) * nxy + cxy);
        {  // phase A: step t of the extended tile's cells of plane pz
            const bool own_plane = p >= c.z0 && p < c.z1;
            const MMToTile<S> io{{}, {tile.slot(0, p), tile.slot(1, p), tile.slot(2, p)}, (int)threadIdx.x,
                                 own_plane && c.core};
            mm_update<S, M, false, false, kRecord>(aA, pz * nxy + cxy, 0, io);
            const int lo = off[pz], hi = off[pz + 1];
            if (hi > lo) {  // the source cells among them replace their ordinary update
                __syncthreads();
                for (int k = lo + threadIdx.x; k < hi; k += Tile::kCells) {
                    const int2 e = T.entries[k];
                    const MMToTile<S> sio{{}, {io.dst[0], io.dst[1], io.dst[2]}, e.y,
                                          own_plane && tile_core<Tile>(e.y, c.bx, c.by, aA.g.nx, aA.g.ny)};
                    mm_update<S, M, true, false, kRecord>(aA, aA.sv.cell[e.x], e.x, sio);
                }
            }
        }
        __syncthreads();
        if (p > c.z0) {  // phase B: step t + 1 of the tile's own cells of plane q = p - 1
            const int q = p - 1;
            const MMFromTile<S> io{{}, {tile.slot(0, q), tile.slot(1, q - 1), tile.slot(2, q + 1)}, (int)threadIdx.x};
            if (c.core) mm_update<S, M, false, false, kRecord>(aB, q * nxy + cxy, 0, io);
            const int lo = off[q], hi = off[q + 1];
            if (hi > lo) {
                __syncthreads();
                for (int k = lo + threadIdx.x; k < hi; k += Tile::kCells) {
                    const int2 e = T.entries[k];
                    if (!tile_core<Tile>(e.y, c.bx, c.by, aA.g.nx, aA.g.ny)) continue;
                    const MMFromTile<S> sio{{}, {io.src[0], io.src[1], io.src[2]}, e.y};
                    mm_update<S, M, true, false, kRecord>(aB, aB.sv.cell[e.x], e.x, sio);
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------------------------
// Adjoint of one MM step. With per-velocity adjoints (a0^, a1^, c0^, c1^) of the post-collision
// values, the transpose of eq. CollisionMiller through eq. equilibriumsMiller is
//   adjoint of 2s_d = a0^ + a1^ + c0^ + c1^,  of 2 alpha_d = a0^ - a1^,  of 2 beta_d = c0^ - c1^,
//   gJ = sum_d (2s_d)^ v_d / 8,   gE = sum_d (2 beta_d)^ e_d / 2 + sigma gJ   (e_d = e_{d0}, e_h = 2 e_d),
//   gB = sum_d [(2 alpha_d)^ / (4 mu_r) + (2 beta_d)^ / 4] b_d,
//   gDpp = sum_d (2 alpha_d)^ e_d / 2 + gE / eps_r   (E = Dpp / eps_r),   gX = g gDpp   (Dpp = X g),
//   D' = sum_d (f_d0 - f_d1) e_d  ->  nu(f_d0) = e_d . gX - a0^,  nu(f_d1) = -e_d . gX - a1^,
//   B  = sum_d (f'_d0 - f'_d1) b_d ->  nu(c0) = b_d . gB - c0^,  nu(c1) = -b_d . gB - c1^,
// and the parameter derivatives (g = 1 / (1 + mu0 sigma / (4 eps_r)), mu0 = 2):
//   dL/d eps_r += -gE . E / eps_r + gDpp . X * g^2 sigma / (2 eps_r^2),
//   dL/d sigma += gJ . E - gDpp . X * g^2 / (2 eps_r).
// Imposed cells output f_eq(E_imp, B_imp, 0): nothing flows back to f, and
// d alpha_d / d eps_r = e_h . E_imp / 8. The plane loss |E|^2 adds 2E to gE.
// Where a backward step reads lambda, writes nu^n and adds its gradient terms. (Written out in
// mm_adjoint_cell instead, the same operations spill more: 128^3 with a medium per cell 265 us per step
// against 261.)
// kReadOnly: see read().
template <bool kReadOnly>
struct MMAdjGlobal {
    __device__ void lam(const AdjointArgs& A, const Neighbourhood& h, float4 (&lam)[12]) const {
        const int n = A.a.g.n;
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            const int dst = shifted<kMMV[d][0], kMMV[d][1], kMMV[d][2]>(h);
            lam[d] = read<kReadOnly>(static_cast<const float4*>(A.nu_in) + (size_t)d * n + dst);
        });
    }
    __device__ void put_nu(const AdjointArgs& A, int d, int i, float4 o) const {
        static_cast<float4*>(A.nu_out)[(size_t)d * A.a.g.n + i] = o;
    }
    __device__ void grad_load(const AdjointArgs& A, int i, float& ge, float& gs) const {
        ge = A.grad_eps[i];
        if (A.grad_sigma) gs = A.grad_sigma[i];
    }
    __device__ void grad_store(const AdjointArgs& A, int i, float ge, float gs) const {
        A.grad_eps[i] = ge;
        if (A.grad_sigma) A.grad_sigma[i] = gs;
    }
};

template <int M, bool kSpecial, bool kTerminal, bool kReadOnly = false>
__device__ __forceinline__ void mm_adjoint_cell(const AdjointArgs& A, int i, int m) {
    const MMAdjGlobal<kReadOnly> io;
    const StepArgs& a = A.a;
    const int n = a.g.n;
    const Neighbourhood h = neighbourhood(a.g, i);
    const MatCoef mat = load_coef<kModelMM, M>(a.media, i, a.eps0, a.mu0);
    CellSource cs;
    bool imposed = false;
    if constexpr (kSpecial) {
        cs = cell_source(a.sv, a.sc, m);
        imposed = cs.imposed;
    }
    // Every load is issued up front: the source-cell mask of the main launch only gates the stores,
    // so it adds no round trip before the others.
    const bool skip = !kSpecial && !kTerminal && A.special_mask[i] != 0;
    float geps_old = 0.f, gsig_old = 0.f;
    io.grad_load(A, i, geps_old, gsig_old);
    // E and X of f^n: X from the forward step's record (E recomputed from it), or (terminal) the final state
    float3 E, X;
    if constexpr (kTerminal) {
        float4 f[12];
        mm_pull<kF32>(a, h, f);
        const MMFields F = mm_fields<false>(f, 0.f, mat, make_float3(0.f, 0.f, 0.f));
        E = F.E;
        X = F.X;
    } else {
        X = make_float3(read<kReadOnly>(&a.rec[i]), read<kReadOnly>(&a.rec[n + i]), read<kReadOnly>(&a.rec[2 * n + i]));
        E = mm_e_of_dpp(mm_dpp(X, mat.c0.z), mat.c0.x, mat.c0.y);  // as the forward step computed it
    }
    struct {
        float3 E, X;
    } F{E, X};
    const float inv_er = mat.c0.y, g = mat.c0.z, inv4mu = mat.c0.w, sigma = mat.c1.x;
    float4 lam[12];
    if constexpr (kTerminal) {
        static_for<0, 12>([&](auto dc) { lam[decltype(dc)::value] = make_float4(0.f, 0.f, 0.f, 0.f); });
    } else {
        io.lam(A, h, lam);
    }
    float gJx = 0.f, gJy = 0.f, gJz = 0.f, gAx = 0.f, gAy = 0.f, gAz = 0.f, gEx = 0.f, gEy = 0.f, gEz = 0.f;
    float gBx = 0.f, gBy = 0.f, gBz = 0.f, geps_imposed = 0.f;
    if (!imposed) {
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            const float s2 = (lam[d].x + lam[d].y) + (lam[d].z + lam[d].w);
            const float a2 = lam[d].x - lam[d].y, b2 = lam[d].z - lam[d].w;
            acc<kMMV[d][0]>(gJx, s2);
            acc<kMMV[d][1]>(gJy, s2);
            acc<kMMV[d][2]>(gJz, s2);
            acc<kMMEh[d][0]>(gAx, a2);
            acc<kMMEh[d][1]>(gAy, a2);
            acc<kMMEh[d][2]>(gAz, a2);
            acc<kMMEh[d][0]>(gEx, b2);
            acc<kMMEh[d][1]>(gEy, b2);
            acc<kMMEh[d][2]>(gEz, b2);
            const float bcoef = __fmaf_rn(a2, inv4mu, 0.25f * b2);
            acc<kMMB[d][0]>(gBx, bcoef);
            acc<kMMB[d][1]>(gBy, bcoef);
            acc<kMMB[d][2]>(gBz, bcoef);
        });
        gJx *= 0.125f; gJy *= 0.125f; gJz *= 0.125f;
        gEx = __fmaf_rn(sigma, gJx, 0.25f * gEx);
        gEy = __fmaf_rn(sigma, gJy, 0.25f * gEy);
        gEz = __fmaf_rn(sigma, gJz, 0.25f * gEz);
    } else if constexpr (kSpecial) {
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            const float ee = sdot<kMMEh[d][0], kMMEh[d][1], kMMEh[d][2]>(cs.E.x, cs.E.y, cs.E.z);
            geps_imposed = __fmaf_rn(lam[d].x - lam[d].y, 0.125f * ee, geps_imposed);
        });
    }
    if (A.loss_active && in_plane(h, a.g, A.plane_axis, A.plane_index)) {  // |E|^2 of time n
        gEx = __fmaf_rn(2.f, F.E.x, gEx);
        gEy = __fmaf_rn(2.f, F.E.y, gEy);
        gEz = __fmaf_rn(2.f, F.E.z, gEz);
        add_plane_loss<kTerminal>(A, h, F.E);
    }
    const float gDx = __fmaf_rn(gEx, inv_er, 0.25f * gAx), gDy = __fmaf_rn(gEy, inv_er, 0.25f * gAy),
                gDz = __fmaf_rn(gEz, inv_er, 0.25f * gAz);
    // __fmul_rn: the products must not fuse into the sums below differently in different kernels
    const float gXx = __fmul_rn(g, gDx), gXy = __fmul_rn(g, gDy), gXz = __fmul_rn(g, gDz);
    if (skip) return;  // a source cell: the source-cell pass writes it
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        const float gde = 0.5f * sdot<kMMEh[d][0], kMMEh[d][1], kMMEh[d][2]>(gXx, gXy, gXz);
        const float gdb = sdot<kMMB[d][0], kMMB[d][1], kMMB[d][2]>(gBx, gBy, gBz);
        float4 o;
        if (imposed) o = make_float4(gde, -gde, gdb, -gdb);
        else o = make_float4(gde - lam[d].x, -gde - lam[d].y, gdb - lam[d].z, -gdb - lam[d].w);
        io.put_nu(A, d, i, o);
    });
    // explicit fused multiply-adds wherever a product meets a sum (the same bits in every kernel)
    const float gEdotE = __fmaf_rn(gEz, F.E.z, __fmaf_rn(gEy, F.E.y, __fmul_rn(gEx, F.E.x)));
    const float gDdotX = __fmaf_rn(gDz, F.X.z, __fmaf_rn(gDy, F.X.y, __fmul_rn(gDx, F.X.x)));
    const float gJdotE = __fmaf_rn(gJz, F.E.z, __fmaf_rn(gJy, F.E.y, __fmul_rn(gJx, F.E.x)));
    const float gg = g * g * inv_er;
    float deps = __fmaf_rn(-gEdotE, inv_er, geps_imposed);
    deps = __fmaf_rn(gDdotX, gg * 0.5f * sigma * inv_er, deps);
    const float dsig = __fmaf_rn(-gDdotX, 0.5f * gg, gJdotE);
    io.grad_store(A, i, geps_old + deps, gsig_old + dsig);
}

// Source cells (skipped by the ordinary update through the mask) are stepped back at the end of
// their block (block_source_cells).
// kReadOnly: launched plainly, so that nu^{n+1} and the record are read-only for its lifetime. Plain loads
// spill more, 112 bytes a thread against 72 with a medium per cell: on large lattices of that kind the plain
// launch costs less (128^3, 64 steps in segments of 8: 367.8 us per step against 371.5; 112^3 235.2 / 237.3;
// 96^3 150.9 / 150.2; 64^3 48.5 / 46.8). Uniform media and tables: 322.7 and 336.5 with plain loads, 324.4 and
// 336.2 launched plainly at 128^3.
constexpr int kReadOnlyBackwardCells = 1200000;
template <int M, bool kReadOnly>
__global__ void __launch_bounds__(kBlock, 3) mm_adjoint_kernel(AdjointArgs A) {
    if constexpr (kReadOnly) let_successor();
    else wait_predecessor();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < A.a.g.n) mm_adjoint_cell<M, false, false, kReadOnly>(A, i, 0);
    block_source_cells(A.a.sv, blockIdx.x, [&](int c, int m) { mm_adjoint_cell<M, true, false, kReadOnly>(A, c, m); });
}

template <int M>
__global__ void __launch_bounds__(kBlock) mm_adjoint_terminal_kernel(AdjointArgs A, int n_plane) {
    after_predecessor();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_plane) return;
    mm_adjoint_cell<M, false, true>(A, plane_cell(A.a.g, A.plane_axis, A.plane_index, k), 0);
}

}  // namespace

int mm_launch_step(const StepArgs& a, cudaStream_t st) {
    const bool rho = a.rho_in != nullptr;
    int launched = 0;
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            const int nb = blocks_for(a.cell_end - a.cell_begin);
            if (rho) launch_after(mm_step_kernel<S, M, true>, nb, kBlock, 0, st, a);
            else if (a.sv.block_begin && nb <= kEarlySourceBlocks) launch_after(mm_step_early_kernel<S, M>, nb, kBlock, 0, st, a);
            else launch_after(mm_step_kernel<S, M, false>, nb, kBlock, 0, st, a);
            launched = 1;
        });
    });
    return launched;
}

int mm_launch_init(const StepArgs& a, const float* E, const float* B, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            launch_after(mm_init_kernel<S, M>, blocks_for(a.g.n), kBlock, 0, st, a, E, B);
        });
    });
    return 1;
}

int mm_launch_fields(const StepArgs& a, FieldsOut out, cudaStream_t st) {
    int launched = 0;
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            launch_after(mm_fields_kernel<S, M>, blocks_for(a.g.n), kBlock, 0, st, a, out);
            launched = 1;
            if (a.sv.n_special > 0 && a.cell_begin != 0) {
                launch_after(mm_fields_special_kernel<S, M>, blocks_for(a.sv.n_special), kBlock, 0, st, a, out);
                launched = 2;
            }
        });
    });
    return launched;
}

int mm_launch_get(const StepArgs& a, float* out, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        launch_after(mm_get_kernel<S>, blocks_for(a.g.n), kBlock, 0, st, a, static_cast<const float*>(a.fin2), out);
    });
    return 1;
}

int mm_launch_set(const StepArgs& a, const float* in, cudaStream_t st) {
    with_storage(a.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        launch_after(mm_set_kernel<S>, blocks_for(a.g.n), kBlock, 0, st, a, in, static_cast<float*>(a.fout2));
    });
    return 1;
}

int mm_launch_reduce(const StepArgs& a, double* partials, int n_blocks, double* result, cudaStream_t st) {
    const bool rho = a.rho_in != nullptr;
    const float* rest1 = static_cast<const float*>(a.fin2);
    int total = n_blocks, launched = 1;
    with_storage(a.storage, [&](auto sc) {
        with_media(a.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            if (rho) launch_after(mm_reduce_kernel<S, M, true>, n_blocks, kBlock, 0, st, a, rest1, partials);
            else launch_after(mm_reduce_kernel<S, M, false>, n_blocks, kBlock, 0, st, a, rest1, partials);
            if (a.sv.n_special > 0) {
                const int ns = blocks_for(a.sv.n_special);
                launch_after(mm_reduce_special_kernel<S, M>, ns, kBlock, 0, st, a, partials + 3 * n_blocks);
                total += ns;
                ++launched;
            }
        });
    });
    return launched + launch_reduce_partials(partials, total, result, st);
}

int mm_launch_batch_step(const BatchLaunch& b, int j, int n_tiles, int n_stiles, cudaStream_t st) {
    int launched = 0;
    with_storage(b.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        if (n_tiles > 0) {
            const int grid = b.grid_cap > 0 ? (n_tiles < b.grid_cap ? n_tiles : b.grid_cap) : n_tiles;
            if (b.block == 128) {
                if (b.rho) launch_after(mm_batch_kernel<S, 128, true>, grid, 128, 0, st, b.lat, b.tiles, n_tiles, j);
                else launch_after(mm_batch_kernel<S, 128, false>, grid, 128, 0, st, b.lat, b.tiles, n_tiles, j);
            } else {
                if (b.rho) launch_after(mm_batch_kernel<S, 256, true>, grid, 256, 0, st, b.lat, b.tiles, n_tiles, j);
                else launch_after(mm_batch_kernel<S, 256, false>, grid, 256, 0, st, b.lat, b.tiles, n_tiles, j);
            }
            ++launched;
        }
        if (n_stiles > 0) {
            if (b.rho) launch_after(mm_batch_special_kernel<S, true>, n_stiles, kBlock, 0, st, b.lat, b.stiles, j);
            else launch_after(mm_batch_special_kernel<S, false>, n_stiles, kBlock, 0, st, b.lat, b.stiles, j);
            ++launched;
        }
    });
    return launched;
}

int mm_batch_occupancy(int storage, int block, bool rho) {
    int blocks = 0;
    with_storage(storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        if (block == 128)
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &blocks, rho ? mm_batch_kernel<S, 128, true> : mm_batch_kernel<S, 128, false>, 128, 0);
        else
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                &blocks, rho ? mm_batch_kernel<S, 256, true> : mm_batch_kernel<S, 256, false>, 256, 0);
    });
    return blocks;
}

int mm_launch_adjoint(const AdjointArgs& A, cudaStream_t st) {
    int launched = 0;
    with_media(A.a.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        if constexpr (M == kPerCell) {
            if (A.a.g.n > kReadOnlyBackwardCells) {
                mm_adjoint_kernel<M, true><<<blocks_for(A.a.g.n), kBlock, 0, st>>>(A);
                launched = 1;
                return;
            }
        }
        launch_after(mm_adjoint_kernel<M, false>, blocks_for(A.a.g.n), kBlock, 0, st, A);
        launched = 1;
    });
    return launched;
}

int mm_launch_adjoint_terminal(const AdjointArgs& A, int n_plane, cudaStream_t st) {
    with_media(A.a.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        launch_after(mm_adjoint_terminal_kernel<M>, blocks_for(n_plane), kBlock, 0, st, A, n_plane);
    });
    return 1;
}

int mm_fused2_occupancy(int storage, int media_mode) {
    int blocks = 0;
    with_pass_storage(storage, [&](auto sc) {
        with_media(media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, mm_fused2_kernel<S, M>, kFusedThreads, 0);
        });
    });
    return blocks;
}

int mm_launch_fused2(const StepArgs& aA, const StepArgs& aB, const FusedArgs& F, cudaStream_t st) {
    if (aA.storage == kF24) return 0;  // no 24-bit form of the passes
    const int grid = fused_grid(mm_fused2_occupancy(aA.storage, aA.media_mode));
    with_pass_storage(aA.storage, [&](auto sc) {
        with_media(aA.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            mm_fused2_kernel<S, M><<<grid, kFusedThreads, 0, st>>>(aA, aB, F);
        });
    });
    return 1;
}

template <int S, int M, bool kRecord = false>
bool mm_tile2_prepare() {
    static std::atomic<unsigned long long> done{0};
    return allow_shared(done, mm_tile2_kernel<S, M, kRecord>, MMTile<S>::kBytes);
}

int mm_tile2_occupancy(int storage, int media_mode) {
    int blocks = 0;
    with_pass_storage(storage, [&](auto sc) {
        with_media(media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            if (!mm_tile2_prepare<S, M>() ||
                cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, mm_tile2_kernel<S, M>, Tile::kCells,
                                                              MMTile<S>::kBytes) != cudaSuccess) {
                cudaGetLastError();
                blocks = 0;
            }
        });
    });
    return blocks;
}

int mm_launch_tile2(const StepArgs& aA, const StepArgs& aB, const TileArgs& T, cudaStream_t st) {
    if (aA.storage == kF24) return 0;  // no 24-bit form of the passes
    const dim3 grid(T.tiles_x * T.tiles_y, (aA.g.nz + T.chunk - 1) / T.chunk);
    int launched = 0;
    with_pass_storage(aA.storage, [&](auto sc) {
        with_media(aA.media_mode, [&](auto mc) {
            constexpr int S = decltype(sc)::value, M = decltype(mc)::value;
            if (!mm_tile2_prepare<S, M>()) return;  // the caller reads the error
            mm_tile2_kernel<S, M><<<grid, Tile::kCells, MMTile<S>::kBytes, st>>>(aA, aB, T);
            launched = 1;
        });
    });
    return launched;
}

int mm_launch_record_tile2(const StepArgs& aA, const StepArgs& aB, const TileArgs& T, cudaStream_t st) {
    if (aA.storage != kF32 || !aA.rec || !aB.rec) return 0;
    const dim3 grid(T.tiles_x * T.tiles_y, (aA.g.nz + T.chunk - 1) / T.chunk);
    int launched = 0;
    with_media(aA.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        if (!mm_tile2_prepare<kF32, M, true>()) return;  // the caller reads the error
        mm_tile2_kernel<kF32, M, true><<<grid, Tile::kCells, MMTile<kF32>::kBytes, st>>>(aA, aB, T);
        launched = 1;
    });
    return launched;
}

int mm_halo_dirs(int vz_sign, int* dirs) {
    int k = 0;
    for (int d = 0; d < 12; ++d)
        if (kMMV[d][2] == vz_sign) dirs[k++] = d;
    return k;
}

int mm_launch_record_step(const StepArgs& a, cudaStream_t st) {
    int launched = 0;
    const bool rho = a.rho_in != nullptr;
    with_media(a.media_mode, [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        if (rho) launch_after(mm_record_kernel<M, true>, blocks_for(a.g.n), kBlock, 0, st, a);
        else launch_after(mm_record_kernel<M, false>, blocks_for(a.g.n), kBlock, 0, st, a);
        launched = 1;
    });
    return launched;
}

}  // namespace lbm
