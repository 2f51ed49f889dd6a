// Many time steps per launch on line lattices (nx = ny = 1), both models.
//
// The paper's one-dimensional tests (arXiv 2309.08068 Sections IV-A, IV-B, IV-D) run some hundred to
// some thousand cells for about as many steps. One launch per step leaves the GPU idle: a step of
// such a lattice is a launch gap and one chain of loads, update and stores (4.1 us per step for MM
// on 1024 cells, 6.2 us with an imposed source cell), on a handful of blocks. Here a
// block takes `core` cells and a halo of `steps` cells on either side, one thread per cell, and
// runs `steps` steps without leaving the SM: the populations stay in registers, and only those that
// move along the line (8 of MM's 12 velocities, 2 of HV's 6) pass between neighbouring threads through
// shared memory, double-buffered so that a step takes one barrier. With nx = ny = 1 the other
// velocities lead back to the cell itself. A halo cell's value is wrong once the halo's end has
// reached it, one cell per step, so the core is right after `steps` steps; blocks never wait for one
// another. What bounds it is the chain of one step (shared-memory read, moments, collision,
// shared-memory write, barrier), which one warp per scheduler runs at its own latency: 128 threads.
// Measured on GB300 (FP32, us per step; one launch per step in brackets, as launched before kernels were set
// up early): MM 0.36 (4.1) at 1024 cells, 0.52 (6.2) at 4000 with an imposed cell, 0.40 (4.1) at 8192,
// 1.04 (4.1) at 30000; HV 0.20 (4.1), 0.29 (6.2), 0.22 (4.1), 0.55 (4.1). A million cells: MM 22 (59), HV
// 16 (46). 96 threads are 5 % faster on 500 to 1024 MM cells and 37 % slower at 8192; 64 and 160 slower.
// The medium and the sources of a cell do not depend on the launch before, so they are looked up before it
// is waited for; the launch after is let in before the last step, not at once: its blocks, set up while
// all of this launch's still ran, came to lie two to an SM (4000 HV cells, 3000 steps: 1034 us let in at
// once, 836 late, 797 with the early look-ups).
//
// The arithmetic is the single step's, and what a step hands to the next is rounded to the storage
// format at every step, so a launch equals `steps` single steps bit for bit.
#include "hv_core.cuh"
#include "mm_core.cuh"

namespace lbm {
namespace {

// v as it reads back after being stored (identity for FP32).
template <int S>
__device__ __forceinline__ float f24_round(float v, float scale, float inv) {
    const unsigned s = F24::split(v, scale);  // h in bits 15..0, q in bits 23..16
    return F24::join((s << 16) | ((s >> 8) & 0xff00u), inv);
}
template <int S>
__device__ __forceinline__ float4 stored4(float4 v, float scale, float inv) {
    if constexpr (S == kF24)
        return make_float4(f24_round<S>(v.x, scale, inv), f24_round<S>(v.y, scale, inv),
                           f24_round<S>(v.z, scale, inv), f24_round<S>(v.w, scale, inv));
    else
        return Pack4<S>::unpack(Pack4<S>::pack(v, scale), inv);
}
template <int S>
__device__ __forceinline__ float2 stored2(float2 v, float scale, float inv) {
    if constexpr (S == kF24) return make_float2(f24_round<S>(v.x, scale, inv), f24_round<S>(v.y, scale, inv));
    else return Pack2<S>::unpack(Pack2<S>::pack(v, scale), inv);
}

// Coefficients of cell i, the media mode taken at run time (once per launch).
template <int Model>
__device__ __forceinline__ MatCoef line_coef(const StepArgs& a, int i) {
    if (a.media_mode == kTable) return load_coef<Model, kTable>(a.media, i, a.eps0, a.mu0);
    if (a.media_mode == kPerCell) return load_coef<Model, kPerCell>(a.media, i, a.eps0, a.mu0);
    return a.media.uniform;
}

// The sources of this thread's cell, looked up once per launch. The first current entry and the first
// imposing slot, in nearly every case the only ones, wait in registers: a block with a source cell
// is the longest of its launch (MM, 4000 cells, an imposed cell: 0.62 us per step when every step
// read them from memory).
struct LineSource {
    int begin, end;  // current entries of the cell (none: begin == end)
    int src;         // source slot and weights of the first entry
    float3 w;
    uint32_t mask;   // imposing slots beyond the first one
    int slot;        // first imposing slot, and its vectors
    float3 E0, B0;
    bool imposed;

    __device__ void find(const SourceView& sv, const SourceScalars& sc, int cell) {
        begin = end = src = slot = 0;
        mask = 0;
        w = E0 = B0 = make_float3(0.f, 0.f, 0.f);
        imposed = false;
        int lo = 0, hi = sv.n_special;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (sv.cell[mid] < cell) lo = mid + 1;
            else hi = mid;
        }
        if (lo >= sv.n_special || sv.cell[lo] != cell) return;
        const SpecialCell& first = sv.first[lo];
        begin = first.begin;
        end = first.end;
        if (end > begin) {
            src = first.src;
            w = make_float3(first.w[0], first.w[1], first.w[2]);
        }
        mask = first.impose_mask;
        imposed = mask != 0u;
        if (imposed) {
            slot = __ffs(mask) - 1;
            mask &= mask - 1;
            E0 = make_float3(sc.E0[slot][0], sc.E0[slot][1], sc.E0[slot][2]);
            B0 = make_float3(sc.B0[slot][0], sc.B0[slot][1], sc.B0[slot][2]);
        }
    }

    // J_ext with the step's source values s[]: cell_source's sum, in its order; zero without entries
    // (whatever s holds).
    __device__ __forceinline__ float3 current(const SourceView& sv, const float* s) const {
        const float s0 = s[src];
        float3 J = make_float3(__fmaf_rn(w.x, s0, 0.f), __fmaf_rn(w.y, s0, 0.f), __fmaf_rn(w.z, s0, 0.f));
        for (int k = begin + 1; k < end; ++k) {
            const float sk = s[sv.entry_src[k]];
            J.x = __fmaf_rn(sv.entry_w[3 * k + 0], sk, J.x);
            J.y = __fmaf_rn(sv.entry_w[3 * k + 1], sk, J.y);
            J.z = __fmaf_rn(sv.entry_w[3 * k + 2], sk, J.z);
        }
        if (end <= begin) J = make_float3(0.f, 0.f, 0.f);
        return J;
    }

    // E and B imposed at the step, likewise.
    __device__ __forceinline__ void fields(const SourceScalars& sc, const float* s, CellSource& cs) const {
        const float s0 = s[slot];
        cs.E = make_float3(__fmaf_rn(E0.x, s0, 0.f), __fmaf_rn(E0.y, s0, 0.f), __fmaf_rn(E0.z, s0, 0.f));
        cs.B = make_float3(__fmaf_rn(B0.x, s0, 0.f), __fmaf_rn(B0.y, s0, 0.f), __fmaf_rn(B0.z, s0, 0.f));
        for (uint32_t left = mask; left; left &= left - 1) {
            const int k = __ffs(left) - 1;
            const float sk = s[k];
            cs.E.x = __fmaf_rn(sc.E0[k][0], sk, cs.E.x);
            cs.E.y = __fmaf_rn(sc.E0[k][1], sk, cs.E.y);
            cs.E.z = __fmaf_rn(sc.E0[k][2], sk, cs.E.z);
            cs.B.x = __fmaf_rn(sc.B0[k][0], sk, cs.B.x);
            cs.B.y = __fmaf_rn(sc.B0[k][1], sk, cs.B.y);
            cs.B.z = __fmaf_rn(sc.B0[k][2], sk, cs.B.z);
        }
    }
};

// This thread's cell, and whether it lies in the block's core.
struct LineCell {
    int z;
    bool core;
};
__device__ __forceinline__ LineCell line_cell(const LineArgs& L) {
    const int n = L.a.g.nz, at = (int)blockIdx.x * L.core, t = (int)threadIdx.x - L.steps;
    LineCell c;
    c.core = t >= 0 && t < L.core && at + t < n;
    int z = (at + t) % n;
    c.z = z < 0 ? z + n : z;
    return c;
}

// Rank of MM direction d among those that move along the line (v_z != 0): d - 4.
constexpr int kMMLineDirs = 8;

template <int S>
__global__ void __launch_bounds__(kLineThreads) mm_line_kernel(const __grid_constant__ LineArgs L) {
    __shared__ float4 s_move[2][kMMLineDirs][kLineThreads];
    const StepArgs& a = L.a;
    const int tid = threadIdx.x;
    const LineCell c = line_cell(L);
    const MatCoef mat = line_coef<kModelMM>(a, c.z);
    LineSource ls;
    ls.find(a.sv, a.sc, c.z);
    const bool currents = __any_sync(0xffffffffu, ls.end > ls.begin);  // the same code for the whole warp
    float4 f[12];
    wait_predecessor();
    mm_pull<S>(a, neighbourhood(a.g, c.z), f);
    // One step from f: in-plane directions lead back to the cell itself, the others to `move`; the
    // last step of the launch goes to memory.
    auto step = [&](int j, auto&& put) {
        auto half = [](auto, float&, float&) {};
        const float* s = L.s + j * L.n_src;
        float3 J = make_float3(0.f, 0.f, 0.f);
        if (currents) J = ls.current(a.sv, s);
        mm_collide(mm_fields<false>(f, 0.f, mat, J), f, half, put);
        if (ls.imposed) {
            CellSource cs;
            ls.fields(a.sc, s, cs);
            mm_impose(mat, cs, put);
        }
    };
    for (int j = 0; j + 1 < L.steps; ++j) {
        float4(*move)[kLineThreads] = s_move[j & 1];
        step(j, [&](auto dc, float4 o) {
            constexpr int d = decltype(dc)::value;
            const float4 v = stored4<S>(o, a.scale, a.inv_scale);
            if constexpr (kMMV[d][2] == 0) f[d] = v;
            else move[d - 4][tid] = v;
        });
        __syncthreads();
        const int below = max(tid - 1, 0), above = min(tid + 1, kLineThreads - 1);
        static_for<4, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            constexpr bool up = kMMV[d][2] > 0;
            f[d] = move[d - 4][up ? below : above];
        });
    }
    let_successor();
    step(L.steps - 1, [&](auto dc, float4 o) {
        if (c.core) mm_put<S>(a, decltype(dc)::value, c.z, o);
    });
}

// Slots of the two HV directions that move along the line: k = 4 (-z) and 5 (+z).
template <int S>
__global__ void __launch_bounds__(kLineThreads) hv_line_kernel(const __grid_constant__ LineArgs L) {
    __shared__ float4 s_e[2][2][kLineThreads];
    __shared__ float2 s_h[2][2][kLineThreads];
    const StepArgs& a = L.a;
    const int tid = threadIdx.x;
    const LineCell c = line_cell(L);
    const MatCoef mat = line_coef<kModelHV>(a, c.z);
    LineSource ls;
    ls.find(a.sv, a.sc, c.z);
    const bool currents = __any_sync(0xffffffffu, ls.end > ls.begin);
    float4 e[6];
    float2 hy[6];
    wait_predecessor();
    hv_pull<S>(a, neighbourhood(a.g, c.z), e, hy);
    auto step = [&](int j, auto&& put) {  // as in mm_line_kernel
        auto half = [](auto, float&, float&, float&) {};
        const float* s = L.s + j * L.n_src;
        float3 J = make_float3(0.f, 0.f, 0.f);
        if (currents) J = ls.current(a.sv, s);
        hv_collide(hv_fields<true>(e, hy, mat, J), e, hy, half, put);
        if (ls.imposed) {
            CellSource cs;
            ls.fields(a.sc, s, cs);
            hv_impose(mat, cs, put);
        }
    };
    for (int j = 0; j + 1 < L.steps; ++j) {
        float4(*me)[kLineThreads] = s_e[j & 1];
        float2(*mh)[kLineThreads] = s_h[j & 1];
        step(j, [&](auto kc, float4 eo, float2 ho) {
            constexpr int k = decltype(kc)::value;
            const float4 ve = stored4<S>(eo, a.scale, a.inv_scale);
            const float2 vh = stored2<S>(ho, a.scale, a.inv_scale);
            if constexpr (k < 4) {
                e[k] = ve;
                hy[k] = vh;
            } else {
                me[k - 4][tid] = ve;
                mh[k - 4][tid] = vh;
            }
        });
        __syncthreads();
        const int below = max(tid - 1, 0), above = min(tid + 1, kLineThreads - 1);
        e[4] = me[0][above];
        hy[4] = mh[0][above];
        e[5] = me[1][below];
        hy[5] = mh[1][below];
    }
    let_successor();
    step(L.steps - 1, [&](auto kc, float4 eo, float2 ho) {
        if (c.core) hv_put<S>(a, decltype(kc)::value, c.z, eo, ho);
    });
}

}  // namespace

int launch_line(bool mm, const LineArgs& L, cudaStream_t st) {
    const int blocks = (L.a.g.nz + L.core - 1) / L.core;
    with_storage(L.a.storage, [&](auto sc) {
        constexpr int S = decltype(sc)::value;
        if (mm) launch_after(mm_line_kernel<S>, blocks, kLineThreads, 0, st, L);
        else launch_after(hv_line_kernel<S>, blocks, kLineThreads, 0, st, L);
    });
    return 1;
}

}  // namespace lbm
