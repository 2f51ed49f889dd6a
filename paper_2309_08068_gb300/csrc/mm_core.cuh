// The arithmetic of one MM cell update (arXiv 2309.08068 Section II), shared by every kernel that
// steps MM cells: direction tables, moments, collision, and the pulls and stores of the A/B buffers.
// The tables' derivation is at the head of mm.cu. Every inexact product that meets a sum is an
// explicit fused multiply-add, so that all of them give the same bits.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {
namespace {

constexpr int kMMV[12][3] = {{1, 1, 0},  {-1, 1, 0},  {-1, -1, 0}, {1, -1, 0},
                             {1, 0, 1},  {-1, 0, 1},  {-1, 0, -1}, {1, 0, -1},
                             {0, 1, 1},  {0, -1, 1},  {0, -1, -1}, {0, 1, -1}};
constexpr int kMMEh[12][3] = {{1, -1, 0}, {1, 1, 0},  {-1, 1, 0}, {-1, -1, 0},
                              {1, 0, -1}, {1, 0, 1},  {-1, 0, 1}, {-1, 0, -1},
                              {0, 1, -1}, {0, 1, 1},  {0, -1, 1}, {0, -1, -1}};
constexpr int kMMB[12][3] = {{0, 0, -1}, {0, 0, -1}, {0, 0, -1}, {0, 0, -1},
                             {0, 1, 0},  {0, 1, 0},  {0, 1, 0},  {0, 1, 0},
                             {-1, 0, 0}, {-1, 0, 0}, {-1, 0, 0}, {-1, 0, 0}};

// Dot product of a compile-time {-1,0,1} vector row with (x, y, z).
template <int A, int B, int C>
__device__ __forceinline__ float sdot(float x, float y, float z) {
    float s = 0.f;
    acc<A>(s, x);
    acc<B>(s, y);
    acc<C>(s, z);
    return s;
}

struct MMFields {
    float3 X;    // D' - mu0 J_ext / 4 (so that Dpp = X g)
    float3 Dpp;  // eps_r E = D (physical displacement, eps0 = 1)
    float3 E;
    float3 B;
    float3 J;
    float rho;
    float inv4mu;  // 1 / (4 mu_r)
};

// Moments of the 48 moving populations (eq. MacroscopicFieldsMiller), then E and J with ohmic
// conductivity and an external current (eqs. MacroscopicEMiller, MacorscopicCurrentMiller):
//   eps_r E = (D' - mu0 J_ext / 4) / (1 + mu0 sigma / (4 eps_r)),  J = sigma E + J_ext,  mu0 = 2.
// Position of direction d among the directions whose row of table T has a non-zero component a.
template <const int (&T)[12][3]>
constexpr int rank_in_column(int d, int a) {
    int r = 0;
    for (int k = 0; k < d; ++k) r += T[k][a] != 0;
    return r;
}

// Signed terms of one moment component, sum_d T[d][a] * x_d, summed pairwise in direction order.
// Each component of D' has 8 terms (2 e_{i0} has two non-zero entries), each component of B has 4.
template <const int (&T)[12][3], int A, int N>
__device__ __forceinline__ float moment_component(const float (&x)[12]) {
    float t[N];
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        if constexpr (T[d][A] != 0) {
            constexpr int r = rank_in_column<T>(d, A);
            if constexpr (T[d][A] > 0) t[r] = x[d];
            else t[r] = -x[d];
        }
    });
    return pairwise_sum<0, N>(t);
}

// eps_r E = Dpp = X g and E = Dpp / eps_r, each rounded once (__fmul_rn: never fused into a later
// sum), so that the backward step can recompute E from the recorded X and get the same bits.
__device__ __forceinline__ float3 mm_dpp(float3 X, float g) {
    return make_float3(__fmul_rn(X.x, g), __fmul_rn(X.y, g), __fmul_rn(X.z, g));
}
__device__ __forceinline__ float3 mm_e_of_dpp(float3 Dpp, float er, float inv_er) {
    return make_float3(div_rn(Dpp.x, er, inv_er), div_rn(Dpp.y, er, inv_er), div_rn(Dpp.z, er, inv_er));
}

template <bool kRho>
__device__ __forceinline__ MMFields mm_fields(const float4 (&f)[12], float rest0, const MatCoef& mat, float3 jext) {
    float de[12], db[12];
    float rho = rest0;
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        de[d] = f[d].x - f[d].y;
        db[d] = f[d].z - f[d].w;
        if constexpr (kRho) rho += f[d].x + f[d].y;
    });
    const float dx = moment_component<kMMEh, 0, 8>(de), dy = moment_component<kMMEh, 1, 8>(de),
                dz = moment_component<kMMEh, 2, 8>(de);
    const float bx = moment_component<kMMB, 0, 4>(db), by = moment_component<kMMB, 1, 4>(db),
                bz = moment_component<kMMB, 2, 4>(db);
    MMFields o;
    const float g = mat.c0.z;  // 1 / (1 + mu0 sigma / (4 eps_r))
    const float er = mat.c0.x, inv_er = mat.c0.y, sigma = mat.c1.x;
    o.X = make_float3(0.5f * dx - 0.5f * jext.x, 0.5f * dy - 0.5f * jext.y, 0.5f * dz - 0.5f * jext.z);
    o.Dpp = mm_dpp(o.X, g);
    o.E = mm_e_of_dpp(o.Dpp, er, inv_er);
    o.B = make_float3(bx, by, bz);
    // Explicit fused multiply-adds wherever a product is inexact, so that the result does not
    // depend on the compiler's contraction choices (the batched and single-lattice kernels inline
    // this code in different contexts and must agree bit for bit).
    o.J.x = __fmaf_rn(sigma, o.E.x, jext.x);
    o.J.y = __fmaf_rn(sigma, o.E.y, jext.y);
    o.J.z = __fmaf_rn(sigma, o.E.z, jext.z);
    o.rho = rho;
    o.inv4mu = mat.c0.w;
    return o;
}

// Pull the 12 groups of cell i from the previous step's buffer: direction d from cell i - v_d.
// 24-bit storage: the 12 planes of halves (8 B per group and cell), then the 12 planes of correction
// bytes (4 B per group and cell).
// kReadOnly: see read().
template <int S, bool kReadOnly = false>
__device__ __forceinline__ void mm_pull(const StepArgs& a, const Neighbourhood& h, float4 (&f)[12]) {
    if constexpr (S == kF24) {
        const uint2* hi = static_cast<const uint2*>(a.fin);
        const unsigned* lo = reinterpret_cast<const unsigned*>(hi + 12 * (size_t)a.g.n);
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            const int src = shifted<-kMMV[d][0], -kMMV[d][1], -kMMV[d][2]>(h);
            f[d] = F24::load4(hi, lo, (size_t)d * a.g.n + src, a.inv_scale);
        });
    } else {
        const auto* fin = static_cast<const typename Pack4<S>::T*>(a.fin);
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            const int src = shifted<-kMMV[d][0], -kMMV[d][1], -kMMV[d][2]>(h);
            f[d] = Pack4<S>::template load<kReadOnly>(fin + (size_t)d * a.g.n + src, a.inv_scale);
        });
    }
}

// Prefetch into L2 what the update of cell i will load: the populations mm_pull reads and the medium.
template <int S, int M>
__device__ __forceinline__ void mm_prefetch(const StepArgs& a, int i) {
    prefetch_media<M>(a.media, i);
    const auto* fin = static_cast<const typename Pack4<S>::T*>(a.fin);
    const Neighbourhood h = neighbourhood(a.g, i);
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        prefetch_l2(fin + (size_t)d * a.g.n + shifted<-kMMV[d][0], -kMMV[d][1], -kMMV[d][2]>(h));
    });
}

template <int S>
__device__ __forceinline__ void mm_put(const StepArgs& a, int d, int i, float4 v) {
    if constexpr (S == kF24) {
        uint2* __restrict__ hi = static_cast<uint2*>(a.fout);
        unsigned* __restrict__ lo = reinterpret_cast<unsigned*>(hi + 12 * (size_t)a.g.n);
        F24::store4(hi, lo, (size_t)d * a.g.n + i, v, a.scale);
    } else {
        auto* __restrict__ fout = static_cast<typename Pack4<S>::T*>(a.fout);
        fout[(size_t)d * a.g.n + i] = Pack4<S>::pack(v, a.scale);
    }
}

// Where a step reads its populations and writes its results: the context's A/B buffers.
struct MMBuffers : NoStash {
    template <int S>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&f)[12]) const {
        mm_pull<S>(a, h, f);
    }
    template <int S>
    __device__ void put(const StepArgs& a, int d, int i, float4 v) const {
        mm_put<S>(a, d, i, v);
    }
};

// The collision of a cell with moments F: put(d, o) receives the post-collision values of direction
// d = 0 .. 11 in turn. zw(d, z, w) gives the f^(1) halves of direction d (a kernel may have parked
// them in shared memory).
template <class HalfOf, class Put>
__device__ __forceinline__ void mm_collide(const MMFields& F, const float4 (&f)[12], HalfOf&& zw, Put&& put) {
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        constexpr int v0 = kMMV[d][0], v1 = kMMV[d][1], v2 = kMMV[d][2];
        constexpr int e0 = kMMEh[d][0], e1 = kMMEh[d][1], e2 = kMMEh[d][2];
        constexpr int b0 = kMMB[d][0], b1 = kMMB[d][1], b2 = kMMB[d][2];
        const float two_s = 0.125f * sdot<v0, v1, v2>(F.J.x, F.J.y, F.J.z);
        const float bb = sdot<b0, b1, b2>(F.B.x, F.B.y, F.B.z);
        const float two_alpha = __fmaf_rn(bb, F.inv4mu, 0.25f * sdot<e0, e1, e2>(F.Dpp.x, F.Dpp.y, F.Dpp.z));
        const float two_beta = __fmaf_rn(0.25f, bb, __fmul_rn(0.25f, sdot<e0, e1, e2>(F.E.x, F.E.y, F.E.z)));
        float4 o;
        o.x = two_s + two_alpha - f[d].x;
        o.y = two_s - two_alpha - f[d].y;
        float fz = f[d].z, fw = f[d].w;
        zw(dc, fz, fw);
        o.z = two_s + two_beta - fz;
        o.w = two_s - two_beta - fw;
        put(dc, o);
    });
}

// What an imposed cell holds after its collision (Appendix B "impose fields"):
// f' = f_eq(E_imp, B_imp, J = 0), by direction as in mm_collide.
template <class Put>
__device__ __forceinline__ void mm_impose(const MatCoef& mat, const CellSource& cs, Put&& put) {
    static_for<0, 12>([&](auto dc) {
        constexpr int d = decltype(dc)::value;
        const float bi = sdot<kMMB[d][0], kMMB[d][1], kMMB[d][2]>(cs.B.x, cs.B.y, cs.B.z);
        const float ee = sdot<kMMEh[d][0], kMMEh[d][1], kMMEh[d][2]>(cs.E.x, cs.E.y, cs.E.z);
        const float alpha = __fmaf_rn(0.5f * bi, mat.c0.w, 0.125f * __fmul_rn(mat.c0.x, ee));
        const float beta = 0.125f * ee + 0.125f * bi;
        put(dc, make_float4(alpha, -alpha, beta, -beta));
    });
}

// Update of cell i with the sources cs, known beforehand.
template <int S, int M>
__device__ __forceinline__ void mm_update_sourced(const StepArgs& a, int i, const CellSource& cs) {
    float4 f[12];
    mm_pull<S>(a, neighbourhood(a.g, i), f);
    const MatCoef mat = load_coef<kModelMM, M>(a.media, i, a.eps0, a.mu0);
    const MMFields F = mm_fields<false>(f, 0.f, mat, cs.J);
    auto put = [&](auto dc, float4 o) { mm_put<S>(a, decltype(dc)::value, i, o); };
    if (cs.imposed) mm_impose(mat, cs, put);
    else mm_collide(F, f, [](auto, float&, float&) {}, put);
}

// Update of cell i; m is its index in the special-cell list when kSpecial.
template <int S, int M, bool kSpecial, bool kRho, bool kRecord = false, class IO = MMBuffers>
__device__ __forceinline__ void mm_update(const StepArgs& a, int i, int m, const IO& io = IO{}) {
    const Neighbourhood h = neighbourhood(a.g, i);
    float4 f[12];
    io.template pull<S>(a, h, f);
    if constexpr (IO::kStash)  // the f^(1) halves wait in shared memory until the collision
        static_for<0, 12>([&](auto dc) {
            constexpr int d = decltype(dc)::value;
            io.stash_put(d, f[d].z, f[d].w);
        });
    const MatCoef mat = load_coef<kModelMM, M>(a.media, i, a.eps0, a.mu0);
    float rest0 = 0.f;
    if constexpr (kRho) rest0 = a.rho_in[i];
    CellSource cs;
    float3 jext = make_float3(0.f, 0.f, 0.f);
    if constexpr (kSpecial) {
        cs = cell_source(a.sv, a.sc, m);
        jext = cs.J;
    }
    const MMFields F = mm_fields<kRho>(f, rest0, mat, jext);
    auto half = [&](auto dc, float& fz, float& fw) {
        if constexpr (IO::kStash) io.stash_get(decltype(dc)::value, fz, fw);
    };
    auto put = [&](auto dc, float4 o) { io.template put<S>(a, decltype(dc)::value, i, o); };
    bool imposed = false;
    if constexpr (kSpecial) imposed = cs.imposed;
    if (imposed) mm_impose(mat, cs, put);
    else mm_collide(F, f, half, put);
    if constexpr (kRho) a.rho_out[i] = 2.f * F.rho - rest0;  // f_0^(0)eq = rho_c; stays in place
    if constexpr (kRecord) {  // what the adjoint of this step needs: X (E follows from it)
        if (!io.keeps_record()) return;
        const int n = a.g.n;
        a.rec[i] = F.X.x;
        a.rec[n + i] = F.X.y;
        a.rec[2 * n + i] = F.X.z;
    }
}

}  // namespace
}  // namespace lbm
