// The arithmetic of one HV cell update (arXiv 2309.08068 Section III), shared by every kernel that
// steps HV cells: directions, moments, collision, and the pulls and stores of the A/B buffers. The
// formulas are at the head of hv.cu.
#pragma once

#include "lbm_internal.cuh"

namespace lbm {
namespace {

// Axis (0, 1, 2) and sign of v_i, i = 1..6.
constexpr int kHVAxis[6] = {0, 1, 0, 1, 2, 2};
constexpr int kHVSign[6] = {1, 1, -1, -1, -1, 1};

// s * (a x X) for the unit axis a.
template <int A, int S>
__device__ __forceinline__ float3 axis_cross(float3 X) {
    float3 r;
    if constexpr (A == 0) r = make_float3(0.f, -X.z, X.y);
    else if constexpr (A == 1) r = make_float3(X.z, 0.f, -X.x);
    else r = make_float3(-X.y, X.x, 0.f);
    if constexpr (S < 0) r = make_float3(-r.x, -r.y, -r.z);
    return r;
}

// Offset of the cell x - v_i.
template <int I>
__device__ __forceinline__ int pull_index(const Neighbourhood& h) {
    constexpr int a = kHVAxis[I], s = kHVSign[I];
    return shifted<a == 0 ? -s : 0, a == 1 ? -s : 0, a == 2 ? -s : 0>(h);
}

// Offset of the cell x + v_i.
template <int I>
__device__ __forceinline__ int push_index(const Neighbourhood& h) {
    constexpr int a = kHVAxis[I], s = kHVSign[I];
    return shifted<a == 0 ? s : 0, a == 1 ? s : 0, a == 2 ? s : 0>(h);
}

// 24-bit storage: in each of the two arrays the 6 planes of halves, then the 6 planes of correction
// bytes.
template <int S>
__device__ __forceinline__ void hv_pull(const StepArgs& a, const Neighbourhood& h, float4 (&e)[6], float2 (&hy)[6]) {
    if constexpr (S == kF24) {
        const size_t n6 = 6 * (size_t)a.g.n;
        const uint2* ehi = static_cast<const uint2*>(a.fin);
        const unsigned* elo = reinterpret_cast<const unsigned*>(ehi + n6);
        const unsigned* hhi = static_cast<const unsigned*>(a.fin2);
        const unsigned short* hlo = reinterpret_cast<const unsigned short*>(hhi + n6);
        static_for<0, 6>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            const size_t idx = (size_t)i * a.g.n + pull_index<i>(h);
            e[i] = F24::load4(ehi, elo, idx, a.inv_scale);
            hy[i] = F24::load2(hhi, hlo, idx, a.inv_scale);
        });
    } else {
        const auto* ein = static_cast<const typename Pack4<S>::T*>(a.fin);
        const auto* hin = static_cast<const typename Pack2<S>::T*>(a.fin2);
        static_for<0, 6>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            const int src = pull_index<i>(h);
            e[i] = Pack4<S>::load(ein + (size_t)i * a.g.n + src, a.inv_scale);
            hy[i] = Pack2<S>::load(hin + (size_t)i * a.g.n + src, a.inv_scale);
        });
    }
}

template <int S>
__device__ __forceinline__ void hv_put(const StepArgs& a, int k, int i, float4 e, float2 hy) {
    if constexpr (S == kF24) {
        const size_t n6 = 6 * (size_t)a.g.n, idx = (size_t)k * a.g.n + i;
        uint2* __restrict__ ehi = static_cast<uint2*>(a.fout);
        unsigned* __restrict__ hhi = static_cast<unsigned*>(a.fout2);
        F24::store4(ehi, reinterpret_cast<unsigned*>(ehi + n6), idx, e, a.scale);
        F24::store2(hhi, reinterpret_cast<unsigned short*>(hhi + n6), idx, hy, a.scale);
    } else {
        auto* __restrict__ eout = static_cast<typename Pack4<S>::T*>(a.fout);
        auto* __restrict__ hout = static_cast<typename Pack2<S>::T*>(a.fout2);
        eout[(size_t)k * a.g.n + i] = Pack4<S>::pack(e, a.scale);
        hout[(size_t)k * a.g.n + i] = Pack2<S>::pack(hy, a.scale);
    }
}

struct HVFields {
    float3 D, B, E, H, J;
};

// kPacked: the six sums as three of register pairs, (x, y), (z, h_x) and (h_y, h_z) as they were loaded:
// 15 additions instead of 30, the same bits. For the kernels that issue bounds: the line kernel (1024
// cells 0.26 -> 0.22 us per step on GB300) and the tiled pass (128^3 with a medium per cell 59.8 -> 58.0
// us, 512 x 64 x 64 56.2 -> 55.4); the memory-bound single steps are not faster, 16-bit ones 0.7 % slower.
template <bool kPacked = false>
__device__ __forceinline__ HVFields hv_fields(const float4 (&e)[6], const float2 (&hy)[6], const MatCoef& mat,
                                              float3 jext) {
    HVFields F;
    // Pairwise sums ((1 + 2) + (3 + 4)) + (5 + 6) over the directions.
    float dx, dy, dz, bx, by, bz;
    if constexpr (kPacked) {
        float2 xy[6], zh[6];
        static_for<0, 6>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            xy[i] = make_float2(e[i].x, e[i].y);
            zh[i] = make_float2(e[i].z, e[i].w);
        });
        auto six = [](const float2 (&t)[6]) {
            return __fadd2_rn(__fadd2_rn(__fadd2_rn(t[0], t[1]), __fadd2_rn(t[2], t[3])), __fadd2_rn(t[4], t[5]));
        };
        const float2 s0 = six(xy), s1 = six(zh), s2 = six(hy);
        dx = s0.x, dy = s0.y, dz = s1.x, bx = s1.y, by = s2.x, bz = s2.y;
    } else {
        float tx[6], ty[6], tz[6], ux[6], uy[6], uz[6];
        static_for<0, 6>([&](auto ic) {
            constexpr int i = decltype(ic)::value;
            tx[i] = e[i].x;
            ty[i] = e[i].y;
            tz[i] = e[i].z;
            ux[i] = e[i].w;
            uy[i] = hy[i].x;
            uz[i] = hy[i].y;
        });
        dx = pairwise_sum<0, 4>(tx) + pairwise_sum<4, 6>(tx);
        dy = pairwise_sum<0, 4>(ty) + pairwise_sum<4, 6>(ty);
        dz = pairwise_sum<0, 4>(tz) + pairwise_sum<4, 6>(tz);
        bx = pairwise_sum<0, 4>(ux) + pairwise_sum<4, 6>(ux);
        by = pairwise_sum<0, 4>(uy) + pairwise_sum<4, 6>(uy);
        bz = pairwise_sum<0, 4>(uz) + pairwise_sum<4, 6>(uz);
    }
    const float eps = mat.c0.x, inv_eps = mat.c0.y, mu = mat.c0.z, inv_mu = mat.c0.w, sigma = mat.c1.x;
    F.D = make_float3(dx, dy, dz);
    F.B = make_float3(bx, by, bz);
    F.E = make_float3(div_rn(dx, eps, inv_eps), div_rn(dy, eps, inv_eps), div_rn(dz, eps, inv_eps));
    F.H = make_float3(div_rn(bx, mu, inv_mu), div_rn(by, mu, inv_mu), div_rn(bz, mu, inv_mu));
    F.J = make_float3(__fmaf_rn(sigma, F.E.x, jext.x), __fmaf_rn(sigma, F.E.y, jext.y),
                      __fmaf_rn(sigma, F.E.z, jext.z));
    return F;
}

constexpr float kInv3 = 1.0f / 3.0f;  // RN(1/3)
constexpr float kInv6 = 1.0f / 6.0f;  // RN(1/6)

__device__ __forceinline__ float3 sixth(float3 v) {
    return make_float3(div_rn(v.x, 6.f, kInv6), div_rn(v.y, 6.f, kInv6), div_rn(v.z, 6.f, kInv6));
}
// D / 6 with D = eps E.
__device__ __forceinline__ float3 hv_sixth_of_d(float3 E, const MatCoef& mat) {
    const float eps = mat.c0.x;
    return sixth(make_float3(eps * E.x, eps * E.y, eps * E.z));
}
// H = B / mu.
__device__ __forceinline__ float3 hv_h(float3 B, const MatCoef& mat) {
    const float mu = mat.c0.z, inv_mu = mat.c0.w;
    return make_float3(div_rn(B.x, mu, inv_mu), div_rn(B.y, mu, inv_mu), div_rn(B.z, mu, inv_mu));
}

// Where a step reads its populations and writes its results: the context's A/B buffers.
struct HVBuffers : NoStash {
    template <int S>
    __device__ void pull(const StepArgs& a, const Neighbourhood& h, float4 (&e)[6], float2 (&hy)[6]) const {
        hv_pull<S>(a, h, e, hy);
    }
    template <int S>
    __device__ void put(const StepArgs& a, int k, int i, float4 e, float2 hy) const {
        hv_put<S>(a, k, i, e, hy);
    }
};

// The collision of a cell with moments F: put(k, e', (h_y', h_z')) receives the post-collision values
// of direction k = 0 .. 5 in turn, e' with h_x' as its fourth component. half(k, hx, hy, hz) gives
// the h components of direction k (a kernel may have parked them in shared memory).
template <class HalfOf, class Put>
__device__ __forceinline__ void hv_collide(const HVFields& F, const float4 (&e)[6], const float2 (&hy)[6],
                                           HalfOf&& half, Put&& put) {
    // Isotropic share of 2 e^eq and 2 h^eq: D / 3 and B / 3, correctly rounded (a multiplication by
    // RN(1/3) would bias every step by the same relative 3e-8 and drift D and B on long runs).
    const float3 q = make_float3(div_rn(F.D.x, 3.f, kInv3), div_rn(F.D.y, 3.f, kInv3), div_rn(F.D.z, 3.f, kInv3));
    const float3 p = make_float3(div_rn(F.B.x, 3.f, kInv3), div_rn(F.B.y, 3.f, kInv3), div_rn(F.B.z, 3.f, kInv3));
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        constexpr int A = kHVAxis[k], G = kHVSign[k];
        const float3 vH = axis_cross<A, G>(F.H);
        const float3 vE = axis_cross<A, G>(F.E);
        float3 eo = make_float3(q.x - vH.x - e[k].x, q.y - vH.y - e[k].y, q.z - vH.z - e[k].z);
        // eq. SourceTermHV: T_i = -(J . v_i) v_i / 2 = -(J_A / 2) along axis A.
        if constexpr (A == 0) eo.x -= 0.5f * F.J.x;
        else if constexpr (A == 1) eo.y -= 0.5f * F.J.y;
        else eo.z -= 0.5f * F.J.z;
        float hx = e[k].w, hyx = hy[k].x, hyy = hy[k].y;
        half(ic, hx, hyx, hyy);
        float3 ho = make_float3(p.x + vE.x - hx, p.y + vE.y - hyx, p.z + vE.z - hyy);
        put(ic, make_float4(eo.x, eo.y, eo.z, ho.x), make_float2(ho.y, ho.z));
    });
}

// What an imposed cell holds after its collision (Appendix B "impose fields"):
// f' = f_eq(E_imp, B_imp, J = 0), by direction as in hv_collide.
template <class Put>
__device__ __forceinline__ void hv_impose(const MatCoef& mat, const CellSource& cs, Put&& put) {
    const float3 H = hv_h(cs.B, mat), d6 = hv_sixth_of_d(cs.E, mat), b6 = sixth(cs.B);
    static_for<0, 6>([&](auto ic) {
        constexpr int k = decltype(ic)::value;
        const float3 cH = axis_cross<kHVAxis[k], kHVSign[k]>(H), cE = axis_cross<kHVAxis[k], kHVSign[k]>(cs.E);
        put(ic, make_float4(d6.x - 0.5f * cH.x, d6.y - 0.5f * cH.y, d6.z - 0.5f * cH.z, b6.x + 0.5f * cE.x),
            make_float2(b6.y + 0.5f * cE.y, b6.z + 0.5f * cE.z));
    });
}

// Update of cell i with the sources cs, known beforehand.
template <int S, int M>
__device__ __forceinline__ void hv_update_sourced(const StepArgs& a, int i, const CellSource& cs) {
    float4 e[6];
    float2 hy[6];
    hv_pull<S>(a, neighbourhood(a.g, i), e, hy);
    const MatCoef mat = load_coef<kModelHV, M>(a.media, i, a.eps0, a.mu0);
    const HVFields F = hv_fields(e, hy, mat, cs.J);
    auto put = [&](auto kc, float4 eo, float2 ho) { hv_put<S>(a, decltype(kc)::value, i, eo, ho); };
    if (cs.imposed) hv_impose(mat, cs, put);
    else hv_collide(F, e, hy, [](auto, float&, float&, float&) {}, put);
}

// Update of cell i; m is its index in the special-cell list when kSpecial.
template <int S, int M, bool kSpecial, bool kRecord = false, class IO = HVBuffers>
__device__ __forceinline__ void hv_update(const StepArgs& a, int i, int m, const IO& io = IO{}) {
    const Neighbourhood h = neighbourhood(a.g, i);
    float4 e[6];
    float2 hy[6];
    io.template pull<S>(a, h, e, hy);
    if constexpr (IO::kStash)  // the h components wait in shared memory until the collision
        static_for<0, 6>([&](auto ic) {
            constexpr int k = decltype(ic)::value;
            io.stash_put(k, hy[k].x, hy[k].y);
            io.stash_put(6 + k, e[k].w, 0.f);  // h_x, which shares the float4 with e
        });
    const MatCoef mat = load_coef<kModelHV, M>(a.media, i, a.eps0, a.mu0);
    CellSource cs;
    float3 jext = make_float3(0.f, 0.f, 0.f);
    if constexpr (kSpecial) {
        cs = cell_source(a.sv, a.sc, m);
        jext = cs.J;
    }
    const HVFields F = hv_fields(e, hy, mat, jext);
    auto half = [&](auto kc, float& hx, float& hyx, float& hyy) {
        if constexpr (IO::kStash) {
            float unused;
            io.stash_get(decltype(kc)::value, hyx, hyy);
            io.stash_get(6 + decltype(kc)::value, hx, unused);
        }
    };
    auto put = [&](auto kc, float4 eo, float2 ho) { io.template put<S>(a, decltype(kc)::value, i, eo, ho); };
    bool imposed = false;
    if constexpr (kSpecial) imposed = cs.imposed;
    if (imposed) hv_impose(mat, cs, put);
    else hv_collide(F, e, hy, half, put);
    if constexpr (kRecord) {  // what the adjoint of this step needs: E
        const int n = a.g.n;
        a.rec[i] = F.E.x;
        a.rec[n + i] = F.E.y;
        a.rec[2 * n + i] = F.E.z;
    }
}

}  // namespace
}  // namespace lbm
