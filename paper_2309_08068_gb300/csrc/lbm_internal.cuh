// Internal declarations shared by the kernels and the C-ABI host code of liblbm.so.
//
// Data layout in HBM (pull scheme, two buffers A/B swapped every step). Each buffer holds the
// post-collision populations of one step at the cell that computed them; the next step pulls
// direction d from cell x - v_d.
//   MM: 12 direction groups; group d = p*4 + (i-1) is one float4 per cell:
//       (f^(0)_{d,j=0}, f^(0)_{d,j=1}, f^(1)_{d,j=0}, f^(1)_{d,j=1}), array [12][n].
//       Optional rest population f_0^(0) as float[n] (double-buffered) and f_0^(1) as float[n].
//   HV: 6 directions; direction i is a float4 (e_x, e_y, e_z, h_x) in array [6][n] and a float2
//       (h_y, h_z) in a second array [6][n].
// All 16-byte groups are 16-byte aligned whatever the neighbour shift, so every pull is one
// vector load per group.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <type_traits>
#include <utility>

namespace lbm {

constexpr int kMaxSources = 16;
constexpr int kBlock = 256;

enum MediaMode { kUniform = 0, kTable = 1, kPerCell = 2 };

// Population storage. Arithmetic is FP32 in every case; 16- and 24-bit storage convert at the pull
// and the store. A stored value is f * scale (scale a power of two, so the scaling itself is exact).
// kF24: an FP16 value h plus an 8-bit correction in units of ulp(h) / 256 (see F24 below).
enum StorageKind { kF32 = 0, kBF16 = 1, kF16 = 2, kF24 = 3 };

// Lattice shape. Cell coordinates come from the linear index by multiplication with host-computed
// magic numbers (Granlund and Montgomery, "Division by invariant integers using multiplication"):
// floor(i / d) = (i * M) >> (32 + k) with k = ceil(log2 d), M = ceil(2^(32+k) / d), exact for every
// i < 2^31.
struct Geometry {
    int nx, ny, nz;
    int n;  // nx * ny * nz, < 2^31
    unsigned long long mx, mxy;  // magic multipliers for division by nx and by nx * ny
    int kx, kxy;
};

// Per-material coefficients, computed on the host in double precision and rounded once (reciprocals
// as RN(1/d) of the stored float d, so that div_rn below is exact).
//   MM: c0 = (eps_r, 1/eps_r, g = 1/(1 + mu0 sigma/(4 eps_r)), 1/(4 mu_r)),  c1 = (sigma, mu_r, 0, 0)
//   HV: c0 = (eps, 1/eps, mu, 1/mu) with eps = eps0 eps_r, mu = mu0 mu_r,   c1 = (sigma, eps_r, 0, 0)
struct MatCoef {
    float4 c0, c1;
};

// Media as the kernels see them.
struct MediaView {
    MatCoef uniform;         // kUniform
    const uint8_t* id;       // kTable: material id per cell
    const MatCoef* table;    // kTable: coefficients per material
    const float* eps_r;      // kPerCell: raw values; coefficients are formed per cell
    const float* mu_r;
    const float* sigma;
};

// One cell touched by sources: its current entries, the first of them (in nearly every case the only
// one) held here, and the source slots that impose fields. One record, so that a cell's sources take
// one round trip to memory instead of a chain of two.
struct __align__(16) SpecialCell {
    float w[3];     // first current entry: weights and source slot
    int src;
    int begin, end;  // its entries in entry_src / entry_w (begin == end: no current)
    uint32_t impose_mask;  // bit k set: source slot k imposes fields at this cell
    int unused;
};

// Merged list of cells touched by sources ("special cells"), sorted by cell index.
struct SourceView {
    int n_special;
    const int* cell;              // [n_special]
    const SpecialCell* first;     // [n_special]
    const int* entry_src;         // source slot of each current entry
    const float* entry_w;         // 3 weights per current entry
    const int* block_begin;       // [blocks + 1] for the blocks of kBlock cells of the step range
                                  // [cell_begin, cell_end): where each block's cells start in `cell`
                                  // (null without source cells)
};

// The source cells of block `b` of a launch over the step range (one thread per cell), recomputed
// after the block's ordinary updates: a barrier, so that their values replace the ordinary ones,
// then update(i, m) for every source cell i = cell[m] of the block. Every thread of the block must
// call this (the barrier), whether or not it had a cell of its own.
template <class Update>
__device__ __forceinline__ void block_source_cells(const SourceView& sv, int b, Update&& update) {
    if (!sv.block_begin) return;
    const int lo = sv.block_begin[b], hi = sv.block_begin[b + 1];
    if (hi <= lo) return;
    __syncthreads();
    for (int m = lo + (int)threadIdx.x; m < hi; m += (int)blockDim.x) update(sv.cell[m], m);
}

// Per-step source values s_k(t) and the constant imposed-field vectors of each slot.
struct SourceScalars {
    float s[kMaxSources];
    float E0[kMaxSources][3];
    float B0[kMaxSources][3];
};

struct StepArgs {
    const void* fin;    // MM: float4[12][n]; HV: float4[6][n]
    void* fout;
    const void* fin2;   // HV: float2[6][n]
    void* fout2;
    const float* rho_in;  // MM rest population f_0^(0) (track_rho), else null
    float* rho_out;
    Geometry g;
    int media_mode;
    MediaView media;
    SourceView sv;
    SourceScalars sc;
    float eps0, mu0;
    int storage;      // StorageKind
    float scale;      // 16-bit storage: stored = f * scale
    float inv_scale;  // 1 / scale
    float* rec;       // adjoint record of this step (recording kernels only): kRecordFloats[model] x n
    int cell_begin, cell_end;  // cells the step and reduction launches cover (a z-slab skips its ghost planes)
};

// Per-cell record an adjoint step needs from its forward step: MM X = D' - mu0 J_ext / 4 (E is an
// exact function of X and the medium, recomputed by the same operations), HV E.
constexpr int kRecordFloatsMM = 3;
constexpr int kRecordFloatsHV = 3;

// Field output: for each selected field a 3 x n block; null pointers are skipped.
struct FieldsOut {
    float* E;
    float* B;
    float* D;
    float* H;
    float* J;
};

// --- population storage traits -----------------------------------------------------------
// Pack4<S>: four populations (one MM direction group, or HV's e_x, e_y, e_z, h_x) as one vector;
// Pack2<S>: two populations (HV's h_y, h_z). FP32: float4 / float2; 16-bit: 8 / 4 bytes.
// kReadOnly: nothing writes *p while the kernel exists, not even its predecessor (see launch_after).
template <bool kReadOnly, class T>
__device__ __forceinline__ T read(const T* p) {
    if constexpr (kReadOnly) return __ldg(p);
    else return *p;
}

template <int S>
struct Pack4;
template <int S>
struct Pack2;

template <>
struct Pack4<kF32> {
    using T = float4;
    __device__ static float4 unpack(T u, float) { return u; }
    template <bool kReadOnly = false>
    __device__ static float4 load(const T* p, float) { return read<kReadOnly>(p); }
    __device__ static T pack(float4 v, float) { return v; }
};
template <>
struct Pack2<kF32> {
    using T = float2;
    __device__ static float2 unpack(T u, float) { return u; }
    __device__ static float2 load(const T* p, float) { return *p; }
    __device__ static T pack(float2 v, float) { return v; }
};

template <>
struct Pack4<kF16> {
    using T = uint2;
    template <bool kReadOnly = false>
    __device__ static float4 load(const T* p, float inv) { return unpack(read<kReadOnly>(p), inv); }
    __device__ static float4 unpack(T u, float inv) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
        return make_float4(a.x * inv, a.y * inv, b.x * inv, b.y * inv);
    }
    __device__ static T pack(float4 v, float scale) {
        const __half2 a = __floats2half2_rn(v.x * scale, v.y * scale);
        const __half2 b = __floats2half2_rn(v.z * scale, v.w * scale);
        return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
};
template <>
struct Pack2<kF16> {
    using T = uint32_t;
    __device__ static float2 load(const T* p, float inv) { return unpack(*p, inv); }
    __device__ static float2 unpack(T u, float inv) {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&u));
        return make_float2(a.x * inv, a.y * inv);
    }
    __device__ static T pack(float2 v, float scale) {
        const __half2 a = __floats2half2_rn(v.x * scale, v.y * scale);
        return *reinterpret_cast<const uint32_t*>(&a);
    }
};

template <>
struct Pack4<kBF16> {
    using T = uint2;
    template <bool kReadOnly = false>
    __device__ static float4 load(const T* p, float inv) { return unpack(read<kReadOnly>(p), inv); }
    __device__ static float4 unpack(T u, float inv) {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
        const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
        return make_float4(a.x * inv, a.y * inv, b.x * inv, b.y * inv);
    }
    __device__ static T pack(float4 v, float scale) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x * scale, v.y * scale);
        const __nv_bfloat162 b = __floats2bfloat162_rn(v.z * scale, v.w * scale);
        return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
};
template <>
struct Pack2<kBF16> {
    using T = uint32_t;
    __device__ static float2 load(const T* p, float inv) { return unpack(*p, inv); }
    __device__ static float2 unpack(T u, float inv) {
        const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
        return make_float2(a.x * inv, a.y * inv);
    }
    __device__ static T pack(float2 v, float scale) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x * scale, v.y * scale);
        return *reinterpret_cast<const uint32_t*>(&a);
    }
};

// 24-bit storage. A value x (already scaled) is kept as h = x rounded toward zero to FP16 and an
// unsigned byte q = |x - h| / (ulp(h) / 256) rounded to nearest, where ulp(h) = 2^(max(E, 1) - 25)
// for h's biased exponent E (2^-24 for zero and subnormal h). x - h is exact in FP32 (h is x cut to
// fewer digits) and lies in [0, ulp(h)) in magnitude, so q is 0 ... 256; 256 carries into h, which
// moves one FP16 value away from zero (the bit pattern + 1), with q = 0, exactly. The value
// h + sign(h) q ulp(h) / 256 then keeps 19 significant bits where FP16 keeps 11 (relative error at
// most 2^-19 for normal h), and it decodes exactly: it needs at most 20 bits. |x| beyond FP16's
// largest value saturates there. The halves of a direction group and their bytes live in separate
// planes (a group's 4 halves as one 8-byte word, its 4 bytes as one 4-byte word), so each is one
// coalesced access.
//
// The common cases are computed without branches and without conversion instructions, on the
// value's FP32 bits. Write W for the FP32 pattern of |stored value| * 2^-112: for a normal h it is
// [0][e5 as the exponent field][h's 10 mantissa bits][q][5 zero bits], for a zero or subnormal h the
// denormal (h's bits * 256 + q) * 2^5; in both cases W = (h without its sign) << 13 | q << 5.
//   Decode: W from the stored bits, then W * 2^112 * 2^112, the sign, * 2^-112 / scale. The first
//   product is exact; the second overflows to infinity exactly for h's infinities and NaN (exponent
//   31, values >= 2^16; a NaN decodes as an infinity), and is exact otherwise. Denormal W needs FP32
//   denormals kept, which this build does (no flush to zero).
//   Encode, 2^-14 <= |x| < 2^15 (h normal): |x| * 2^-112 is exact and normal; its bits rounded to
//   nearest at bit 5 (halves to even) are W. |x| < 2^-14: |x| + 2^-9 rounds |x| to a multiple of
//   2^-32 (halves to even) and its low 23 bits are h's bits * 256 + q. Either way a carry out of q
//   runs into h, as the definition's carry does.
//   |x| >= 2^15, infinities and NaN go to encode_rare, the definition written out.
static __device__ __noinline__ void f24_encode_rare(float x, unsigned& h, unsigned& q);
struct F24 {
    __device__ static float join(unsigned z, float inv) {  // z: h in bits 31..16, q in bits 15..8
        const float w = __uint_as_float((z >> 3) & 0x0fffffe0u);
        const float m = (w * 0x1p112f) * 0x1p112f;
        return (__uint_as_float(__float_as_uint(m) | (z & 0x80000000u)) * 0x1p-112f) * inv;
    }
    // Bits of the stored pair of x = v * scale: h in bits 15..0, q in bits 23..16 (for packing).
    __device__ static unsigned split(float v, float scale) {
        const float x = v * scale, a = fabsf(x);
        const unsigned b = __float_as_uint(x);
        const unsigned zn = __float_as_uint(a * 0x1p-112f);
        const unsigned wn = zn + 0xfu + ((zn >> 5) & 1u);                         // to nearest at bit 5
        const unsigned ws = (__float_as_uint(a + 0x1p-9f) & 0x7fffffu) << 5;       // multiple of 2^-32
        const unsigned w = (a < 0x1p-14f ? ws : wn) | ((b >> 3) & 0x10000000u);    // sign into bit 28
        unsigned out = (w >> 13) | ((w << 11) & 0x00ff0000u);
        if (!(a < 0x1p15f)) {
            unsigned h, q;
            f24_encode_rare(x, h, q);
            out = h | (q << 16);
        }
        return out;
    }
    // Four values: halves at hi[idx], bytes at lo[idx].
    __device__ static float4 load4(const uint2* hi, const unsigned* lo, size_t idx, float inv) {
        const uint2 h = hi[idx];
        const unsigned q = lo[idx];
        return make_float4(join(__byte_perm(h.x, q, 0x1040), inv), join(__byte_perm(h.x, q, 0x3250), inv),
                           join(__byte_perm(h.y, q, 0x1060), inv), join(__byte_perm(h.y, q, 0x3270), inv));
    }
    __device__ static void store4(uint2* hi, unsigned* lo, size_t idx, float4 v, float scale) {
        const unsigned s0 = split(v.x, scale), s1 = split(v.y, scale), s2 = split(v.z, scale), s3 = split(v.w, scale);
        hi[idx] = make_uint2(__byte_perm(s0, s1, 0x5410), __byte_perm(s2, s3, 0x5410));
        lo[idx] = __byte_perm(__byte_perm(s0, s1, 0x0062), __byte_perm(s2, s3, 0x0062), 0x5410);
    }
    // Two values: halves at hi[idx], bytes at lo[idx].
    __device__ static float2 load2(const unsigned* hi, const unsigned short* lo, size_t idx, float inv) {
        const unsigned h = hi[idx];
        const unsigned q = lo[idx];
        return make_float2(join(__byte_perm(h, q, 0x1040), inv), join(__byte_perm(h, q, 0x3250), inv));
    }
    __device__ static void store2(unsigned* hi, unsigned short* lo, size_t idx, float2 v, float scale) {
        const unsigned s0 = split(v.x, scale), s1 = split(v.y, scale);
        hi[idx] = __byte_perm(s0, s1, 0x5410);
        lo[idx] = (unsigned short)__byte_perm(s0, s1, 0x0062);
    }
};

// The definition itself, for |x| >= 2^15, infinities and NaN (x already scaled).
static __device__ __noinline__ void f24_encode_rare(float x, unsigned& h, unsigned& q) {
    const __half hh = __float2half_rz(x);
    h = __half_as_ushort(hh);
    const float r = fabsf(x - __half2float(hh));
    const unsigned e = max((h >> 10) & 0x1fu, 1u);
    const int k = __float2int_rn(r * __uint_as_float((160u - e) << 23));  // |r| / 2^(e - 33)
    if (k < 256) {
        q = (unsigned)max(k, 0);
    } else if (k == 256 && (h & 0x7fffu) < 0x7bffu) {
        h += 1;  // the next FP16 value away from zero
        q = 0;
    } else {
        q = 255;  // beyond FP16's largest value
    }
}

// Host-side dispatch of a runtime storage kind / media mode to a compile-time constant.
template <class F>
inline void with_storage(int s, F&& f) {
    if (s == kBF16) f(std::integral_constant<int, kBF16>{});
    else if (s == kF16) f(std::integral_constant<int, kF16>{});
    else if (s == kF24) f(std::integral_constant<int, kF24>{});
    else f(std::integral_constant<int, kF32>{});
}
// The same for the two-step passes, which keep populations in their storage format in shared
// memory or L2 and have no 24-bit form (the host never selects a pass for kF24 storage).
template <class F>
inline void with_pass_storage(int s, F&& f) {
    if (s == kBF16) f(std::integral_constant<int, kBF16>{});
    else if (s == kF16) f(std::integral_constant<int, kF16>{});
    else if (s == kF32) f(std::integral_constant<int, kF32>{});
}
template <class F>
inline void with_media(int m, F&& f) {
    if (m == kTable) f(std::integral_constant<int, kTable>{});
    else if (m == kPerCell) f(std::integral_constant<int, kPerCell>{});
    else f(std::integral_constant<int, kUniform>{});
}

inline int blocks_for(int n) { return (n + kBlock - 1) / kBlock; }

// Grid of a persistent launch: resident blocks per SM x the current device's SM count.
inline int fused_grid(int blocks_per_sm) {
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    return std::max(1, blocks_per_sm) * std::max(1, sms);
}

// Allows `kernel` dynamic shared memory beyond 48 KB on the current device; false with the error left for
// cudaGetLastError. The attribute belongs to the kernel on one device, so it is set once on each that runs
// it: bit d of `done`, the kernel's own record, says that device d has it (threads that meet here set it
// twice, to the same value).
template <class Kernel>
inline bool allow_shared(std::atomic<unsigned long long>& done, Kernel* kernel, size_t bytes) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return false;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (done.load(std::memory_order_relaxed) & bit) return true;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) != cudaSuccess) return false;
    done.fetch_or(bit, std::memory_order_relaxed);
    return true;
}

// --- dependent launches ---------------------------------------------------------------------------
// Consecutive kernels of a lattice depend on one another, so a stream leaves a gap between them:
// drain, completion, launch, first loads. A kernel launched with launch_after may be set up while its
// predecessor still runs; every thread calls after_predecessor() before it touches memory, which
// waits until the predecessor has completed and its writes are visible, and then lets the next such
// kernel be set up. A predecessor that is no such kernel (a copy, a memset, the caller's own kernel)
// is waited for in the same way or by the stream itself. What a predecessor may write (populations,
// records, gradients, partial sums, the caller's arrays) is therefore not read-only for such a kernel's
// lifetime: it is read with plain loads through pointers that are not both const and __restrict__, which the
// wait's memory clobber holds back; __ldg is for what only the host writes, before the launch (media, source
// lists). That costs nothing measurable but in the MM tiled pass, whose loads the compiler then no longer
// moves across its barriers (256^3: 637 us per step against 592), and in the MM backward step of large
// lattices with a medium per cell: these are launched plainly.
// Measured on GB300 (us per single step, against plain launches, both with source cells recomputed at the
// end): MM 32^3 4.3 (6.2), 64^3 11.7 (14.1), 128^3 115.3 (117.6); HV 32^3 3.6 (6.2), 64^3 7.5 (10.3),
// 97 x 53 x 71 12.4 (14.4). The ring passes keep plain launches too: a memset of their counter lies between
// them.
// The single, recording, backward and batched steps and the line kernel wait alone and let the next launch in
// late (wait_predecessor; a block's end lets it in by itself): blocks set up while all of a small launch's
// still run come to lie unevenly on the SMs (us per step, let in at once / at the blocks' ends: MM 40^3 4.9 /
// 3.8, HV 48^3 4.8 / 3.8, 24^3 the other way round, 2.2 / 2.4; batched, 62,768 cells of F24 MM 8.8 / 6.6;
// adjoint of 40^3, MM 11.4 / 9.2, HV 9.1 / 7.5). So do loads of fields and populations of up to kLetLateBlocks blocks (init MM 56^3, 686 blocks, 9.2 / 6.7; 72^3,
// 1458, 12.4 / 12.3; 80^3, 2000, 18.0 / 18.2; 256^3 549 / 557).
constexpr unsigned kLetLateBlocks = 1500;
__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void after_predecessor() {
    wait_predecessor();
    let_successor();
}
__device__ __forceinline__ void after_predecessor_by_size() {
    wait_predecessor();
    if (gridDim.x > kLetLateBlocks) let_successor();
}

template <class... Params, class... Args>
inline void launch_after(void (*kernel)(Params...), dim3 grid, int block, size_t smem, cudaStream_t st, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);  // errors: cudaGetLastError by the caller
}

// --- compile-time loop ---------------------------------------------------------------------
template <int I, int N, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        static_for<I + 1, N>(f);
    }
}

// Signed term c * x for a compile-time c in {-1, 0, 1}; adds nothing for c = 0.
template <int C>
__device__ __forceinline__ void acc(float& sum, float x) {
    if constexpr (C > 0) sum += x;
    else if constexpr (C < 0) sum -= x;
}

// Pairwise (tree) sum of t[B..E) with compile-time bounds. The moment sums use it: on long runs
// it halves the accumulated FP32 error of a left-to-right sum at no extra cost.
template <int B, int E, int N>
__device__ __forceinline__ float pairwise_sum(const float (&t)[N]) {
    static_assert(E > B, "empty sum");
    if constexpr (E - B == 1) {
        return t[B];
    } else {
        constexpr int M = B + (E - B) / 2;
        return pairwise_sum<B, M>(t) + pairwise_sum<M, E>(t);
    }
}

// --- periodic neighbour addressing ---------------------------------------------------------
// Linear-index contributions of the three coordinates shifted by -1, 0, +1 with periodic wrap.
struct Neighbourhood {
    int xo[3], yo[3], zo[3];
    int x, y, z;
};

__device__ __forceinline__ Neighbourhood neighbourhood(const Geometry& g, int i) {
    const int nxy = g.nx * g.ny;
    const int z = (int)(((unsigned long long)(unsigned)i * g.mxy) >> (32 + g.kxy));
    const int r = i - z * nxy;
    const int y = (int)(((unsigned long long)(unsigned)r * g.mx) >> (32 + g.kx));
    const int x = r - y * g.nx;
    Neighbourhood h;
    h.x = x;
    h.y = y;
    h.z = z;
    h.xo[0] = x == 0 ? g.nx - 1 : x - 1;
    h.xo[1] = x;
    h.xo[2] = x == g.nx - 1 ? 0 : x + 1;
    const int ym = y == 0 ? g.ny - 1 : y - 1, yp = y == g.ny - 1 ? 0 : y + 1;
    h.yo[0] = ym * g.nx;
    h.yo[1] = y * g.nx;
    h.yo[2] = yp * g.nx;
    const int zm = z == 0 ? g.nz - 1 : z - 1, zp = z == g.nz - 1 ? 0 : z + 1;
    h.zo[0] = zm * nxy;
    h.zo[1] = z * nxy;
    h.zo[2] = zp * nxy;
    return h;
}

// Ask L2 to fetch the line holding p ahead of a load of it; nothing waits for it and no register
// receives it. Callers pass only addresses they are about to load themselves.
__device__ __forceinline__ void prefetch_l2(const void* p) {
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Prefetch into L2 the medium of cell i (nothing for a uniform medium).
template <int M>
__device__ __forceinline__ void prefetch_media(const MediaView& m, int i) {
    if constexpr (M == kTable) {
        prefetch_l2(&m.id[i]);
    } else if constexpr (M == kPerCell) {
        prefetch_l2(&m.eps_r[i]);
        prefetch_l2(&m.mu_r[i]);
        prefetch_l2(&m.sigma[i]);
    }
}

// Ask L1 to fetch the line holding p ahead of a load of it; nothing waits for it and no register
// receives it. Callers pass only addresses that they or their block are about to load.
__device__ __forceinline__ void prefetch_l1(const void* p) {
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// Index of the cell at offset (sx, sy, sz) in {-1, 0, 1}^3.
template <int SX, int SY, int SZ>
__device__ __forceinline__ int shifted(const Neighbourhood& h) {
    return h.xo[SX + 1] + h.yo[SY + 1] + h.zo[SZ + 1];
}

// x / d rounded to nearest, from r = RN(1/d): q = RN(x r), e = x - q d (exact with a fused
// multiply-add), result RN(q + e r). By Markstein's theorem on FMA-based division this is the
// correctly rounded quotient (away from underflow and overflow), without a divide instruction or
// its special-case branch.
__device__ __forceinline__ float div_rn(float x, float d, float r) {
    const float q = __fmul_rn(x, r);
    const float e = __fmaf_rn(-q, d, x);
    return __fmaf_rn(e, r, q);
}

enum ModelKind { kModelMM = 0, kModelHV = 1 };

// What is stored of cell i's medium, before the coefficients are looked up or formed from it.
template <int M>
struct RawMedium {
    unsigned id = 0;                        // kTable
    float eps_r = 1.f, mu_r = 1.f, sigma = 0.f;  // kPerCell
    __device__ __forceinline__ void load(const MediaView& m, int i) {
        if constexpr (M == kTable) {
            id = __ldg(&m.id[i]);
        } else if constexpr (M == kPerCell) {
            eps_r = __ldg(&m.eps_r[i]);
            mu_r = __ldg(&m.mu_r[i]);
            sigma = __ldg(&m.sigma[i]);
        }
    }
};

// Coefficients from it. Per-cell media form them here from the raw values (true divisions).
template <int Model, int M>
__device__ __forceinline__ MatCoef coef_of(const MediaView& m, const RawMedium<M>& raw, float eps0, float mu0) {
    if constexpr (M == kUniform) {
        return m.uniform;
    } else if constexpr (M == kTable) {
        const MatCoef* t = &m.table[raw.id];
        MatCoef c;
        c.c0 = __ldg(&t->c0);
        c.c1 = __ldg(&t->c1);
        return c;
    } else {
        const float er = raw.eps_r, mr = raw.mu_r, sg = raw.sigma;
        MatCoef c;
        if constexpr (Model == kModelMM) {
            c.c0 = make_float4(er, 1.f / er, 1.f / (1.f + 0.5f * (sg / er)), 0.25f / mr);
            c.c1 = make_float4(sg, mr, 0.f, 0.f);
        } else {
            const float eps = eps0 * er, mu = mu0 * mr;
            c.c0 = make_float4(eps, 1.f / eps, mu, 1.f / mu);
            c.c1 = make_float4(sg, er, 0.f, 0.f);
        }
        return c;
    }
}

template <int Model, int M>
__device__ __forceinline__ MatCoef load_coef(const MediaView& m, int i, float eps0, float mu0) {
    RawMedium<M> raw;
    raw.load(m, i);
    return coef_of<Model, M>(m, raw, eps0, mu0);
}

// External current and imposed fields of special cell m at the current step.
struct CellSource {
    float3 J;
    float3 E;
    float3 B;
    bool imposed;
};

// The sums are explicit fused multiply-adds, so that every kernel that inlines this gets the same bits.
__device__ __forceinline__ CellSource cell_source(const SourceView& sv, const SourceScalars& sc, int m) {
    CellSource cs;
    cs.J = make_float3(0.f, 0.f, 0.f);
    cs.E = make_float3(0.f, 0.f, 0.f);
    cs.B = make_float3(0.f, 0.f, 0.f);
    const int b = sv.first[m].begin, e = sv.first[m].end;
    for (int k = b; k < e; ++k) {
        const float s = sc.s[sv.entry_src[k]];
        cs.J.x = __fmaf_rn(sv.entry_w[3 * k + 0], s, cs.J.x);
        cs.J.y = __fmaf_rn(sv.entry_w[3 * k + 1], s, cs.J.y);
        cs.J.z = __fmaf_rn(sv.entry_w[3 * k + 2], s, cs.J.z);
    }
    const uint32_t mask = sv.first[m].impose_mask;
    cs.imposed = mask != 0u;
    for (int k = 0; k < kMaxSources; ++k) {
        if ((mask >> k) & 1u) {
            const float s = sc.s[k];
            cs.E.x = __fmaf_rn(sc.E0[k][0], s, cs.E.x);
            cs.E.y = __fmaf_rn(sc.E0[k][1], s, cs.E.y);
            cs.E.z = __fmaf_rn(sc.E0[k][2], s, cs.E.z);
            cs.B.x = __fmaf_rn(sc.B0[k][0], s, cs.B.x);
            cs.B.y = __fmaf_rn(sc.B0[k][1], s, cs.B.y);
            cs.B.z = __fmaf_rn(sc.B0[k][2], s, cs.B.z);
        }
    }
    return cs;
}

// Block-wide sum of three doubles (blockDim.x == kBlock), stored by thread 0 in a fixed order.
__device__ __forceinline__ void block_sum3_store(double a0, double a1, double a2, double* out) {
    __shared__ double sh[3][kBlock / 32];
    for (int off = 16; off > 0; off >>= 1) {
        a0 += __shfl_down_sync(0xffffffffu, a0, off);
        a1 += __shfl_down_sync(0xffffffffu, a1, off);
        a2 += __shfl_down_sync(0xffffffffu, a2, off);
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) {
        sh[0][w] = a0;
        sh[1][w] = a1;
        sh[2][w] = a2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double s0 = 0.0, s1 = 0.0, s2 = 0.0;
        for (int k = 0; k < kBlock / 32; ++k) {
            s0 += sh[0][k];
            s1 += sh[1][k];
            s2 += sh[2][k];
        }
        out[0] = s0;
        out[1] = s1;
        out[2] = s2;
    }
}

// --- batched stepping of several lattices -------------------------------------------------
// One lattice of a batch as the batched kernels read it from device memory. The host rewrites the
// array before every batched call, so a captured graph of the call replays on fresh contents.
struct BatchLattice {
    StepArgs base;         // geometry, media, special cells, imposed vectors, storage, eps0, mu0
    void* buf[2];          // population buffers; step j reads buf[(cur0 + j) & 1]
    void* buf2[2];         // HV second arrays (MM: unused)
    float* rho[2];         // MM rest population f_0^(0) when tracked, else null
    const float* s_table;  // source values s_k(t0 + j + 1) at [k * s_stride + j]
    int s_stride;
    int n_src;
    int cur0;   // buffer index holding the state when the call starts
    int steps;  // steps this lattice advances in the call
};

// A block's share of the batch: cells [begin, begin + blockDim) of one lattice (or, for the
// source-cell launch, special cells [begin, begin + blockDim)).
struct BatchTile {
    int lattice;
    int begin;
};

// StepArgs of lattice L at batch step j (buffers and storage; sources are filled by the caller).
__device__ __forceinline__ StepArgs batch_args(const BatchLattice* __restrict__ L, int j) {
    StepArgs a;
    a.g = L->base.g;
    a.media_mode = L->base.media_mode;
    a.media = L->base.media;
    const int in = (L->cur0 + j) & 1, out = in ^ 1;
    a.fin = L->buf[in];
    a.fout = L->buf[out];
    a.fin2 = L->buf2[in];
    a.fout2 = L->buf2[out];
    a.rho_in = L->rho[in];
    a.rho_out = L->rho[out];
    a.eps0 = L->base.eps0;
    a.mu0 = L->base.mu0;
    a.storage = L->base.storage;
    a.scale = L->base.scale;
    a.inv_scale = L->base.inv_scale;
    a.sv = L->base.sv;
    return a;
}

// Source values of lattice L at batch step j, and its imposed-field vectors.
__device__ __forceinline__ void batch_sources(const BatchLattice* __restrict__ L, int j, StepArgs& a) {
    for (int k = 0; k < L->n_src; ++k) {
        a.sc.s[k] = L->s_table[k * L->s_stride + j];
        for (int q = 0; q < 3; ++q) {
            a.sc.E0[k][q] = L->base.sc.E0[k][q];
            a.sc.B0[k][q] = L->base.sc.B0[k][q];
        }
    }
}

struct BatchLaunch {
    const BatchLattice* lat;
    const BatchTile* tiles;   // main tiles, lattices in decreasing step count
    const BatchTile* stiles;  // special-cell tiles, same lattice order
    int block;                // threads per block of the main launch (128 or 256)
    int grid_cap;             // persistent launch: blocks in the grid (0 = one block per tile)
    int storage;
    bool rho;
};

// --- adjoint (gradients of a plane loss with respect to eps_r and sigma) ---------------------
// One backward step reverses the forward iteration n -> n+1. nu^{n+1} = dL/df^{n+1} holds the adjoint
// of every cell's pre-collision populations (FP32, the population group layout). The adjoint of
// cell x's post-collision values is nu^{n+1} at x + v_d (advection reversed); the transposed
// collision gives nu^n(x), plus the derivative of the loss of time n when x lies in the loss plane.
struct AdjointArgs {
    StepArgs a;            // media, sources of iteration n + 1; record of the forward step in a.rec
                           // (the terminal launch reads the final state from a.fin / a.fin2 instead)
    const void* nu_in;     // nu^{n+1} (null for the terminal launch)
    const void* nu_in2;    // HV second array
    void* nu_out;          // nu^n
    void* nu_out2;
    float* grad_eps;       // dL/d eps_r per cell, accumulated
    float* grad_sigma;     // dL/d sigma per cell, accumulated (null: not computed)
    const uint8_t* special_mask;  // non-zero at source cells, which the second launch handles
    int plane_axis, plane_index;  // loss plane: cells whose coordinate on plane_axis is plane_index
    int loss_active;              // add the plane loss term of time n
    double* loss_plane;           // |E|^2 summed over time, per plane cell (slot k as in plane_cell);
                                  // the terminal launch writes it, the others add
};

// Cells of the loss plane, and whether a cell lies in it.
__device__ __forceinline__ int plane_cells(const Geometry& g, int axis) {
    return axis == 0 ? g.ny * g.nz : (axis == 1 ? g.nx * g.nz : g.nx * g.ny);
}
__device__ __forceinline__ int plane_cell(const Geometry& g, int axis, int index, int k) {
    if (axis == 0) return index + g.nx * k;  // k = y + ny z
    if (axis == 1) {
        const int z = k / g.nx, x = k - z * g.nx;
        return x + g.nx * (index + g.ny * z);
    }
    return k + g.nx * g.ny * index;  // k = x + nx y
}
// Slot k of a plane cell: the inverse of plane_cell.
__device__ __forceinline__ int plane_slot(const Neighbourhood& h, const Geometry& g, int axis) {
    return axis == 0 ? h.y + g.ny * h.z : (axis == 1 ? h.x + g.nx * h.z : h.x + g.nx * h.y);
}
__device__ __forceinline__ bool in_plane(const Neighbourhood& h, const Geometry& g, int axis, int index) {
    if (axis == 0) return h.xo[1] == index;
    if (axis == 1) return h.yo[1] == index * g.nx;
    return h.zo[1] == index * g.nx * g.ny;
}

// |E|^2 of a plane cell into its loss slot: written by the terminal launch (time T), then added by
// the launch of each earlier time, so every slot sums its times in the order T, T-1, ..., 1.
template <bool kFirst>
__device__ __forceinline__ void add_plane_loss(const AdjointArgs& A, const Neighbourhood& h, float3 E) {
    const double e2 = (double)E.x * E.x + (double)E.y * E.y + (double)E.z * E.z;
    double* slot = A.loss_plane + plane_slot(h, A.a.g, A.plane_axis);
    if constexpr (kFirst) *slot = e2;
    else *slot += e2;
}

// --- two time steps per pass over the populations ---------------------------------------------
// A step of cell x reads only the populations of its 3 x 3 x 3 neighbourhood. So step t + 1 of a
// cell can run as soon as step t has produced its 27 neighbours. One persistent launch runs both
// steps as a wavefront along z:
//   phase A(p): step t of plane p, from the A/B buffer into an intermediate plane;
//   phase B(p): step t + 1 of plane p, from the intermediate planes p - 1, p, p + 1 into the other
//     A/B buffer.
// The intermediate planes of 1 .. nz - 2 live in a ring of R plane slots, small enough to stay in
// L2. Planes 0 and nz - 1 are needed at both ends of the periodic wavefront, so they have slots
// of their own. Each step's HBM traffic is then one read or one write of the populations instead
// of both.
// Phases run in the order A(nz-1), A(0), .., A(L-1), then B(k), A(k + L) for k = 0 .. nz-2-L,
// then the remaining B phases (L >= 2: B(k) needs A(k + 1); R >= L + 1 keeps every wait on an
// earlier item). A phase is `tiles` tiles of tile_cells consecutive cells of its plane. A tile
// also recomputes the source cells among its own cells (after a barrier of its compute threads, so
// that their values replace those of the ordinary update), so a finished tile is final, however
// many source cells a plane holds. Blocks take tiles in that order from a counter, and a tile waits
// only for tiles taken before it:
//   * tile j of B(p) waits for the tiles of A(p - 1), A(p), A(p + 1) holding the rows next to its
//     own (the cells it pulls from);
//   * tile j of A(p) waits for the same neighbourhood of tiles of the three B phases that read the
//     slot's previous plane, p - R.
// Tiles publish the pass number in a flag of their own, so the flags need no reset between passes.
// Every wait has a time limit; past it the pass sets `abort` and every block stops. A negative
// limit makes every item that depends on another give up at its first check, met or not: the host
// uses it to drive the time-out path deterministically in tests.
struct FusedArgs {
    void* ring;   // R slots of one plane of intermediate populations (the model's group layout)
    void* lo;     // slot of plane 0
    void* hi;     // slot of plane nz - 1
    void* ring2;  // HV: the same for the pair arrays (null for MM)
    void* lo2;
    void* hi2;
    int R;
    int L;                      // A runs L planes ahead of B in the item order (R >= L + 1)
    int tile_cells;             // cells per tile: a multiple of kBlock (each thread takes every kBlock-th)
    int tiles;                  // tiles per plane
    int epoch;                  // this pass's number (>= 1); flags hold the last pass they finished
    int* next;                  // item counter (zero at launch)
    int* tile_flag;             // 2 nz tiles flags, A then B
    int* abort;                 // set when a wait timed out
    const int* tile_special;    // nz tiles + 1 offsets of each tile's cells in the special-cell list
    long long timeout_ns;       // < 0: give up at the first dependency check
};

enum { kPhaseA = 0, kPhaseB = 1 };

__host__ __device__ __forceinline__ void fused_phase(int q, int nz, int L, int* type, int* plane) {
    if (q < L + 1) {
        *type = kPhaseA;
        *plane = q == 0 ? nz - 1 : q - 1;
        return;
    }
    const int j = q - (L + 1), pairs = nz - 1 - L;
    if (j < 2 * pairs) {
        *type = (j & 1) ? kPhaseA : kPhaseB;
        *plane = (j & 1) ? (j >> 1) + L : (j >> 1);
        return;
    }
    *type = kPhaseB;
    *plane = pairs + (j - 2 * pairs);
}

__device__ __forceinline__ long long global_ns() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ int load_acquire(const int* p) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Wait until *ctr >= target; false when the pass was aborted or the wait timed out (then aborts).
// The loop does not sleep: the L2 round trip of each look paces it, and the pass is bound by how
// soon a published item is seen (sleeping backoff measured 0.6 % (MM) and 1 % (HV) slower).
__device__ inline bool fused_wait(const FusedArgs& F, const int* ctr, int target) {
    if (load_acquire(ctr) >= target) return true;
    const long long t0 = global_ns();
    while (load_acquire(ctr) < target) {
        if (load_acquire(F.abort)) return false;
        if (global_ns() - t0 > F.timeout_ns) {
            atomicExch(F.abort, 1);
            return false;
        }
    }
    return true;
}

// Tiles holding the rows y0 - 1 .. y1 + 1 (cyclically) around the rows y0 .. y1 of tile j: the
// first tile and how many. A cell pulls from (x +- 1, y +- 1), and the x wrap stays in its row.
__host__ __device__ __forceinline__ void tile_window(int j, int tiles, int tile_cells, int nx, int nxy, int* first,
                                                     int* count) {
    const int c0 = j * tile_cells, c1 = (c0 + tile_cells < nxy ? c0 + tile_cells : nxy) - 1;
    const int y0 = c0 / nx, y1 = c1 / nx;
    const long long span = (long long)(y1 - y0 + 3) * nx;
    if (span >= nxy) {
        *first = 0;
        *count = tiles;
        return;
    }
    int lo = (y0 - 1) * nx;
    if (lo < 0) lo += nxy;
    const int hi = lo + (int)span - 1;  // may pass nxy: wraps
    *first = lo / tile_cells;
    *count = hi < nxy ? hi / tile_cells - *first + 1 : (tiles - *first) + ((hi - nxy) / tile_cells + 1);
    if (*count > tiles) *count = tiles;
}

// The phases a tile of phase (type, plane) waits for: the tiles of planes q[0..2] in phase *wtype
// within its window. B(p) reads the intermediate planes p - 1, p, p + 1 written by A; A(p) rewrites
// the ring slot whose previous plane, p - R, the B phases p - R - 1 .. p - R + 1 read. Returns the
// number of planes (0: nothing to wait for).
__host__ __device__ __forceinline__ int fused_waits_on(int type, int plane, int nz, int R, int* wtype, int* q) {
    if (type == kPhaseB) {
        *wtype = kPhaseA;
        q[0] = (plane + nz - 1) % nz;
        q[1] = plane;
        q[2] = (plane + 1) % nz;
        return 3;
    }
    const int prev = plane - R;
    if (!(plane >= 1 && plane <= nz - 2 && prev >= 1)) return 0;
    *wtype = kPhaseB;
    q[0] = prev - 1;
    q[1] = prev;
    q[2] = prev + 1;
    return 3;
}

// An item of a pass: tile j of phase (type, plane).
struct FusedItem {
    int type, plane, j;
};

__device__ __forceinline__ FusedItem fused_item(int item, int tiles, int nz, int L) {
    FusedItem it;
    const int q = item / tiles;
    it.j = item - q * tiles;
    fused_phase(q, nz, L, &it.type, &it.plane);
    return it;
}

// Dependencies of item `it`, checked by the 32 lanes of one warp at once: the tile flags of three
// planes' windows are spread over the lanes, so a satisfied item costs one round of loads. `own`
// is the item the same block runs just before this one: it is complete by the time this one
// starts (the block's barriers order it), so it is not waited for. Same verdict in every lane.
__device__ inline bool fused_ready_warp(const FusedArgs& F, int nz, FusedItem it, FusedItem own, int nx, int nxy,
                                        bool wait) {
    const int lane = threadIdx.x & 31;
    bool ok = true;
    // one look (wait == false) or a bounded wait
    auto reached = [&](const int* p, int target) { return wait ? fused_wait(F, p, target) : load_acquire(p) >= target; };
    int q[3];
    int wtype = 0;
    if (fused_waits_on(it.type, it.plane, nz, F.R, &wtype, q) == 0) return true;
    if (F.timeout_ns < 0) {  // negative limit: stop the pass at the first item with a dependency
        if (lane == 0) atomicExch(F.abort, 1);
        return false;
    }
    int first, count;
    tile_window(it.j, F.tiles, F.tile_cells, nx, nxy, &first, &count);
    for (int idx = lane; ok && idx < 3 * count; idx += 32) {
        const int k = idx / count;
        int t = first + (idx - k * count);
        if (t >= F.tiles) t -= F.tiles;
        if (own.type == wtype && own.plane == q[k] && own.j == t) continue;
        ok = reached(F.tile_flag + ((size_t)wtype * nz + q[k]) * F.tiles + t, F.epoch);
    }
    return __all_sync(0xffffffffu, ok);
}

// Publish a finished tile (after every store of the block: the caller's barrier orders them).
__device__ __forceinline__ void fused_publish(const FusedArgs& F, int nz, FusedItem it) {
    __threadfence();
    atomicExch(F.tile_flag + ((size_t)it.type * nz + it.plane) * F.tiles + it.j, F.epoch);
}

// Threads of a two-step block: kBlock compute threads and one scheduler warp.
constexpr int kFusedThreads = kBlock + 32;

// Shared-memory slots of one compute thread of a two-step pass, a float2 each, laid out [slot]
// [compute thread] so that a warp's accesses do not conflict. Populations wait there between a
// cell's pull and its collision instead of holding registers: at the pass's 72 registers per
// thread the compiler would otherwise spill more to local memory, whose stores go through to L2
// (256^3 dipole on GB300: the MM pass 2.5 % and the HV pass 1.7 % faster with the slots). The
// accesses are volatile so that the compiler keeps the round trip instead of forwarding the
// stored values in registers.
struct FusedStash {
    static constexpr bool kStash = true;
    __device__ bool keeps_record() const { return true; }  // a recording step writes this cell's record
    unsigned slot;  // shared address of this thread's slot 0; slot k lies k * kBlock * 8 bytes on
    __device__ void stash_put(int k, float x, float y) const {
        asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(slot + k * kBlock * 8), "f"(x), "f"(y));
    }
    __device__ void stash_get(int k, float& x, float& y) const {
        asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "r"(slot + k * kBlock * 8));
    }
};
// The same hooks for the single-step paths, which keep every value in registers.
struct NoStash {
    static constexpr bool kStash = false;
    __device__ bool keeps_record() const { return true; }  // a recording step writes this cell's record
    __device__ void stash_put(int, float, float) const {}
    __device__ void stash_get(int, float&, float&) const {}
};
__device__ __forceinline__ unsigned fused_stash_slot(const float2* slots) {
    return static_cast<unsigned>(__cvta_generic_to_shared(slots + threadIdx.x));
}

__device__ __forceinline__ void named_sync(int id, int count) {
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int count) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// The persistent loop. The scheduler warp (threads kBlock ..) takes the next item from the
// counter and looks at its inputs while the kBlock compute threads run the current one:
//   compute: bar.sync(handoff) -> read the item -> work -> bar.arrive(done) -> repeat;
//   scheduler: take item n+1 and look once at its inputs -> bar.sync(done) (item n finished) ->
//     if they were all there: hand n+1 over (bar.arrive(handoff)), then publish n while it runs;
//     otherwise: publish n first, then wait for n+1's inputs and hand it over.
// Publishing never waits behind another item's inputs, so the earliest unpublished item can
// always proceed (every item waits only for earlier ones); and in the usual case neither the
// check nor the publication's fence delays the compute threads. Item n+1's dependence on n
// itself is not looked up: the block's barriers order n before n+1.
// The scheduler also works out what the compute threads need of an item (`describe`: phase,
// plane, tile and the ring slots it reads or writes) while they run the previous one, and hands
// it over in shared memory, so the compute threads do no index arithmetic per item.
struct FusedDesc {
    int type, plane, j;
    int s_lo, s_hi;  // the tile's source cells: entries s_lo .. s_hi - 1 of the special-cell list
    void* ptr[6];
};

// Barrier of a two-step block's compute threads alone (ids 1 and 2 are the hand-off barriers).
constexpr int kComputeBarrier = 3;

template <class Describe, class Work>
__device__ inline void fused_loop(const FusedArgs& F, int nx, int nxy, int nz, Describe&& describe, Work&& work) {
    constexpr int kHandoff = 1, kDone = 2;
    __shared__ int s_item[2], s_ok[2];
    __shared__ FusedDesc s_desc[2];
    const int per_phase = F.tiles;
    const int total = 2 * nz * per_phase;
    if (threadIdx.x < kBlock) {
        for (int buf = 0;; buf ^= 1) {
            named_sync(kHandoff, kFusedThreads);
            const int item = s_item[buf];
            if (item >= total || !s_ok[buf]) return;
            work(s_desc[buf]);
            named_arrive(kDone, kFusedThreads);
        }
    }
    // scheduler warp
    const int lane = threadIdx.x & 31;
    const FusedItem none{-1, -1, -1};
    auto make_desc = [&](const FusedItem& it) {
        FusedDesc d;
        d.type = it.type;
        d.plane = it.plane;
        d.j = it.j;
        const int* ts = F.tile_special + (size_t)it.plane * F.tiles + it.j;
        d.s_lo = ts[0];
        d.s_hi = ts[1];
        describe(it, d);
        return d;
    };
    int item = 0;
    if (lane == 0) item = atomicAdd(F.next, 1);
    item = __shfl_sync(0xffffffffu, item, 0);
    bool ok = item >= total || fused_ready_warp(F, nz, fused_item(item, per_phase, nz, F.L), none, nx, nxy, true);
    if (lane == 0) {
        s_item[0] = item;
        s_ok[0] = ok ? 1 : 0;
        if (item < total) s_desc[0] = make_desc(fused_item(item, per_phase, nz, F.L));
    }
    named_arrive(kHandoff, kFusedThreads);
    for (int buf = 1;; buf ^= 1) {
        if (item >= total || !ok) return;
        const FusedItem cur = fused_item(item, per_phase, nz, F.L);
        int nxt = 0;
        if (lane == 0) nxt = atomicAdd(F.next, 1);
        nxt = __shfl_sync(0xffffffffu, nxt, 0);
        const FusedItem next = nxt < total ? fused_item(nxt, per_phase, nz, F.L) : none;
        const bool ready = nxt >= total || fused_ready_warp(F, nz, next, cur, nx, nxy, false);
        if (lane == 0) {  // slot `buf` held the item before `cur`, which every compute thread has finished
            s_item[buf] = nxt;
            if (nxt < total) s_desc[buf] = make_desc(next);
        }
        named_sync(kDone, kFusedThreads);  // the compute threads finished `cur`
        bool ok2 = true;
        if (ready) {
            if (lane == 0) s_ok[buf] = 1;
            named_arrive(kHandoff, kFusedThreads);
            if (lane == 0) fused_publish(F, nz, cur);
        } else {
            if (lane == 0) fused_publish(F, nz, cur);
            __syncwarp();
            ok2 = fused_ready_warp(F, nz, next, none, nx, nxy, true);
            if (lane == 0) s_ok[buf] = ok2 ? 1 : 0;
            named_arrive(kHandoff, kFusedThreads);
        }
        item = nxt;
        ok = ok2;
    }
}

// --- two time steps per pass in shared memory (overlapped tiles) ------------------------------
// A block owns a tile of TX x TY cells of each plane of a chunk of planes and works on it and a ring of
// one cell around it, the EX x EY = (TX + 2) x (TY + 2) "extended" cells. Marching up its chunk, it steps
// plane p of the extended tile (phase A, step t: pulls from the A/B buffer in HBM, results into
// shared memory), then an earlier plane q of the tile itself (phase B, step t + 1: pulls from the
// shared planes q - 1, q, q + 1, results into the other A/B buffer). The ring is what phase B's pulls
// reach outside the tile, so blocks never wait for one another; the ring's cells are stepped twice
// (by this block and by their own), the price of that independence. The intermediate step never
// leaves the SM: each pair of steps reads and writes the populations in HBM once, and writes them into
// L2 only twice (the fill and the output). Phase B pulls a direction with v_z = +1 from plane q - 1,
// v_z = 0 from q, v_z = -1 from q + 1, so each plane's directions are kept by v_z class only as long
// as they are read. The arithmetic is the single step's, so a pass equals two single steps bit for bit.
template <int EX_, int EY_>
struct TileShape {
    static constexpr int EX = EX_, EY = EY_, TX = EX - 2, TY = EY - 2, kCells = EX * EY;
};
using Tile = TileShape<16, 16>;
constexpr int kTileMin = 16;  // least nx and ny of a tiled lattice

struct TileArgs {
    int tiles_x, tiles_y;  // tiles per plane along x and y (a ragged last tile covers the rest)
    int chunk;             // planes per block; blockIdx.y selects the chunk
    const int* entry_off;  // tiles_x tiles_y nz + 1 offsets into entries, by (tile, plane)
    const int2* entries;   // (special-cell index m, extended-tile position) of every source cell of the
                           // tile's extended cells, by tile then plane
};

// Where an extended cell lies. Positions wrap periodically (on a lattice narrower than the extended tile
// some cells take two positions, stepped alike); a ragged last tile's core positions past the lattice's
// edge are not its own (the first tile steps those cells).
struct TileCell {
    int tile, bx, by;
    int x, row;  // the cell's x, and nx y
    bool core;
    int z0, z1;  // the block's planes
};

template <class Shape>
__host__ __device__ __forceinline__ bool tile_core(int local, int bx, int by, int nx, int ny) {
    const int ex = local % Shape::EX, ey = local / Shape::EX;
    return ex >= 1 && ex <= Shape::TX && ey >= 1 && ey <= Shape::TY && bx * Shape::TX + ex - 1 < nx &&
           by * Shape::TY + ey - 1 < ny;
}

__host__ __device__ __forceinline__ int tile_wrap(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// Lattice x (or y) of extended position e of tile b, for tiles of t own cells. With n >= kTileMin one wrap
// is enough: the last tile starts below n and an extended tile reaches at most t + 1 beyond its start.
__host__ __device__ __forceinline__ int tile_coord(int b, int e, int t, int n) { return tile_wrap(b * t - 1 + e, n); }

template <class Shape>
__device__ __forceinline__ TileCell tile_cell(const Geometry& g, const TileArgs& T, int local) {
    TileCell c;
    c.tile = blockIdx.x;
    c.by = blockIdx.x / T.tiles_x;
    c.bx = blockIdx.x - c.by * T.tiles_x;
    c.x = tile_coord(c.bx, local % Shape::EX, Shape::TX, g.nx);
    c.row = g.nx * tile_coord(c.by, local / Shape::EX, Shape::TY, g.ny);
    c.core = tile_core<Shape>(local, c.bx, c.by, g.nx, g.ny);
    c.z0 = blockIdx.y * T.chunk;
    c.z1 = min(c.z0 + T.chunk, g.nz);
    return c;
}

// In-plane parts of the cells around (x, row) and the planes around p: a pull reads
// plane[1 - vz] + x[1 - vx] + row[1 - vy]. Worked out anew for every plane: a dozen integer
// operations against six registers held throughout.
struct TilePull {
    int x[3], row[3], plane[3];
};
__device__ __forceinline__ TilePull tile_pull(const Geometry& g, const TileCell& c, int p) {
    const int nxy = g.nx * g.ny;
    TilePull t;
    t.x[0] = c.x == 0 ? g.nx - 1 : c.x - 1;
    t.x[1] = c.x;
    t.x[2] = c.x == g.nx - 1 ? 0 : c.x + 1;
    t.row[0] = c.row == 0 ? nxy - g.nx : c.row - g.nx;
    t.row[1] = c.row;
    t.row[2] = c.row == nxy - g.nx ? 0 : c.row + g.nx;
    for (int k = 0; k < 3; ++k) t.plane[k] = tile_wrap(p - 1 + k, g.nz) * nxy;
    return t;
}

// The source cells of a tile, plane by plane, found a plane ahead so that phase A does not wait for
// the lists: while plane p is stepped, prepare(p + 1) writes the special-cell index of each source
// cell of plane p + 1 into the slot of its extended position and touches its record; the barrier at
// the end of plane p orders that before take(p + 1) reads and empties the slot of this thread's own
// cell. Where each plane's entries start is kept in shared memory for the whole chunk, so a plane
// without source cells costs one look at those bounds.
constexpr int kTileMaxChunk = 254;

template <class Shape>
struct TileSources {
    struct Shared {
        int2 bounds[kTileMaxChunk + 2];  // entries of planes z0 - 1 .. z1
        int slots[2][Shape::kCells];
    };
    Shared* sh;
    const int2* entries;
    const SpecialCell* first;
    int p0;  // z0 - 1

    // A plane's entries have distinct positions, so one per thread is enough.
    __device__ __forceinline__ void prepare(int p) const {
        const int2 b = sh->bounds[p - p0];
        if (b.x + (int)threadIdx.x < b.y) {
            const int2 e = entries[b.x + threadIdx.x];
            sh->slots[p & 1][e.y] = e.x;
            prefetch_l1(first + e.x);
        }
    }
    __device__ __forceinline__ int take(int p) const {
        const int2 b = sh->bounds[p - p0];
        if (b.y <= b.x) return -1;
        int* s = &sh->slots[p & 1][threadIdx.x];
        const int m = *s;
        *s = -1;
        return m;
    }
    // The chunk's bounds, empty slots, and plane z0 - 1's entries in them; ends with a barrier of the block.
    __device__ __forceinline__ void start(const TileArgs& T, const TileCell& c, int nz) const {
        const int* off = T.entry_off + (size_t)c.tile * nz;
        for (int k = threadIdx.x; k <= c.z1 - p0; k += Shape::kCells) {
            const int pz = tile_wrap(p0 + k, nz);
            sh->bounds[k] = make_int2(off[pz], off[pz + 1]);
        }
        sh->slots[0][threadIdx.x] = sh->slots[1][threadIdx.x] = -1;
        __syncthreads();
        prepare(p0);
        __syncthreads();
    }
};

// Sources of special cell m (m < 0: none) at the step of `a`: cell_source's sums, in its order, the first
// current entry from the record itself. (Not cell_source's own form: inlined in the MM tiled pass
// it made that 7 % slower, which has its source cells recomputed apart.)
__device__ __forceinline__ CellSource tile_source(const StepArgs& a, int m) {
    CellSource cs;
    cs.J = cs.E = cs.B = make_float3(0.f, 0.f, 0.f);
    cs.imposed = false;
    if (m < 0) return cs;
    const float4* r = reinterpret_cast<const float4*>(a.sv.first + m);
    const float4 first = __ldg(r), rest = __ldg(r + 1);
    const int b = __float_as_int(rest.x), e = __float_as_int(rest.y);
    const uint32_t mask = __float_as_uint(rest.z);
    if (e > b) {
        const float s0 = a.sc.s[__float_as_int(first.w)];
        cs.J = make_float3(__fmaf_rn(first.x, s0, 0.f), __fmaf_rn(first.y, s0, 0.f), __fmaf_rn(first.z, s0, 0.f));
        for (int k = b + 1; k < e; ++k) {
            const float s = a.sc.s[a.sv.entry_src[k]];
            cs.J.x = __fmaf_rn(a.sv.entry_w[3 * k + 0], s, cs.J.x);
            cs.J.y = __fmaf_rn(a.sv.entry_w[3 * k + 1], s, cs.J.y);
            cs.J.z = __fmaf_rn(a.sv.entry_w[3 * k + 2], s, cs.J.z);
        }
    }
    cs.imposed = mask != 0u;
    for (uint32_t left = mask; left; left &= left - 1) {
        const int k = __ffs(left) - 1;
        const float s = a.sc.s[k];
        cs.E.x = __fmaf_rn(a.sc.E0[k][0], s, cs.E.x);
        cs.E.y = __fmaf_rn(a.sc.E0[k][1], s, cs.E.y);
        cs.E.z = __fmaf_rn(a.sc.E0[k][2], s, cs.E.z);
        cs.B.x = __fmaf_rn(a.sc.B0[k][0], s, cs.B.x);
        cs.B.y = __fmaf_rn(a.sc.B0[k][1], s, cs.B.y);
        cs.B.z = __fmaf_rn(a.sc.B0[k][2], s, cs.B.z);
    }
    return cs;
}

// --- source cells of a small lattice's single step -------------------------------------------------
// On a lattice of a few waves of blocks a step is one chain: wait for the predecessor, pull, collide,
// store; a block with source cells then went on to look them up, pull them again and overwrite them,
// which made it the launch's longest. What the sources are does not depend on the predecessor, so
// such a block looks them up before it waits for it, and updates each cell once. Larger lattices keep
// the recomputation at the end (block_source_cells): there the look at the block's offsets would
// come before the loads of every block, not only of those that wait anyway. Measured on GB300 (us per
// step, dipole lattices; recomputation at the end in brackets): MM 32^3 2.7 (4.3), 48^3 4.8 (6.1), 64^3
// (1024 blocks) 11.1 (11.7), 72^3 (1458) 19.5 (19.0); HV 24^3 2.2 (3.6), 32^3 2.7 (3.6), 48^3 4.5
// (5.9), 64^3 7.3 (7.5), 72^3 12.2 (12.2). The line lies between 64^3 and 72^3: 2.5 waves of 3 blocks per SM.
constexpr int kEarlySourceBlocks = 1140;

// Whether block b of a step launch holds source cells; if so, *cs gets the sources of this thread's cell i
// (zero for other cells). Block-uniform; two barriers where it holds some.
__device__ __forceinline__ bool early_source(const StepArgs& a, int b, int i, CellSource* cs) {
    __shared__ int s_of[kBlock];
    if (!a.sv.block_begin) return false;
    const int lo = a.sv.block_begin[b], hi = a.sv.block_begin[b + 1];
    if (hi <= lo) return false;
    s_of[threadIdx.x] = -1;
    __syncthreads();
    if (lo + (int)threadIdx.x < hi)  // at most one source cell per thread of the block
        s_of[a.sv.cell[lo + threadIdx.x] - (i - (int)threadIdx.x)] = lo + threadIdx.x;
    __syncthreads();
    *cs = tile_source(a, s_of[threadIdx.x]);
    return true;
}

// --- many steps per launch on line lattices (nx = ny = 1) ----------------------------------------
constexpr int kLineThreads = 128;    // cells of a block, halo included
constexpr int kLineScalars = 512;    // source values of a launch: steps x sources
struct LineArgs {
    StepArgs a;    // buffers, media, source cells and imposed vectors (a.sc.s is not used)
    int steps;     // time steps of the launch = halo cells on either side
    int core;      // cells a block owns: at most kLineThreads - 2 steps
    int n_src;
    float s[kLineScalars];  // value of source k at step j: s[j * n_src + k]
};

// --- host-side launchers (one set per model) -----------------------------------------------
// Each returns the number of kernels it enqueued (errors are read with cudaGetLastError).
int mm_launch_step(const StepArgs& a, cudaStream_t st);
int mm_launch_init(const StepArgs& a, const float* E, const float* B, cudaStream_t st);
int mm_launch_fields(const StepArgs& a, FieldsOut out, cudaStream_t st);
int mm_launch_get(const StepArgs& a, float* out, cudaStream_t st);
int mm_launch_set(const StepArgs& a, const float* in, cudaStream_t st);
int mm_launch_reduce(const StepArgs& a, double* partials, int n_blocks, double* result, cudaStream_t st);

int hv_launch_step(const StepArgs& a, cudaStream_t st);
int hv_launch_init(const StepArgs& a, const float* E, const float* B, cudaStream_t st);
int hv_launch_fields(const StepArgs& a, FieldsOut out, cudaStream_t st);
int hv_launch_get(const StepArgs& a, float* out, cudaStream_t st);
int hv_launch_set(const StepArgs& a, const float* in, cudaStream_t st);
int hv_launch_reduce(const StepArgs& a, double* partials, int n_blocks, double* result, cudaStream_t st);

int launch_line(bool mm, const LineArgs& L, cudaStream_t st);

// Deterministic double reduction of per-block partial sums (3 values per block, fixed order).
int launch_reduce_partials(const double* partials, int n_blocks, double* result, cudaStream_t st);
// Deterministic sum of v[0..count) into result[0] (one block, fixed order; result[1], [2] are 0).
int launch_sum_doubles(const double* v, int count, double* result, cudaStream_t st);

// Up to 8 independent device-to-device copies in one launch (sizes and addresses multiples of 4 B).
struct HaloChunk {
    const char* src;
    char* dst;
    long long bytes;
    int width;  // set by launch_halo_copy
};
struct HaloCopy {
    HaloChunk c[8];
    int count;
};
int launch_halo_copy(HaloCopy h, cudaStream_t st);
// Directions whose velocity has z component vz_sign (+1 or -1); returns their number.
int mm_halo_dirs(int vz_sign, int* dirs);
int hv_halo_dirs(int vz_sign, int* dirs);

// Batched step j: main launch over the first n_tiles tiles, source-cell launch over the first
// n_stiles special tiles. Returns the number of kernels enqueued.
int mm_launch_batch_step(const BatchLaunch& b, int j, int n_tiles, int n_stiles, cudaStream_t st);
int hv_launch_batch_step(const BatchLaunch& b, int j, int n_tiles, int n_stiles, cudaStream_t st);
// Resident blocks per SM of the main batched kernel for this configuration.
int mm_batch_occupancy(int storage, int block, bool rho);
int hv_batch_occupancy(int storage, int block);

// Adjoint launches (FP32 storage). adjoint: main launch over every cell not in special_mask, then
// the source cells. terminal: nu^T over the loss plane (nu_out must be zeroed first), and the
// first term of loss_plane. record_step: a forward step that also writes the adjoint record of
// every cell into a.rec.
int mm_launch_record_step(const StepArgs& a, cudaStream_t st);
// Two steps in one pass: aA is step t (fin = the current buffer), aB step t + 1 (fout = the other
// buffer); F describes the ring and the counters (zeroed by the caller). Returns launches.
int mm_launch_fused2(const StepArgs& aA, const StepArgs& aB, const FusedArgs& F, cudaStream_t st);
int hv_launch_fused2(const StepArgs& aA, const StepArgs& aB, const FusedArgs& F, cudaStream_t st);
// Resident blocks per SM of the two-step kernel.
int mm_fused2_occupancy(int storage, int media_mode);
int hv_fused2_occupancy(int storage, int media_mode);
// Two steps in one pass over shared-memory tiles: aA is step t, aB step t + 1; T the tiling. Returns
// launches. _occupancy: resident blocks per SM (0: the device refuses the pass).
int mm_launch_tile2(const StepArgs& aA, const StepArgs& aB, const TileArgs& T, cudaStream_t st);
int hv_launch_tile2(const StepArgs& aA, const StepArgs& aB, const TileArgs& T, cudaStream_t st);
int mm_tile2_occupancy(int storage, int media_mode);
int hv_tile2_occupancy(int storage, int media_mode);
// The MM tiled pass that also writes both steps' adjoint records (aA.rec, aB.rec; FP32 storage only,
// else 0 launches).
int mm_launch_record_tile2(const StepArgs& aA, const StepArgs& aB, const TileArgs& T, cudaStream_t st);
int hv_launch_record_step(const StepArgs& a, cudaStream_t st);
int mm_launch_adjoint(const AdjointArgs& A, cudaStream_t st);
int mm_launch_adjoint_terminal(const AdjointArgs& A, int n_plane, cudaStream_t st);
int hv_launch_adjoint(const AdjointArgs& A, cudaStream_t st);
int hv_launch_adjoint_terminal(const AdjointArgs& A, int n_plane, cudaStream_t st);

}  // namespace lbm
