// Shared device/host helpers of the DDA CUDA library (sm_103a).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

#include "../../include/dda.h"
#include "df.cuh"

namespace dda {

// ------------------------------------------------------------ complex types
// complex128, complex64 and complex double-float (df.cuh)
template <typename T> struct cpx;
template <> struct cpx<double> { using t = double2; };
template <> struct cpx<float> { using t = float2; };
template <> struct cpx<DF> { using t = cdf; };
template <typename T> using C = typename cpx<T>::t;
// element type of the vectors a product of element type T reads and writes
// (the double-float product reads and writes complex128 vectors)
template <typename T> struct io_of { using t = T; };
template <> struct io_of<DF> { using t = double; };
template <typename T> using IO = typename io_of<T>::t;
template <typename T> __device__ __forceinline__ C<T> from_io(C<IO<T>> v) { return v; }
template <> __device__ __forceinline__ cdf from_io<DF>(double2 v) { return make_cdf(df_split(v.x), df_split(v.y)); }
template <typename T> __device__ __forceinline__ C<IO<T>> to_io(C<T> v) { return v; }
template <> __device__ __forceinline__ double2 to_io<DF>(cdf v) {
    return make_double2(df_widen(v.h.x) + df_widen(v.l.x), df_widen(v.h.y) + df_widen(v.l.y));
}
// read-only cached load of one complex value
template <typename T> __device__ __forceinline__ C<T> ldg_c(const C<T>* p) { return __ldg(p); }
template <> __device__ __forceinline__ cdf ldg_c<DF>(const cdf* p) {
    const float4 f = __ldg(reinterpret_cast<const float4*>(p));
    return cdf{make_float2(f.x, f.y), make_float2(f.z, f.w)};
}

template <typename T> __host__ __device__ __forceinline__ C<T> mk(T re, T im) { C<T> z; z.x = re; z.y = im; return z; }
template <typename T> __device__ __forceinline__ C<T> cadd(C<T> a, C<T> b) { return mk<T>(a.x + b.x, a.y + b.y); }
template <typename T> __device__ __forceinline__ C<T> csub(C<T> a, C<T> b) { return mk<T>(a.x - b.x, a.y - b.y); }
template <typename T> __device__ __forceinline__ C<T> cmul(C<T> a, C<T> b) {
    return mk<T>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
template <typename T> __device__ __forceinline__ C<T> cmulc(C<T> a, C<T> b) {
    return mk<T>(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
template <typename T> __device__ __forceinline__ C<T> cscale(C<T> a, T s) { return mk<T>(a.x * s, a.y * s); }
template <typename T> __device__ __forceinline__ C<T> cneg(C<T> a) { return mk<T>(-a.x, -a.y); }
template <typename T> __device__ __forceinline__ C<T> cconj(C<T> a) { return mk<T>(a.x, -a.y); }
// acc += a * b
template <typename T> __device__ __forceinline__ C<T> cfma(C<T> a, C<T> b, C<T> acc) {
    return mk<T>(fma(a.x, b.x, fma(-a.y, b.y, acc.x)), fma(a.x, b.y, fma(a.y, b.x, acc.y)));
}
// a x + b y + c z
template <typename T> __device__ __forceinline__ C<T> cdot3(C<T> a, C<T> x, C<T> b, C<T> y, C<T> c, C<T> z) {
    return cfma<T>(c, z, cfma<T>(b, y, cmul<T>(a, x)));
}
// the double-float forms (pairs of high and low parts, df.cuh)
template <> __host__ __device__ __forceinline__ cdf mk<DF>(DF re, DF im) { return make_cdf(re, im); }
template <> __device__ __forceinline__ cdf cadd<DF>(cdf a, cdf b) { return df_add(a, b); }
template <> __device__ __forceinline__ cdf csub<DF>(cdf a, cdf b) { return df_sub(a, b); }
template <> __device__ __forceinline__ cdf cmul<DF>(cdf a, cdf b) { return df_cmul(a, b); }
template <> __device__ __forceinline__ cdf cscale<DF>(cdf a, DF s) { return df_cscale(a, s); }
template <> __device__ __forceinline__ cdf cneg<DF>(cdf a) {
    return cdf{make_float2(-a.h.x, -a.h.y), make_float2(-a.l.x, -a.l.y)};
}
template <> __device__ __forceinline__ cdf cconj<DF>(cdf a) {
    return cdf{make_float2(a.h.x, -a.h.y), make_float2(a.l.x, -a.l.y)};
}
template <> __device__ __forceinline__ cdf cfma<DF>(cdf a, cdf b, cdf acc) { return df_cfma(a, b, acc); }

// --------------------------------------------------------------- limits
constexpr int kTwEntries = 3072 + 5120;   // twiddle tables exp(-2 pi i m / 3072) and exp(-2 pi i m / 5120)
constexpr int kMaxEdge = 512;

// ------------------------------------------------------- error reporting
void set_error(const std::string& msg);
int fail(int status, const std::string& msg);
int cuda_fail(cudaError_t e, const char* what);

#define DDA_CUDA_TRY(expr)                                         \
    do {                                                           \
        cudaError_t e__ = (expr);                                  \
        if (e__ != cudaSuccess) return ::dda::cuda_fail(e__, #expr); \
    } while (0)

void note_launches(int64_t n);

// true for device or managed memory of any device; false for host memory,
// stale or foreign pointers (checked on the host before any launch)
bool is_device_ptr(const void* p);

// after every kernel launch: count it and turn a launch error into a status
#define DDA_LAUNCH_CHECK(what)                                           \
    do {                                                                 \
        ::dda::note_launches(1);                                         \
        cudaError_t e__ = cudaGetLastError();                            \
        if (e__ != cudaSuccess) return ::dda::cuda_fail(e__, what);      \
    } while (0)

// Dependent launches: a kernel launched with launch_after(ahead = true) may be
// scheduled as soon as the blocks of the kernel before it in the stream have
// ended, so that its launch overlaps the completion of that kernel.  Such a
// kernel calls grid_wait in every thread before it touches memory that an
// earlier kernel writes or reads: it waits until all earlier kernels have
// completed and their writes are visible.  It must not return without that
// wait: its completion stands for that of its predecessors.  The wait orders
// ordinary loads and stores; read-only loads (__ldg, const __restrict__
// parameters) assume memory that nothing writes while the kernel is resident,
// which may start before the wait ends.  So what earlier kernels write
// (vectors, work arrays, status words) is read with ordinary loads, and only a
// context's tables, bit fields, ranks and spectrum, complete before its first
// product, with read-only ones.
// No kernel lets its successor start earlier than that
// (griddepcontrol.launch_dependents).  Called at the start, several later
// kernels pile up on the SMs that have room and their blocks are spread
// unevenly (complex64 24 x 40 x 40 took 40 us that way, 34 with ordinary
// launches, 20.7 this way; complex128 32^3 203 us that way, 138 with ordinary
// launches).  Called before the final stores, it changed the compiler's
// schedule of them (x pass of 192-point rows, four of 95 x 94 x 105: 102 -> 122
// us).  In an ordinary launch the wait is skipped: with many short blocks it
// alone made passes up to 1.9 times as long.
__device__ __forceinline__ void grid_wait(int ahead) {
    if (ahead) asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <typename... P, typename... A>
inline cudaError_t launch_after(bool ahead, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                A&&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = ahead ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }

// -------------------------------------------------------- lattice geometry
struct Geometry {
    int K, J, P;          // lattice edges (x, y, z)
    int Lx, Ly, Lz;       // padded DFT lengths (padded_length)
    int Hx, Hy, Hz;       // stored half-spectrum extents L/2 + 1
    int Pb;               // pitch of the z columns of the xy-transformed volume (>= P)
    int64_t nsites;       // K J P
    int64_t nwords;       // occupancy words
    int64_t nd;           // occupied sites
    int nmat;             // materials
    int cbits;            // composition bits per field
    int cfields;          // fields per word
};

// lines of 3 * 2^a and 5 * 2^a points (the other supported lengths are 2^a)
__host__ __device__ constexpr bool wide_len(int N) { return N % 3 == 0 || N % 5 == 0; }

// Element of the half spectrum (my, mx, mz, component q): columns
// [Hy][Hx], every z line contiguous.  For z lines of 2^a points the six
// components of a point sit side by side ([Hz][6]: one 48-byte record per
// point, read whole by the z-pass thread that holds all three components);
// for 3 * 2^a and 5 * 2^a points, whose z pass gives each component its own
// threads, each component's line is contiguous ([6][Hz]).
__host__ __device__ __forceinline__ int64_t spec_index(const Geometry& g, int my, int mx, int mz, int q) {
    const int64_t col = ((int64_t)my * g.Hx + mx) * 6 * g.Hz;
    return col + (wide_len(g.Lz) ? (int64_t)q * g.Hz + mz : (int64_t)mz * 6 + q);
}

// circulant length of an n-point Toeplitz level: the smallest L >= 2n - 1
// (and >= 2) of the form 2^a, 3 * 2^a or 5 * 2^a (a >= 3 for the last two;
// Sec. 3: K'' = 2K - 1 + kf with kf chosen for a fast DFT)
inline int padded_length(int n) {
    const int need = 2 * n - 1 > 2 ? 2 * n - 1 : 2;
    int best = 0;
    for (int start : {2, 24, 40}) {
        int L = start;
        while (L < need) L *= 2;
        if (!best || L < best) best = L;
    }
    return best;
}
// Column pitch of the xy-transformed volume: P rounded up to a multiple of
// 8 elements, and to an odd multiple of 8 (so that the columns, read and
// written 64 or 128 bytes at a time across x by the x passes, do not start
// at a power-of-two stride)
inline int column_pitch(int P) {
    int p = (P + 7) / 8 * 8;
    if ((p / 8) % 2 == 0) p += 8;
    return p;
}
inline int ilog2(int n) { int l = 0; while ((1 << l) < n) ++l; return l; }

// device view of the target for the expand / compress kernels
struct TargetView {
    const uint32_t* occ;     // occupancy words
    const uint32_t* rank;    // exclusive prefix count per word
    const uint32_t* comp;    // composition words or nullptr
    int cbits, cfields;
};

__device__ __forceinline__ bool occupied(const TargetView& t, int64_t s) {
    return (__ldg(t.occ + (s >> 5)) >> (s & 31)) & 1u;
}
__device__ __forceinline__ uint32_t site_rank(const TargetView& t, int64_t s) {
    const uint32_t w = __ldg(t.occ + (s >> 5));
    return __ldg(t.rank + (s >> 5)) + __popc(w & ((1u << (s & 31)) - 1u));
}
__device__ __forceinline__ int material(const TargetView& t, int64_t s, int axis) {
    if (t.comp == nullptr) return 0;
    const int64_t q = 3 * s + axis;
    const uint32_t w = __ldg(t.comp + q / t.cfields);
    return (w >> ((q % t.cfields) * t.cbits)) & ((1u << t.cbits) - 1u);
}

}  // namespace dda
