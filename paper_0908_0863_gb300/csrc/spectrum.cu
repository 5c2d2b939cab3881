// Green's-tensor spectrum of the level-three Toeplitz interaction matrix
// (OpenDDA Sec. 3, App. A, Table 1), built once per target in FP64.
//
// Section 1 of the embedding holds the six independent components
// t_m(i, j, k), m = xx, xy, xz, yy, yz, zz, of the interaction tensor at
// displacements 0 <= i < K, 0 <= j < J, 0 <= k < P (t = 0 at the origin, the
// diagonal being added in the matvec).  The Toeplitz-to-circulant conversion
// and the DFT are fused line by line: every line of n values is extended to
// length L by mirroring entries 1..n-1 to L-1..L-n+1 with the Table-1 sign
// of that axis (zeros in between), transformed, and only the first L/2 + 1
// outputs are kept -- first along x, then y, then z, so each later pass
// works on the already reduced array.  The stored half spectrum is scaled by
// 1/(Lx Ly Lz) (the iDFT normalisation of Sec. 3 step 4) and copied to
// complex64 and double-float form for the mixed-precision matvec.
//
// A mirrored line is even or odd (Table 1), and so is its transform.  An
// even line a and an odd one b of two components therefore share one
// transform: with X the DFT of a + b, the DFT of a is (X[k] + X[L-k]) / 2 and
// that of b (X[k] - X[L-k]) / 2.  On each axis two components are odd and
// four even, so the six take four transforms (this step is bound by the FP64
// units).  The halvings are left to the final scale: with the yz component
// doubled at the start, the two components of every pair carry the same power
// of two, so that neither adds more than its share to the other's rounding.
#include "fft.cuh"
#include "matvec.cuh"
#include "spectrum.cuh"

namespace dda {

namespace {

// Components transformed together on an axis: job q takes the even component
// pair_even and, where there is one, the odd component pair_odd (else -1)
__device__ __forceinline__ int pair_even(int axis, int q) {
    constexpr int e[3][4] = {{0, 3, 4, 5}, {0, 2, 3, 5}, {0, 1, 3, 5}};
    return e[axis][q];
}
__device__ __forceinline__ int pair_odd(int axis, int q) {
    constexpr int o[3][4] = {{1, 2, -1, -1}, {1, 4, -1, -1}, {2, 4, -1, -1}};
    return o[axis][q];
}
// power of two a component carries through the pairings (the yz component's
// starting 2 included), as its reciprocal
__device__ __forceinline__ double pair_unscale(int m) {
    constexpr double u[6] = {0.125, 0.125, 0.125, 0.5, 0.125, 1.0};
    return u[m];
}

// t_m at r = (i, j, k) != 0 (the yz component doubled):
//   exp(ikr)/r^3 [ k^2 (r_a r_b - r^2 d_ab) + (ikr - 1)/r^2 (3 r_a r_b - r^2 d_ab) ]
__global__ void k_section1(Geometry g, double kw, double2* __restrict__ t1) {
    const int64_t n = g.nsites;
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(s % g.K);
        const int j = (int)((s / g.K) % g.J);
        const int k = (int)(s / ((int64_t)g.K * g.J));
        const double x = i, y = j, z = k;
        const double r2 = x * x + y * y + z * z;
        double2 out[6];
        if (r2 == 0.0) {
            for (int m = 0; m < 6; ++m) out[m] = make_double2(0.0, 0.0);
        } else {
            const double r = sqrt(r2);
            double sn, cs;
            sincos(kw * r, &sn, &cs);
            const double inv_r3 = 1.0 / (r2 * r);
            const double2 e = make_double2(cs * inv_r3, sn * inv_r3);           // exp(ikr)/r^3
            const double2 f = make_double2(-1.0 / r2, kw * r / r2);             // (ikr - 1)/r^2
            const double rr[6] = {x * x, x * y, x * z, y * y, y * z, z * z};
            const int diag[6] = {1, 0, 0, 1, 0, 1};
            for (int m = 0; m < 6; ++m) {
                const double d = diag[m] ? r2 : 0.0;
                const double a = kw * kw * (rr[m] - d);
                const double b = 3.0 * rr[m] - d;
                const double2 inner = make_double2(a + f.x * b, f.y * b);
                out[m] = make_double2(e.x * inner.x - e.y * inner.y, e.x * inner.y + e.y * inner.x);
            }
        }
        out[4].x *= 2.0;
        out[4].y *= 2.0;
        for (int m = 0; m < 6; ++m) t1[m * n + s] = out[m];
    }
}

constexpr int kV = 8;

// point n of a mirrored line, or of a pair of them: src(i) is entry i < nline
// of the even line, src2(i) of the odd one
template <typename Src, typename Src2>
__device__ __forceinline__ double2 mirrored(int n, int nline, int N, bool pair, Src src, Src2 src2) {
    if (n < nline) {
        double2 v = src(n);
        if (pair) { const double2 o = src2(n); v.x += o.x; v.y += o.y; }
        return v;
    }
    if (n > N - nline) {
        double2 v = src(N - n);
        if (pair) { const double2 o = src2(N - n); v.x -= o.x; v.y -= o.y; }
        return v;
    }
    return make_double2(0.0, 0.0);
}

// x lines: rows of K values (t1 [6][P][J][K]) -> rows of Hx ([6][P][J][Hx]); grid (row tiles, 4 jobs)
__global__ void __launch_bounds__(512) k_tensor_x(Geometry g, int logW, const double2* __restrict__ tw,
                                                  const double2* __restrict__ in, double2* __restrict__ out) {
    extern __shared__ unsigned char smem_raw[];
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    const int W = 1 << logW, ld = W + 1, N = g.Lx;
    const int64_t rows = (int64_t)g.P * g.J, r0 = (int64_t)blockIdx.x * W;
    const int me = pair_even(0, blockIdx.y), mo = pair_odd(0, blockIdx.y);
    for (int e = threadIdx.x; e < W * N; e += blockDim.x) {
        const int w = e / N, n = e - w * N;
        const int64_t row = r0 + w;
        double2 v = make_double2(0.0, 0.0);
        if (row < rows) {
            const double2 *a = in + (me * rows + row) * g.K, *b = in + (mo * rows + row) * g.K;
            v = mirrored(n, g.K, N, mo >= 0, [&](int i) { return a[i]; }, [&](int i) { return b[i]; });
        }
        buf[n * ld + w] = v;
    }
    __syncthreads();
    fft_tile<double, kV, false>(buf, ld, logW, N, tw);
    for (int e = threadIdx.x; e < W * g.Hx; e += blockDim.x) {
        const int w = e / g.Hx, n = e - w * g.Hx;
        const int64_t row = r0 + w;
        if (row >= rows) continue;
        const double2 x = buf[n * ld + w];
        double2* oe = out + (me * rows + row) * g.Hx + n;
        if (mo < 0) {
            *oe = x;
        } else {
            const double2 y = buf[(n ? N - n : 0) * ld + w];
            *oe = make_double2(x.x + y.x, x.y + y.y);
            out[(mo * rows + row) * g.Hx + n] = make_double2(x.x - y.x, x.y - y.y);
        }
    }
}

// strided lines along y (axis 1) or z (axis 2) on arrays whose rows are Hx
// long.  in: [6][n_outer][n_line][Hx] slices -> out: [6][n_outer][H][Hx]
// (y pass: outer = P, line = J -> Hy; z pass: the line is the outermost
// index of [6][P][Hy][Hx] -> the z-line layout of spec_index, scaled, with
// the complex64 and double-float copies).  Grid (x tiles, outer, 4 jobs).
template <int AXIS>
__global__ void __launch_bounds__(512) k_tensor_col(Geometry g, int logW, const double2* __restrict__ tw,
                                                    const double2* __restrict__ in, double2* __restrict__ out,
                                                    double scale, float2* __restrict__ out32, cdf* __restrict__ outdf) {
    extern __shared__ unsigned char smem_raw[];
    double2* buf = reinterpret_cast<double2*>(smem_raw);
    const int W = 1 << logW, ld = W + 1;
    const int N = AXIS == 1 ? g.Ly : g.Lz;
    const int nline = AXIS == 1 ? g.J : g.P;
    const int H = AXIS == 1 ? g.Hy : g.Hz;
    const int x0 = blockIdx.x * W;
    const int outer = blockIdx.y;   // y pass: z plane k; z pass: row my
    const int me = pair_even(AXIS, blockIdx.z), mo = pair_odd(AXIS, blockIdx.z);
    // first element of component m's line at x = 0, and the step along it
    auto in_base = [&](int m) -> int64_t {
        return AXIS == 1 ? (((int64_t)m * g.P + outer) * g.J) * g.Hx : ((int64_t)m * g.P * g.Hy + outer) * g.Hx;
    };
    const int64_t in_step = AXIS == 1 ? g.Hx : (int64_t)g.Hy * g.Hx;
    const double2 *a = in + in_base(me), *b = in + in_base(mo >= 0 ? mo : me);
    for (int e = threadIdx.x; e < W * N; e += blockDim.x) {
        const int n = e >> logW, w = e & (W - 1), x = x0 + w;
        double2 v = make_double2(0.0, 0.0);
        if (x < g.Hx)
            v = mirrored(n, nline, N, mo >= 0, [&](int i) { return a[i * in_step + x]; },
                         [&](int i) { return b[i * in_step + x]; });
        buf[n * ld + w] = v;
    }
    __syncthreads();
    fft_tile<double, kV, false>(buf, ld, logW, N, tw);
    auto store = [&](int m, int n, int x, double2 v) {
        if (AXIS == 1) {
            out[(((int64_t)m * g.P + outer) * g.Hy + n) * g.Hx + x] = v;
        } else {
            // final spectrum: every z line contiguous (spec_index), so the z
            // pass reads a column's line in one stream
            const double f = scale * pair_unscale(m);
            v.x *= f;
            v.y *= f;
            const int64_t o = spec_index(g, outer, x, n, m);
            out[o] = v;
            const cdf d = from_io<DF>(v);
            outdf[o] = d;
            out32[o] = d.h;   // the nearest floats
        }
    };
    for (int e = threadIdx.x; e < W * H; e += blockDim.x) {
        const int n = e >> logW, w = e & (W - 1), x = x0 + w;
        if (x >= g.Hx) continue;
        const double2 p = buf[n * ld + w];
        if (mo < 0) {
            store(me, n, x, p);
        } else {
            const double2 q = buf[(n ? N - n : 0) * ld + w];
            store(me, n, x, make_double2(p.x + q.x, p.y + q.y));
            store(mo, n, x, make_double2(p.x - q.x, p.y - q.y));
        }
    }
}

int pick_logW_rows(int N) {   // rows of length N, V = 8 values per thread, <= 512 threads
    int logW = 0;
    while ((1 << logW) * 16 < 128 && (2 << logW) * N / kV <= 512) ++logW;
    while ((1 << logW) * N < kV) ++logW;
    return logW;
}

int pick_logW_cols(int N, int ncols) {
    int logW = 0;
    while ((1 << logW) * 16 < 128 && (2 << logW) * N / kV <= 512) ++logW;
    while (logW > 0 && (1 << (logW - 1)) >= ncols) --logW;
    while ((1 << logW) * N < kV) ++logW;
    return logW;
}

int smem_attr(const void* fn, size_t bytes) {
    if (bytes > 48 * 1024)
        DDA_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    return 0;
}

}  // namespace

size_t spectrum_scratch_elems(const Geometry& g) {
    const size_t a = 6ull * g.P * g.J * g.K;
    const size_t b = 6ull * g.P * g.J * g.Hx;
    const size_t c = 6ull * g.P * g.Hy * g.Hx;
    return std::max(a, std::max(b, c));
}

int build_spectrum(const Geometry& g, double k, const double2* tw, double2* s0, double2* s1,
                   double2* spec64, float2* spec32, cdf* specdf, cudaStream_t st) {
    int rc;
    // section 1
    {
        const int threads = 256;
        const int64_t blocks = std::min<int64_t>((g.nsites + threads - 1) / threads, 152 * 64);
        k_section1<<<(unsigned)blocks, threads, 0, st>>>(g, k, s0);
        DDA_LAUNCH_CHECK("tensor section 1");
    }
    // x lines
    {
        const int logW = pick_logW_rows(g.Lx), W = 1 << logW;
        const size_t sm = (size_t)g.Lx * (W + 1) * sizeof(double2);
        if ((rc = smem_attr((const void*)k_tensor_x, sm))) return rc;
        const int64_t rows = (int64_t)g.P * g.J;
        k_tensor_x<<<dim3((unsigned)((rows + W - 1) / W), 4), W * g.Lx / kV, sm, st>>>(g, logW, tw, s0, s1);
        DDA_LAUNCH_CHECK("tensor x DFT");
    }
    // y lines
    {
        const int logW = pick_logW_cols(g.Ly, g.Hx), W = 1 << logW;
        const size_t sm = (size_t)g.Ly * (W + 1) * sizeof(double2);
        if ((rc = smem_attr((const void*)k_tensor_col<1>, sm))) return rc;
        dim3 grid((g.Hx + W - 1) / W, g.P, 4);
        k_tensor_col<1><<<grid, W * g.Ly / kV, sm, st>>>(g, logW, tw, s1, s0, 1.0, nullptr, nullptr);
        DDA_LAUNCH_CHECK("tensor y DFT");
    }
    // z lines, scaled, with the complex64 and double-float copies
    {
        const int logW = pick_logW_cols(g.Lz, g.Hx), W = 1 << logW;
        const size_t sm = (size_t)g.Lz * (W + 1) * sizeof(double2);
        if ((rc = smem_attr((const void*)k_tensor_col<2>, sm))) return rc;
        dim3 grid((g.Hx + W - 1) / W, g.Hy, 4);
        const double scale = 1.0 / ((double)g.Lx * g.Ly * g.Lz);
        k_tensor_col<2><<<grid, W * g.Lz / kV, sm, st>>>(g, logW, tw, s0, spec64, scale, spec32, specdf);
        DDA_LAUNCH_CHECK("tensor z DFT");
    }
    return 0;
}

// the spectrum in the exported order [Hy][Hx][Hz][6] from the stored one
template <typename T>
__global__ void __launch_bounds__(256) k_spec_export(Geometry g, const C<T>* __restrict__ in, C<T>* __restrict__ out) {
    const int64_t n = 6LL * g.Hz * g.Hy * g.Hx;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
        const int q = (int)(e % 6);
        const int64_t r = e / 6;
        const int mz = (int)(r % g.Hz);
        const int64_t col = r / g.Hz;
        out[e] = in[spec_index(g, (int)(col / g.Hx), (int)(col % g.Hx), mz, q)];
    }
}

int export_spectrum(const Geometry& g, const void* in, void* out, bool c128, cudaStream_t st) {
    const size_t ns = 6ull * g.Hz * g.Hy * g.Hx;
    if (!wide_len(g.Lz)) {   // stored in the exported order
        DDA_CUDA_TRY(cudaMemcpyAsync(out, in, ns * (c128 ? sizeof(double2) : sizeof(float2)),
                                     cudaMemcpyDeviceToDevice, st));
        return 0;
    }
    const unsigned blocks = (unsigned)std::min<size_t>((ns + 255) / 256, 152 * 16);
    if (c128) k_spec_export<double><<<blocks, 256, 0, st>>>(g, static_cast<const double2*>(in), static_cast<double2*>(out));
    else k_spec_export<float><<<blocks, 256, 0, st>>>(g, static_cast<const float2*>(in), static_cast<float2*>(out));
    DDA_LAUNCH_CHECK("spectrum export");
    return 0;
}

}  // namespace dda
