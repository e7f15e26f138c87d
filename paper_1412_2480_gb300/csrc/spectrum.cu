// spectrum.cu -- Fourier diagnostics of a grid quantity (the k-space maps of B_z in
// Sec. 3.1, Fig. 3): the 2D discrete Fourier transform
//   F^(p, q) = sum_{l, m} F(l, m) exp(-2 pi i (p l / nx + q m / ny)),
// returned as the amplitude |F^(p, q)| / (nx ny) in the fields' (ny, nx) layout, p and q
// in FFT order (index p >= nx/2 is the wave number 2 pi (p - nx) / (nx dx)).
//
// Each 1D transform runs in one CTA on shared memory as a Stockham autosort FFT
// (Stockham 1966; the per-stage indexing of Govindaraju et al., SC 2008): stage s with
// radix R combines R sub-transforms of length Ns into one of length Ns R; thread work
// item j reads x[j + t N/R] (t < R), multiplies by exp(-2 pi i t (j mod Ns) / (Ns R)),
// takes the R-point DFT and writes x'[(j / Ns) Ns R + (j mod Ns) + t Ns]. Lengths of the
// form 2^a 3^b 5^c up to kMaxN use radices 4, 2, 3, 5; other lengths fall back to the
// direct O(N^2) sum. Arithmetic is FP64 throughout.
//
// What bounds it is the FP64 pipe (two lanes per cycle and SM here), so the work is cut
// where the result allows it: twiddles come from a table of the N-th roots of unity made
// once per call (a sincospi per element was three quarters of the operations); the field
// is real, so only the columns p <= nx/2 are transformed and the others' amplitudes are
// |F^(nx - p, ny - q)|; the direct sums fold index l with N - l, and take several rows
// (columns) per root. 1024 x 256: 328 -> 69 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <string>

#include "engine.h"
#include "mixed.h"
#include "pic.h"

namespace pic {

namespace {

constexpr int kMaxN = 8192;  // 128 KB of complex FP64 in shared memory
constexpr int kMaxStages = 16;

struct Plan {
    int n;
    int nst;
    int radix[kMaxStages];
    bool direct;  // not of the form 2^a 3^b 5^c (or longer than kMaxN): O(N^2) sum
};

Plan make_plan(int n) {
    Plan p{};
    p.n = n;
    int m = n;
    while (m % 4 == 0 && p.nst < kMaxStages) { p.radix[p.nst++] = 4; m /= 4; }
    while (m % 2 == 0 && p.nst < kMaxStages) { p.radix[p.nst++] = 2; m /= 2; }
    while (m % 3 == 0 && p.nst < kMaxStages) { p.radix[p.nst++] = 3; m /= 3; }
    while (m % 5 == 0 && p.nst < kMaxStages) { p.radix[p.nst++] = 5; m /= 5; }
    p.direct = m != 1 || n > kMaxN;
    return p;
}

__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
    return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// tw[k] = exp(-2 pi i k / n) for both lengths.
__global__ void k_roots(int nx, double2* __restrict__ twx, int ny, double2* __restrict__ twy) {
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    double s, c;
    if (k < nx) {
        sincospi(-2.0 * (double)k / (double)nx, &s, &c);
        twx[k] = make_double2(c, s);
    }
    if (k < ny) {
        sincospi(-2.0 * (double)k / (double)ny, &s, &c);
        twy[k] = make_double2(c, s);
    }
}

// In-place R-point forward DFT of v (exp(-2 pi i jk / R)), R = 2, 3, 4, 5; tw: the n-th
// roots, n a multiple of R.
template <int R>
__device__ __forceinline__ void dft_small(double2 v[R], const double2* __restrict__ tw, int n) {
    if (R == 2) {
        const double2 a = v[0], b = v[1];
        v[0] = make_double2(a.x + b.x, a.y + b.y);
        v[1] = make_double2(a.x - b.x, a.y - b.y);
    } else if (R == 4) {
        const double2 a = make_double2(v[0].x + v[2].x, v[0].y + v[2].y);
        const double2 b = make_double2(v[0].x - v[2].x, v[0].y - v[2].y);
        const double2 c = make_double2(v[1].x + v[3].x, v[1].y + v[3].y);
        const double2 d = make_double2(v[1].x - v[3].x, v[1].y - v[3].y);  // times -i below
        v[0] = make_double2(a.x + c.x, a.y + c.y);
        v[2] = make_double2(a.x - c.x, a.y - c.y);
        v[1] = make_double2(b.x + d.y, b.y - d.x);
        v[3] = make_double2(b.x - d.y, b.y + d.x);
    } else {
        // R = 3, 5: direct sums with index j folded on R - j
        constexpr int H = (R - 1) / 2;
        double2 a[H > 0 ? H : 1], b[H > 0 ? H : 1];
        double2 out[R];
        out[0] = v[0];
#pragma unroll
        for (int j = 1; j <= H; j++) {
            a[j - 1] = make_double2(v[j].x + v[R - j].x, v[j].y + v[R - j].y);
            b[j - 1] = make_double2(v[j].x - v[R - j].x, v[j].y - v[R - j].y);
            out[0].x += a[j - 1].x;
            out[0].y += a[j - 1].y;
        }
#pragma unroll
        for (int k = 1; k <= H; k++) {
            double2 e = v[0], o = make_double2(0.0, 0.0);
#pragma unroll
            for (int j = 1; j <= H; j++) {
                double2 w = __ldg(tw + (j * k) % R * (n / R));  // (cos, -sin)
                if (R == 3) w.x = -0.5;  // (a third is no FP64 number, nor then the table's root)
                e.x += a[j - 1].x * w.x;
                e.y += a[j - 1].y * w.x;
                o.x -= b[j - 1].y * w.y;
                o.y += b[j - 1].x * w.y;
            }
            out[k] = make_double2(e.x + o.x, e.y + o.y);
            out[R - k] = make_double2(e.x - o.x, e.y - o.y);
        }
#pragma unroll
        for (int k = 0; k < R; k++) v[k] = out[k];
    }
}

// One Stockham stage of radix R on buf (length n <= NMAX), sub-transform length ns.
template <int R, int T, int NMAX>
__device__ __forceinline__ void stage(double2* buf, int n, int ns, const double2* __restrict__ tw) {
    constexpr int kPer = (NMAX / R + T - 1) / T;  // work items per thread
    const int items = n / R, step = n / (ns * R);
    double2 v[kPer][R];
#pragma unroll
    for (int b = 0; b < kPer; b++) {
        const int j = threadIdx.x + b * T;
        if (j < items) {
            const int jm = j % ns;
#pragma unroll
            for (int t = 0; t < R; t++) {
                double2 x = buf[j + t * items];
                if (t > 0 && jm > 0) x = cmul(x, __ldg(tw + t * jm * step));
                v[b][t] = x;
            }
            dft_small<R>(v[b], tw, n);
        }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < kPer; b++) {
        const int j = threadIdx.x + b * T;
        if (j < items) {
            const int jm = j % ns;
            const int base = (j / ns) * ns * R + jm;
#pragma unroll
            for (int t = 0; t < R; t++) buf[base + t * ns] = v[b][t];
        }
    }
    __syncthreads();
}

template <int T, int NMAX>
__device__ __forceinline__ void fft_smem(double2* buf, const Plan& p, const double2* __restrict__ tw) {
    int ns = 1;
    for (int s = 0; s < p.nst; s++) {
        switch (p.radix[s]) {
        case 4: stage<4, T, NMAX>(buf, p.n, ns, tw); break;
        case 2: stage<2, T, NMAX>(buf, p.n, ns, tw); break;
        case 3: stage<3, T, NMAX>(buf, p.n, ns, tw); break;
        default: stage<5, T, NMAX>(buf, p.n, ns, tw); break;
        }
        ns *= p.radix[s];
    }
}

// The half spectrum of the rows lies column by column: W[p ny + m] = row m's DFT at p, 0 <=
// p <= nx/2, so a column is contiguous.

// A row as the real part of a transform along x. (Two rows as the real and imaginary part of
// one, 93 -> 81 us for 1024 x 256, 872 -> 635 for 8192 x 512, take an addition more per value:
// the spectrum was 4 to 13% further from the exact one than from transforms of real rows.)
template <int T, int NMAX>
__global__ void __launch_bounds__(T, 1) k_fft_rows(const double* __restrict__ F, int nx, int ny, const Plan p,
                                                const double2* __restrict__ tw, double2* __restrict__ W) {
    extern __shared__ double2 sbuf[];
    const int m = blockIdx.x;
    const double* f0 = F + (long long)m * nx;
    for (int l = threadIdx.x; l < nx; l += T) sbuf[l] = make_double2(f0[l], 0.0);
    __syncthreads();
    fft_smem<T, NMAX>(sbuf, p, tw);
    for (int k = threadIdx.x; k <= nx / 2; k += T) W[(long long)k * ny + m] = sbuf[k];
}

// |.| * scale at wave number (p, q) and at its conjugate (nx - p, ny - q).
__device__ __forceinline__ void put_amplitude(double* __restrict__ out, int nx, int ny, int p, int q, double2 z,
                                              double scale) {
    const double v = hypot(z.x, z.y) * scale;
    out[(long long)q * nx + p] = v;
    if (p > 0 && 2 * p != nx) out[(long long)(q == 0 ? 0 : ny - q) * nx + (nx - p)] = v;
}

// Column p of W -> its DFT along y, as amplitudes.
template <int T, int NMAX>
__global__ void __launch_bounds__(T, 1) k_fft_cols(const double2* __restrict__ W, int nx, int ny, const Plan p,
                                                const double2* __restrict__ tw, double scale, double* __restrict__ out) {
    extern __shared__ double2 sbuf[];
    const int col = blockIdx.x;
    for (int m = threadIdx.x; m < ny; m += T) sbuf[m] = W[(long long)col * ny + m];
    __syncthreads();
    fft_smem<T, NMAX>(sbuf, p, tw);
    for (int q = threadIdx.x; q < ny; q += T) put_amplitude(out, nx, ny, col, q, sbuf[q], scale);
}

// Direct sums for lengths with other prime factors, kDftLines rows (columns) per block and
// one wave number per thread: x_0 + sum_l (x_l + x_(n-l)) cos - i (x_l - x_(n-l)) sin over
// 1 <= l < n/2, and (-1)^k x_(n/2) where n is even. The folded values are staged kDftChunk
// at a time.
constexpr int kDftThreads = 128, kDftLines = 4, kDftChunk = 256;

__global__ void __launch_bounds__(kDftThreads) k_dft_rows(const double* __restrict__ F, int nx, int ny,
                                                          const double2* __restrict__ tw, double2* __restrict__ W) {
    __shared__ double sa[kDftChunk][kDftLines], sb[kDftChunk][kDftLines];
    const int k = blockIdx.x * kDftThreads + threadIdx.x, m0 = blockIdx.y * kDftLines;
    const int half = (nx - 1) / 2;  // l = 1 .. half have a partner n - l
    double re[kDftLines] = {0.0, 0.0, 0.0, 0.0}, im[kDftLines] = {0.0, 0.0, 0.0, 0.0};
    int idx = 0;  // k l mod n of the last l
    for (int l0 = 1; l0 <= half; l0 += kDftChunk) {
        const int nl = min(kDftChunk, half + 1 - l0);
        __syncthreads();
        for (int t = threadIdx.x; t < nl * kDftLines; t += kDftThreads) {
            const int r = t / nl, l = l0 + (t - r * nl);
            double x = 0.0, y = 0.0;
            if (m0 + r < ny) {
                x = F[(long long)(m0 + r) * nx + l];
                y = F[(long long)(m0 + r) * nx + nx - l];
            }
            sa[l - l0][r] = x + y;
            sb[l - l0][r] = x - y;
        }
        __syncthreads();
        if (k <= nx / 2)
            for (int t = 0; t < nl; t++) {
                idx += k;
                if (idx >= nx) idx -= nx;
                const double2 w = __ldg(tw + idx);
#pragma unroll
                for (int r = 0; r < kDftLines; r++) {
                    re[r] += sa[t][r] * w.x;
                    im[r] += sb[t][r] * w.y;
                }
            }
    }
    if (k > nx / 2) return;
#pragma unroll
    for (int r = 0; r < kDftLines; r++) {
        if (m0 + r >= ny) continue;
        const double* f = F + (long long)(m0 + r) * nx;
        re[r] += f[0];
        if (nx % 2 == 0) re[r] += (k & 1) ? -f[nx / 2] : f[nx / 2];
        W[(long long)k * ny + m0 + r] = make_double2(re[r], im[r]);
    }
}

// ... and along y: both wave numbers q and ny - q per thread.
constexpr int kDftCols = 2;

__global__ void __launch_bounds__(kDftThreads) k_dft_cols(const double2* __restrict__ W, int nx, int ny,
                                                          const double2* __restrict__ tw, double scale,
                                                          double* __restrict__ out) {
    __shared__ double2 ss[kDftChunk][kDftCols], sd[kDftChunk][kDftCols];
    const int q = blockIdx.x * kDftThreads + threadIdx.x, p0 = blockIdx.y * kDftCols;
    const int half = (ny - 1) / 2, np = nx / 2 + 1;
    double2 e[kDftCols], o[kDftCols];  // sums with cos and with -sin
#pragma unroll
    for (int c = 0; c < kDftCols; c++) e[c] = o[c] = make_double2(0.0, 0.0);
    int idx = 0;
    for (int l0 = 1; l0 <= half; l0 += kDftChunk) {
        const int nl = min(kDftChunk, half + 1 - l0);
        __syncthreads();
        for (int t = threadIdx.x; t < nl * kDftCols; t += kDftThreads) {
            const int c = t / nl, l = l0 + (t - c * nl);
            double2 x = make_double2(0.0, 0.0), y = x;
            if (p0 + c < np) {
                x = W[(long long)(p0 + c) * ny + l];
                y = W[(long long)(p0 + c) * ny + ny - l];
            }
            ss[l - l0][c] = make_double2(x.x + y.x, x.y + y.y);
            sd[l - l0][c] = make_double2(x.x - y.x, x.y - y.y);
        }
        __syncthreads();
        if (q <= ny / 2)
            for (int t = 0; t < nl; t++) {
                idx += q;
                if (idx >= ny) idx -= ny;
                const double2 w = __ldg(tw + idx);
#pragma unroll
                for (int c = 0; c < kDftCols; c++) {
                    e[c].x += ss[t][c].x * w.x;
                    e[c].y += ss[t][c].y * w.x;
                    o[c].x += sd[t][c].x * w.y;
                    o[c].y += sd[t][c].y * w.y;
                }
            }
    }
    if (q > ny / 2) return;
#pragma unroll
    for (int c = 0; c < kDftCols; c++) {
        if (p0 + c >= np) continue;
        const double2* w = W + (long long)(p0 + c) * ny;
        double2 b = w[0];
        if (ny % 2 == 0) {
            const double2 h = w[ny / 2];
            b.x += (q & 1) ? -h.x : h.x;
            b.y += (q & 1) ? -h.y : h.y;
        }
        // i times the sine sum: (-o.y, o.x)
        put_amplitude(out, nx, ny, p0 + c, q, make_double2(b.x + e[c].x - o[c].y, b.y + e[c].y + o[c].x), scale);
        if (q > 0 && 2 * q != ny)
            put_amplitude(out, nx, ny, p0 + c, ny - q, make_double2(b.x + e[c].x + o[c].y, b.y + e[c].y - o[c].x), scale);
    }
}

// Threads of a transform: 256 up to this length (two radix-4 items each), then 1024.
constexpr int kShort = 2048;

}  // namespace

int spectrum_2d(const double* F, int nx, int ny, double* out, cudaStream_t st, std::string& err) {
    const Plan px = make_plan(nx), py = make_plan(ny);
    const int np = nx / 2 + 1;
    double2* W = nullptr;  // half spectrum, then the roots of both lengths
    const cudaError_t ea = scratch_alloc((void**)&W, ((size_t)np * ny + nx + ny) * sizeof(double2), st);
    if (ea != cudaSuccess) {
        cudaGetLastError();
        err = std::string("spectrum scratch: ") + cudaGetErrorString(ea);
        return PIC_ENOMEM;
    }
    double2 *twx = W + (size_t)np * ny, *twy = twx + nx;
    const int smem = kMaxN * (int)sizeof(double2);
    cudaFuncSetAttribute(k_fft_rows<1024, kMaxN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(k_fft_cols<1024, kMaxN>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    const double scale = 1.0 / ((double)nx * ny);
    const auto blocks = [](int n, int b) { return (unsigned)((n + b - 1) / b); };
    k_roots<<<blocks(std::max(nx, ny), 64), 64, 0, st>>>(nx, twx, ny, twy);
    if (px.direct)
        k_dft_rows<<<dim3(blocks(np, kDftThreads), blocks(ny, kDftLines)), kDftThreads, 0, st>>>(F, nx, ny, twx, W);
    else if (nx <= kShort)
        k_fft_rows<256, kShort><<<(unsigned)ny, 256, nx * sizeof(double2), st>>>(F, nx, ny, px, twx, W);
    else
        k_fft_rows<1024, kMaxN><<<(unsigned)ny, 1024, nx * sizeof(double2), st>>>(F, nx, ny, px, twx, W);
    if (py.direct)
        k_dft_cols<<<dim3(blocks(ny / 2 + 1, kDftThreads), blocks(np, kDftCols)), kDftThreads, 0, st>>>(W, nx, ny, twy,
                                                                                                   scale, out);
    else if (ny <= kShort)
        k_fft_cols<256, kShort><<<(unsigned)np, 256, ny * sizeof(double2), st>>>(W, nx, ny, py, twy, scale, out);
    else
        k_fft_cols<1024, kMaxN><<<(unsigned)np, 1024, ny * sizeof(double2), st>>>(W, nx, ny, py, twy, scale, out);
    const cudaError_t e = cudaGetLastError();
    temp_free(W, st);
    if (e != cudaSuccess) {
        err = std::string("spectrum: ") + cudaGetErrorString(e);
        return PIC_ECUDA;
    }
    return PIC_OK;
}

}  // namespace pic
