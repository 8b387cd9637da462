// Sine-Gordon set-up and read-back: real fields <-> the stepping state
// {uhat^n, d^n, H}, with full or half spectra.
//
// Reading u^n is one row pass (inverse, into full complex rows; half spectra are
// extended as they are read) and one column pass that writes the real parts;
// setting it is one row and one column pass per array.  The start-up (backward
// Taylor step)
//   d^0 = dt F v0 + (dt^2/2) (|k|^2 uhat^0 + F sin u0)
//       = F [dt v0 + (dt^2/2) sin u0] + (dt^2/2) |k|^2 uhat^0
// takes the physical-space sum through one transform; its factor
// (dt^2/2) |k|^2 comes from per-axis tables made in FP64 (FP32: hi + lo).
//
// Half spectra could be read with half the columns (columns first) and with
// half-length rows of packed pairs, as the step's row pass has them.  Both cost
// accuracy: taking the real part at the end drops half of the rounding error
// that a full complex transform has collected.  Read-back alone at 512^2, FP32
// / FP64: as here 1.10e-7 / 2.2e-16, columns first 1.27e-7 / 2.7e-16,
// half-length rows 1.38e-7 / 2.9e-16; 2048^2 x 8 FP32 takes 0.05 ms more per
// level than with half the bytes.
//
// 2048^2 x 8 on half spectra, against transforms of full complex arrays with
// separate copies, conversions and FP64 elementwise kernels (sums of kernel
// times): set-up 3.4 -> 0.5 ms, read-back of both levels 1.2 -> 0.3 ms,
// Hamiltonian 3.6 -> 1.9 ms.
#include <algorithm>

#include "launch.cuh"
#include "sg_sin.cuh"

namespace pss {

namespace {

// H of uhat: column inverse transform of a times scale, into out.  The arithmetic is that of the second half of the step's column
// pass (SgCol), so H made here from uhat is the H the step left, bit for bit.
template <class Rl> struct SgLevelCol {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool EARLY_NEXT = true;
    const V2<Rl> *a;
    V2<Rl> *out;
    Rl scale;
    int64_t nx;
    __device__ const V2<Rl> *in(int) const { return a; }
    template <int N, int P, int BLOCK, class Sm, class H = NoHook>
    __device__ __forceinline__ void col(V2<Rl> (&vv)[1][P], int64_t field, int x, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw, const H &hook = H{}) const
    {
        constexpr int T = N / P;
        V2<Rl>(&v)[P] = vv[0];
        const int64_t base = field * N * nx + x;
#pragma unroll
        for (int m = 0; m < P; ++m) v[m] = cscale(v[m], scale);
        if constexpr (sizeof(Rl) == 4) {
            conj_all(v);
            block_fft<N, P, -1, BLOCK>(v, sm[0], t, tw, hook);
            conj_all(v);
        } else {
            block_fft<N, P, +1, BLOCK>(v, sm[0], t, tw, hook);
        }
        store_line<P, T>(v, out + base, nx, t, true);
    }
};

// the start-up's second term: data = column transform of data + c u,
// c = (dt^2/2) (kx^2 + ky^2) from the per-axis tables
template <class Rl> struct SgStartCol {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool EARLY_NEXT = true;
    V2<Rl> *data;
    const V2<Rl> *u;
    const V2<Rl> *cx, *cy;  // {hi, lo} of (dt^2/2) k^2 per axis
    int64_t nx;
    __device__ const V2<Rl> *in(int) const { return data; }
    template <int N, int P, int BLOCK, class Sm, class H = NoHook>
    __device__ __forceinline__ void col(V2<Rl> (&vv)[1][P], int64_t field, int x, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw, const H &hook = H{}) const
    {
        constexpr int T = N / P;
        V2<Rl>(&v)[P] = vv[0];
        const int64_t base = field * N * nx + x;
        block_fft<N, P, -1, BLOCK>(v, sm[0], t, tw, hook);
        const V2<Rl> kx = __ldg(cx + x);
#pragma unroll
        for (int m = 0; m < P; ++m) {
            const int y = t + T * m;
            const V2<Rl> ky = __ldg(cy + y), un = u[base + int64_t(y) * nx];
            // kx + ky as a sum and its rounding error (Knuth's two-sum) plus the low parts
            const Rl c = kx.x + ky.x, bp = c - kx.x, lo = (kx.x - (c - bp)) + (ky.x - bp) + (kx.y + ky.y);
            v[m] = V2<Rl>{fma_(c, un.x, fma_(lo, un.x, v[m].x)), fma_(c, un.y, fma_(lo, un.y, v[m].y))};
        }
        store_line<P, T>(v, data + base, nx, t, true);
    }
    static __device__ __forceinline__ float fma_(float a, float b, float c) { return __fmaf_rn(a, b, c); }
    static __device__ __forceinline__ double fma_(double a, double b, double c) { return __fma_rn(a, b, c); }
};

// real rows, complex forward row transform, columns 0 .. N/2 (half spectra:
// rows of sx, zeros beyond) or all of them (sx = 0)
template <class Rl> struct RowFromReal {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool DIRECT_LOAD = true;
    const Rl *src;
    V2<Rl> *dst;
    int64_t sx;
    __device__ const V2<Rl> *in(int) const { return nullptr; }
    template <int N, int P>
    __device__ __forceinline__ void load(V2<Rl> (&v)[P], int64_t r, bool ok, int t) const
    {
#pragma unroll
        for (int m = 0; m < P; ++m) v[m] = V2<Rl>{ok ? src[r * N + t + (N / P) * m] : Rl(0), Rl(0)};
    }
    template <int N, int P, int BLOCK, class Sm>
    __device__ __forceinline__ void row(V2<Rl> (&v)[1][P], int64_t r, bool ok, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw) const
    {
        constexpr int T = N / P;
        block_fft<N, P, -1, BLOCK>(v[0], sm[0], t, tw);
        if (!ok) return;
        V2<Rl> *p = dst + r * (sx ? sx : N);
#pragma unroll
        for (int m = 0; m < P; ++m)
            if (!sx || t + T * m <= N / 2) p[t + T * m] = v[0][m];
        for (int64_t x = N / 2 + 1 + t; x < sx; x += T) p[x] = V2<Rl>{Rl(0), Rl(0)};
    }
};

// inverse row transform of full spectra (sx = 0), or of half spectra (rows of sx)
// extended by their Hermitian symmetry, into full complex rows; of the
// difference with a second spectrum where `minus` is set.  With sel, field f is
// in src[sel[f * sel_stride]].
template <class Rl> struct RowInv {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool DIRECT_LOAD = true;
    const V2<Rl> *src[3], *minus;
    const int *sel;
    int64_t sel_stride;
    V2<Rl> *dst;
    int64_t sx, ny;  // ny: a power of two
    int lgy;
    __device__ const V2<Rl> *in(int) const { return nullptr; }
    __device__ __forceinline__ V2<Rl> at(const V2<Rl> *a, int64_t i) const
    {
        return minus ? csub(a[i], minus[i]) : a[i];
    }
    template <int N, int P>
    __device__ __forceinline__ void load(V2<Rl> (&v)[P], int64_t r, bool ok, int t) const
    {
        constexpr int T = N / P;
        if (!ok) {
#pragma unroll
            for (int m = 0; m < P; ++m) v[m] = V2<Rl>{Rl(0), Rl(0)};
            return;
        }
        const int64_t y = r & (ny - 1);
        const int b = sel ? sel[(r >> lgy) * sel_stride] : 0;
        const V2<Rl> *a = b == 0 ? src[0] : b == 1 ? src[1] : src[2];
        const int64_t p = r * (sx ? sx : N), q = (r - y + ((ny - y) & (ny - 1))) * sx;
#pragma unroll
        for (int m = 0; m < P; ++m) {
            const int x = t + T * m;
            if (!sx || x <= N / 2) {
                v[m] = at(a, p + x);
            } else {
                const V2<Rl> c = at(a, q + N - x);
                v[m] = V2<Rl>{c.x, -c.y};
            }
        }
    }
    template <int N, int P, int BLOCK, class Sm>
    __device__ __forceinline__ void row(V2<Rl> (&v)[1][P], int64_t r, bool ok, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw) const
    {
        block_fft<N, P, +1, BLOCK>(v[0], sm[0], t, tw);
        store_line<P, N / P>(v[0], dst + r * N, 1, t, ok);
    }
};

// inverse column transform times scale, real parts into a real array
template <class Rl> struct ColToReal {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool EARLY_NEXT = true;
    const V2<Rl> *src;
    Rl *dst;
    Rl scale;
    int64_t nx;
    __device__ const V2<Rl> *in(int) const { return src; }
    template <int N, int P, int BLOCK, class Sm, class H = NoHook>
    __device__ __forceinline__ void col(V2<Rl> (&v)[1][P], int64_t field, int x, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw, const H &hook = H{}) const
    {
        constexpr int T = N / P;
        block_fft<N, P, +1, BLOCK>(v[0], sm[0], t, tw, hook);
        Rl *p = dst + field * N * nx + x + int64_t(t) * nx;
        const int64_t step = int64_t(T) * nx;
#pragma unroll
        for (int m = 0; m < P; ++m, p += step) *p = v[0][m].x * scale;
    }
};

// Constants of the start-up: dt and dt^2/2 (FP32: and the rests of their rounding)
template <class Rl> struct StartArgs {
    Rl dt, dt_lo, dt2_2, dt2_2_lo;
};

// dt v + (dt^2/2) sin u (v may be null); the rests of the constants enter inside
// the fused multiply-adds, so that their rounding does not scale the whole field
template <class Rl> __global__ void k_sg_start(const Rl *u, const Rl *v, Rl *dst, StartArgs<Rl> g, int64_t n)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const Rl s = sg_sin(u[i]), w = v ? v[i] : Rl(0);
        dst[i] = g.dt * w + (g.dt2_2 * s + (g.dt_lo * w + g.dt2_2_lo * s));
    }
}

}  // namespace

template <class Rl>
cudaError_t sg_level_cols(const V2<Rl> *a, V2<Rl> *out, Rl scale, int64_t nx, int64_t ny, int64_t batch,
                          const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, SgLevelCol<Rl>{a, out, scale, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t sg_start_cols(V2<Rl> *data, const V2<Rl> *u, const V2<Rl> *cx, const V2<Rl> *cy, int64_t nx, int64_t ny,
                          int64_t batch, const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, SgStartCol<Rl>{data, u, cx, cy, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t rows_from_real(const Rl *src, V2<Rl> *dst, int64_t nx, int64_t sx, int64_t ny, int64_t batch,
                           const TW<Rl> *twx, cudaStream_t s)
{
    return launch_row<Rl>(nx, ny, RowFromReal<Rl>{src, dst, sx}, twx, batch, s);
}
template <class Rl>
cudaError_t rows_inverse(V2<Rl> *const src[3], const int *sel, int64_t sel_stride, const V2<Rl> *minus, V2<Rl> *dst,
                         int64_t nx, int64_t sx, int64_t ny, int64_t batch, const TW<Rl> *twx, cudaStream_t s)
{
    int lgy = 0;
    while ((int64_t(1) << lgy) < ny) ++lgy;
    return launch_row<Rl>(nx, ny, RowInv<Rl>{{src[0], src[1], src[2]}, minus, sel, sel_stride, dst, sx, ny, lgy}, twx,
                          batch, s);
}
template <class Rl>
cudaError_t cols_to_real(const V2<Rl> *src, Rl *dst, Rl scale, int64_t nx, int64_t ny, int64_t batch,
                         const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, ColToReal<Rl>{src, dst, scale, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t sg_start_field(const Rl *u, const Rl *v, Rl *dst, double dt, int64_t n, cudaStream_t s)
{
    const double d2 = 0.5 * dt * dt;
    const StartArgs<Rl> g{Rl(dt), Rl(dt - double(Rl(dt))), Rl(d2), Rl(d2 - double(Rl(d2)))};
    const unsigned blocks = unsigned(std::min<int64_t>((n + 255) / 256, 4096));
    k_sg_start<Rl><<<blocks, 256, 0, s>>>(u, v, dst, g, n);
    return cudaGetLastError();
}

#define PSS_INST(Rl)                                                                                             \
    template cudaError_t sg_level_cols<Rl>(const V2<Rl> *, V2<Rl> *, Rl, int64_t, int64_t, int64_t,              \
                                           const TW<Rl> *, cudaStream_t);                                        \
    template cudaError_t sg_start_cols<Rl>(V2<Rl> *, const V2<Rl> *, const V2<Rl> *, const V2<Rl> *, int64_t,    \
                                           int64_t, int64_t, const TW<Rl> *, cudaStream_t);                      \
    template cudaError_t rows_from_real<Rl>(const Rl *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,            \
                                            const TW<Rl> *, cudaStream_t);                                       \
    template cudaError_t rows_inverse<Rl>(V2<Rl> *const[3], const int *, int64_t, const V2<Rl> *, V2<Rl> *,      \
                                          int64_t, int64_t, int64_t, int64_t, const TW<Rl> *, cudaStream_t);     \
    template cudaError_t cols_to_real<Rl>(const V2<Rl> *, Rl *, Rl, int64_t, int64_t, int64_t, const TW<Rl> *,   \
                                          cudaStream_t);                                                         \
    template cudaError_t sg_start_field<Rl>(const Rl *, const Rl *, Rl *, double, int64_t, cudaStream_t);
PSS_INST(float)
PSS_INST(double)

}  // namespace pss
