// Sine-Gordon set-up and read-back: real fields <-> the stepping state
// {uhat^n, d^n, H}, with full or half spectra.
//
// Reading u^n is one column pass (column inverse transform of uhat^n) and one
// row pass that writes real rows; setting it is one row and one column pass
// per array.  The start-up (backward Taylor step)
//   d^0 = dt F v0 + (dt^2/2) (|k|^2 uhat^0 + F sin u0)
//       = F [dt v0 + (dt^2/2) sin u0] + (dt^2/2) |k|^2 uhat^0
// takes the physical-space sum through one transform; its factor
// (dt^2/2) |k|^2 comes from per-axis tables made in FP64 (FP32: hi + lo).
//
// In FP32 uhat^0 and the real fields of the Hamiltonian go through full
// complex rows (RowFromReal, RowInv): half-length transforms of packed pairs
// round differently, which moves the Hamiltonian of a small field by up to
// 1e-8.
//
// 2048^2 x 8 on half spectra, against transforms of full complex arrays with
// separate copies, conversions and FP64 elementwise kernels (sums of kernel
// times): set-up 3.4 -> 0.5 ms, read-back of both levels 1.2 -> 0.3 ms,
// Hamiltonian 3.6 -> 1.9 ms.
#include <algorithm>

#include "k_sg_r2c.cuh"

namespace pss {

namespace {

// a - b (b may be null) of two spectra, column inverse transform times scale,
// into out.  The arithmetic is that of the second half of the step's column
// pass (SgCol), so H made here from uhat is the H the step left, bit for bit.
template <class Rl> struct SgLevelCol {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool EARLY_NEXT = true;
    const V2<Rl> *a, *b;
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
        if (b)
#pragma unroll
            for (int m = 0; m < P; ++m) v[m] = csub(v[m], b[base + int64_t(t + T * m) * nx]);
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

// rows of a complex array, inverse row transform, real parts into real rows
template <class Rl> struct RowToReal {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool EARLY_NEXT = true;
    const V2<Rl> *src;
    Rl *dst;
    __device__ const V2<Rl> *in(int) const { return src; }
    template <int N, int P, int BLOCK, class Sm, class H = NoHook>
    __device__ __forceinline__ void row(V2<Rl> (&v)[1][P], int64_t r, bool ok, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw, const H &hook = H{}) const
    {
        block_fft<N, P, +1, BLOCK>(v[0], sm[0], t, tw, hook);
        if (!ok) return;
#pragma unroll
        for (int m = 0; m < P; ++m) dst[r * N + t + (N / P) * m] = v[0][m].x;
    }
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

// inverse row transform of full spectra (sx = 0) or of half spectra extended
// by their Hermitian symmetry, into full complex rows
template <class Rl> struct RowInv {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool DIRECT_LOAD = true;
    const V2<Rl> *src;
    V2<Rl> *dst;
    int64_t sx, ny;  // ny: a power of two
    __device__ const V2<Rl> *in(int) const { return nullptr; }
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
        const V2<Rl> *p = src + r * (sx ? sx : N), *q = src + (r - y + ((ny - y) & (ny - 1))) * sx;
#pragma unroll
        for (int m = 0; m < P; ++m) {
            const int x = t + T * m;
            if (!sx || x <= N / 2) {
                v[m] = p[x];
            } else {
                const V2<Rl> c = q[N - x];
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

// dt v + (dt^2/2) sin u (v may be null), as a complex array
template <class Rl> __global__ void k_sg_start(const Rl *u, const Rl *v, V2<Rl> *dst, HalfRowArgs<Rl> g, int64_t n)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        dst[i] = V2<Rl>{half_start(g, u[i], v ? v[i] : Rl(0)), Rl(0)};
}

// the start-up's arguments: rows `a`, `b` into half spectra h
template <class Rl> HalfRowArgs<Rl> start_args(V2<Rl> *h, const Rl *a, const Rl *b, int64_t sx, double dt)
{
    const double d2 = 0.5 * dt * dt;
    return {h, reinterpret_cast<const V2<Rl> *>(a), reinterpret_cast<const V2<Rl> *>(b), nullptr, sx,
            Rl(dt), Rl(dt - double(Rl(dt))), Rl(d2), Rl(d2 - double(Rl(d2)))};
}

}  // namespace

template <class Rl>
cudaError_t sg_half_split(const Rl *a, V2<Rl> *h, int64_t nx, int64_t sx, int64_t ny, int64_t batch,
                          const TW<Rl> *twm, const TW<Rl> *twn, cudaStream_t s)
{
    return half_rows<Rl, HalfRow::SPLIT>(start_args<Rl>(h, a, nullptr, sx, 0.0), nx, ny, batch, twm, twn, s);
}
template <class Rl>
cudaError_t sg_half_start(const Rl *u, const Rl *v, V2<Rl> *h, double dt, int64_t nx, int64_t sx, int64_t ny,
                          int64_t batch, const TW<Rl> *twm, const TW<Rl> *twn, cudaStream_t s)
{
    return half_rows<Rl, HalfRow::START>(start_args<Rl>(h, u, v, sx, dt), nx, ny, batch, twm, twn, s);
}
template <class Rl>
cudaError_t sg_half_join(const V2<Rl> *h, Rl *out, int64_t nx, int64_t sx, int64_t ny, int64_t batch,
                         const TW<Rl> *twm, const TW<Rl> *twn, cudaStream_t s)
{
    HalfRowArgs<Rl> g = start_args<Rl>(const_cast<V2<Rl> *>(h), nullptr, nullptr, sx, 0.0);
    g.out = reinterpret_cast<V2<Rl> *>(out);
    return half_rows<Rl, HalfRow::JOIN>(g, nx, ny, batch, twm, twn, s);
}
template <class Rl>
cudaError_t sg_level_cols(const V2<Rl> *a, const V2<Rl> *b, V2<Rl> *out, Rl scale, int64_t nx, int64_t ny,
                          int64_t batch, const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, SgLevelCol<Rl>{a, b, out, scale, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t sg_start_cols(V2<Rl> *data, const V2<Rl> *u, const V2<Rl> *cx, const V2<Rl> *cy, int64_t nx, int64_t ny,
                          int64_t batch, const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, SgStartCol<Rl>{data, u, cx, cy, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t rows_to_real(const V2<Rl> *src, Rl *dst, int64_t nx, int64_t ny, int64_t batch, const TW<Rl> *twx,
                         cudaStream_t s)
{
    return launch_row<Rl>(nx, ny, RowToReal<Rl>{src, dst}, twx, batch, s);
}
template <class Rl>
cudaError_t rows_from_real(const Rl *src, V2<Rl> *dst, int64_t nx, int64_t sx, int64_t ny, int64_t batch,
                           const TW<Rl> *twx, cudaStream_t s)
{
    return launch_row<Rl>(nx, ny, RowFromReal<Rl>{src, dst, sx}, twx, batch, s);
}
template <class Rl>
cudaError_t rows_inverse(const V2<Rl> *src, V2<Rl> *dst, int64_t nx, int64_t sx, int64_t ny, int64_t batch,
                         const TW<Rl> *twx, cudaStream_t s)
{
    return launch_row<Rl>(nx, ny, RowInv<Rl>{src, dst, sx, ny}, twx, batch, s);
}
template <class Rl>
cudaError_t cols_to_real(const V2<Rl> *src, Rl *dst, Rl scale, int64_t nx, int64_t ny, int64_t batch,
                         const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, ColToReal<Rl>{src, dst, scale, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t sg_start_field(const Rl *u, const Rl *v, V2<Rl> *dst, double dt, int64_t n, cudaStream_t s)
{
    const unsigned blocks = unsigned(std::min<int64_t>((n + 255) / 256, 4096));
    k_sg_start<Rl><<<blocks, 256, 0, s>>>(u, v, dst, start_args<Rl>(nullptr, nullptr, nullptr, 0, dt), n);
    return cudaGetLastError();
}

#define PSS_INST(Rl)                                                                                             \
    template cudaError_t sg_half_split<Rl>(const Rl *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,             \
                                           const TW<Rl> *, const TW<Rl> *, cudaStream_t);                        \
    template cudaError_t sg_half_start<Rl>(const Rl *, const Rl *, V2<Rl> *, double, int64_t, int64_t, int64_t,  \
                                           int64_t, const TW<Rl> *, const TW<Rl> *, cudaStream_t);               \
    template cudaError_t sg_half_join<Rl>(const V2<Rl> *, Rl *, int64_t, int64_t, int64_t, int64_t,              \
                                          const TW<Rl> *, const TW<Rl> *, cudaStream_t);                         \
    template cudaError_t sg_level_cols<Rl>(const V2<Rl> *, const V2<Rl> *, V2<Rl> *, Rl, int64_t, int64_t,       \
                                           int64_t, const TW<Rl> *, cudaStream_t);                               \
    template cudaError_t sg_start_cols<Rl>(V2<Rl> *, const V2<Rl> *, const V2<Rl> *, const V2<Rl> *, int64_t,    \
                                           int64_t, int64_t, const TW<Rl> *, cudaStream_t);                      \
    template cudaError_t rows_to_real<Rl>(const V2<Rl> *, Rl *, int64_t, int64_t, int64_t, const TW<Rl> *,       \
                                          cudaStream_t);                                                         \
    template cudaError_t rows_from_real<Rl>(const Rl *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,            \
                                            const TW<Rl> *, cudaStream_t);                                       \
    template cudaError_t rows_inverse<Rl>(const V2<Rl> *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,          \
                                          const TW<Rl> *, cudaStream_t);                                         \
    template cudaError_t cols_to_real<Rl>(const V2<Rl> *, Rl *, Rl, int64_t, int64_t, int64_t, const TW<Rl> *,   \
                                          cudaStream_t);                                                         \
    template cudaError_t sg_start_field<Rl>(const Rl *, const Rl *, V2<Rl> *, double, int64_t, cudaStream_t);
PSS_INST(float)
PSS_INST(double)

}  // namespace pss
