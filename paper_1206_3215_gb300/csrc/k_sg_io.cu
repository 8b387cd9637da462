// Sine-Gordon set-up and read-back: real fields <-> the stepping state
// {uhat^n, d^n, H}, with full or half spectra.
//
// Reading u^n is one row pass (inverse, into full complex rows; half spectra are
// extended as they are read) and one column pass that writes the real parts;
// setting it is one row and one column pass per array.  The start-up (backward
// Taylor step) is
//   d^0 = dt F v0 + (dt^2/2) (|k|^2 uhat^0 + F sin u0),
// each of the three transforms rounded to the grid's precision, their sum
// formed in double (FP32: in pairs of floats) and rounded once, and sin u0 the
// rounded value of the sine in double (FP32: again through pairs where it can be).
//
// Half spectra could be read with half the columns (columns first) and with
// half-length rows of packed pairs, as the step's row pass has them.  Both cost
// accuracy: taking the real part at the end drops half of the rounding error
// that a full complex transform has collected.  Read-back alone at 512^2, FP32
// / FP64: as here 1.10e-7 / 2.2e-16, columns first 1.27e-7 / 2.7e-16,
// half-length rows 1.38e-7 / 2.9e-16.  At 2048^2 x 8 in FP32 a level takes 0.35
// ms, with half-length rows 0.19.
//
// 2048^2 x 8 on half spectra in FP32, against transforms of full complex arrays
// with separate copies, conversions and FP64 elementwise kernels: set-up
// 3.54 -> 0.60 ms (with a velocity 3.64 -> 0.81), read-back of both levels
// 0.99 -> 0.70 ms, Hamiltonian 3.64 -> 2.07 ms.
//
// (The state is set on half spectra.  A field set and read back before its first
// step carries the forward transform's error unhalved, 1.65e-7 at 512^2 in FP32
// where full spectra give 1.49e-7; after a step both layouts always did.)
#include <algorithm>

#include "launch.cuh"

namespace pss {

namespace {

// H of uhat: column inverse transform of a times scale, into out.  The arithmetic
// is that of the second half of the step's column pass (SgCol), so H made here
// from uhat is the H the step left, bit for bit.
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

// A sum of products held as an unevaluated pair of floats: the error of each
// product (fused multiply-add) and of each addition (Knuth's two-sum) collects
// in lo, so that hi + lo rounds once, as a sum in double would.  Roundings are
// written out: the compiler must not fuse across them.
struct PairSum {
    float hi, lo;
    // + (c + cl) x
    __device__ __forceinline__ void add(float c, float cl, float x)
    {
        const float p = __fmul_rn(c, x), e = __fmaf_rn(cl, x, __fmaf_rn(c, x, -p));
        const float s = __fadd_rn(hi, p), b = __fsub_rn(s, hi);
        lo = __fadd_rn(lo, __fadd_rn(e, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(p, b))));
        hi = s;
    }
    __device__ __forceinline__ float value() const { return __fadd_rn(hi, lo); }
};

// constants of the start-up and their rests below the grid's precision (FP64: 0)
template <class Rl> struct StartArgs {
    Rl dt, dt_lo, h, h_lo;  // dt and dt^2/2
    double dt64, h64;
};

// the start-up's column pass: data = dt v + (dt^2/2) (|k|^2 u + column transform
// of data), u and v (may be null) transformed already.  |k|^2 from the per-axis
// tables in double, or (FP32) (dt^2/2) |k|^2 from {hi, lo} tables: the sums in
// FP64 took 0.9 ms at 2048^2 x 8, the whole set-up takes 0.6.
template <class Rl> struct SgStartCol {
    static constexpr int NIN = 1;
    static constexpr bool LEAN = true;
    static constexpr int PMAX = 32;
    static constexpr bool EARLY_NEXT = true;
    V2<Rl> *data;
    const V2<Rl> *u, *v;
    const V2<Rl> *cx, *cy;    // FP32: {hi, lo} of (dt^2/2) k^2 per axis
    const double *kx2, *ky2;  // FP64: k^2 per axis
    StartArgs<Rl> g;
    int64_t nx;
    __device__ const V2<Rl> *in(int) const { return data; }
    template <int N, int P, int BLOCK, class Sm, class H = NoHook>
    __device__ __forceinline__ void col(V2<Rl> (&vv)[1][P], int64_t field, int x, int t, const Sm (&sm)[1],
                                        const TW<Rl> *tw, const H &hook = H{}) const
    {
        constexpr int T = N / P;
        V2<Rl>(&a)[P] = vv[0];
        const int64_t base = field * N * nx + x;
        block_fft<N, P, -1, BLOCK>(a, sm[0], t, tw, hook);
        // u and v four points ahead (the compiler does not move loads over stores
        // or hold them all)
        constexpr int CH = P < 4 ? P : 4;
        V2<Rl> ua[CH], va[CH];
#pragma unroll
        for (int m = 0; m < P; ++m) {
            const int y = t + T * m;
            if (m % CH == 0)
#pragma unroll
                for (int c = 0; c < CH; ++c) {
                    const int64_t o = base + int64_t(t + T * (m + c)) * nx;
                    ua[c] = u[o];
                    va[c] = v ? v[o] : V2<Rl>{Rl(0), Rl(0)};
                }
            const V2<Rl> un = ua[m % CH], vn = va[m % CH];
            if constexpr (sizeof(Rl) == 4) {
                // the tables' sum as a pair
                const float2 kx = __ldg(cx + x), ky = __ldg(cy + y);
                const float c = __fadd_rn(kx.x, ky.x), b = __fsub_rn(c, kx.x);
                const float cl = __fadd_rn(__fadd_rn(__fsub_rn(kx.x, __fsub_rn(c, b)), __fsub_rn(ky.x, b)),
                                           __fadd_rn(kx.y, ky.y));
                auto sum = [&](float s, float uk, float vk) {
                    PairSum r{0.0f, 0.0f};
                    r.add(c, cl, uk);
                    r.add(g.h, g.h_lo, s);
                    r.add(g.dt, g.dt_lo, vk);
                    return r.value();
                };
                a[m] = V2<Rl>{sum(a[m].x, un.x, vn.x), sum(a[m].y, un.y, vn.y)};
            } else {
                const double k2 = __ldg(kx2 + x) + __ldg(ky2 + y);
                a[m] = V2<Rl>{g.dt64 * vn.x + g.h64 * (k2 * un.x + a[m].x), g.dt64 * vn.y + g.h64 * (k2 * un.y + a[m].y)};
            }
        }
        store_line<P, T>(a, data + base, nx, t, true);
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

// sin x rounded to the grid's precision from a value good to 2^-45.  FP32 on
// |x| <= 0.785: x - x^3/6 as pairs of floats (the second term's error is the
// largest), the rest of its Taylor series (up to x^13; the next term is below
// 2^-39) in float; beyond, the sine in double.
__device__ __forceinline__ float sin_rounded(float x)
{
    if (!(fabsf(x) <= 0.785f)) return float(sin(double(x)));
    constexpr float S = float(-1.0 / 6), SL = float(-1.0 / 6 - double(S));
    const float t = __fmul_rn(x, x), tl = __fmaf_rn(x, x, -t);
    const float c = __fmul_rn(x, t), cl = __fmaf_rn(x, tl, __fmaf_rn(x, t, -c));  // x^3
    const float v = __fmul_rn(c, S), vl = __fmaf_rn(cl, S, __fmaf_rn(c, SL, __fmaf_rn(c, S, -v)));
    float w = __fmaf_rn(t, float(1.0 / 6227020800.0), float(-1.0 / 39916800.0));
    w = __fmaf_rn(t, w, float(1.0 / 362880.0));
    w = __fmaf_rn(t, w, float(-1.0 / 5040.0));
    w = __fmaf_rn(t, w, float(1.0 / 120.0));
    w = __fmul_rn(__fmul_rn(c, t), w);
    const float d = __fadd_rn(x, v), e = __fsub_rn(v, __fsub_rn(d, x));  // |v| < |x|: exact
    return __fadd_rn(d, __fadd_rn(e, __fadd_rn(vl, w)));
}
__device__ __forceinline__ double sin_rounded(double x) { return sin(x); }

template <class Rl> __global__ void k_sg_sine(const Rl *u, Rl *dst, int64_t n)
{
    const int64_t step = int64_t(gridDim.x) * blockDim.x;
    int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    for (; i + 3 * step < n; i += 4 * step) {
        Rl x[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) x[k] = u[i + k * step];
#pragma unroll
        for (int k = 0; k < 4; ++k) dst[i + k * step] = sin_rounded(x[k]);
    }
    for (; i < n; i += step) dst[i] = sin_rounded(u[i]);
}

}  // namespace

template <class Rl>
cudaError_t sg_level_cols(const V2<Rl> *a, V2<Rl> *out, Rl scale, int64_t nx, int64_t ny, int64_t batch,
                          const TW<Rl> *twy, cudaStream_t s)
{
    return launch_col<Rl>(ny, nx, SgLevelCol<Rl>{a, out, scale, nx}, twy, batch, s);
}
template <class Rl>
cudaError_t sg_start_cols(V2<Rl> *data, const V2<Rl> *u, const V2<Rl> *v, double dt, const V2<Rl> *cx, const V2<Rl> *cy,
                          const double *kx2, const double *ky2, int64_t nx, int64_t ny, int64_t batch,
                          const TW<Rl> *twy, cudaStream_t s)
{
    const double h = 0.5 * dt * dt;
    const StartArgs<Rl> g{Rl(dt), Rl(dt - double(Rl(dt))), Rl(h), Rl(h - double(Rl(h))), dt, h};
    return launch_col<Rl>(ny, nx, SgStartCol<Rl>{data, u, v, cx, cy, kx2, ky2, g, nx}, twy, batch, s);
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
template <class Rl> cudaError_t sg_sine(const Rl *u, Rl *dst, int64_t n, cudaStream_t s)
{
    const unsigned blocks = unsigned(std::min<int64_t>((n + 255) / 256, 4096));
    k_sg_sine<Rl><<<blocks, 256, 0, s>>>(u, dst, n);
    return cudaGetLastError();
}

#define PSS_INST(Rl)                                                                                             \
    template cudaError_t sg_level_cols<Rl>(const V2<Rl> *, V2<Rl> *, Rl, int64_t, int64_t, int64_t,              \
                                           const TW<Rl> *, cudaStream_t);                                        \
    template cudaError_t sg_start_cols<Rl>(V2<Rl> *, const V2<Rl> *, const V2<Rl> *, double, const V2<Rl> *,     \
                                           const V2<Rl> *, const double *, const double *, int64_t, int64_t,     \
                                           int64_t, const TW<Rl> *, cudaStream_t);                               \
    template cudaError_t rows_from_real<Rl>(const Rl *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,            \
                                            const TW<Rl> *, cudaStream_t);                                       \
    template cudaError_t rows_inverse<Rl>(V2<Rl> *const[3], const int *, int64_t, const V2<Rl> *, V2<Rl> *,      \
                                          int64_t, int64_t, int64_t, int64_t, const TW<Rl> *, cudaStream_t);     \
    template cudaError_t cols_to_real<Rl>(const V2<Rl> *, Rl *, Rl, int64_t, int64_t, int64_t, const TW<Rl> *,   \
                                          cudaStream_t);                                                         \
    template cudaError_t sg_sine<Rl>(const Rl *, Rl *, int64_t, cudaStream_t);
PSS_INST(float)
PSS_INST(double)

}  // namespace pss
