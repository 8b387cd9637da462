// Sine-Gordon step (Eq. 3, Section 4.2) on half spectra: u is real, so its
// Fourier coefficients for kx < 0 are the complex conjugates of those for
// kx > 0 and only kx = 0 .. N/2 are kept (the paper's own programs use
// real-to-complex transforms for this equation, Section 5.2).  Both passes
// then move about half the bytes of the complex-to-complex step.
//
// Layout: complex [batch][ny][sx], sx >= N/2 + 1; columns 0 .. N/2 hold the
// half spectrum in x, the columns beyond hold zeros (the column pass carries
// them along unchanged).
//
// The row pass turns H (x: half spectrum, y: physical) into S, the half
// spectrum in x of sin u.  A row of N real points u_n is handled as M = N/2
// complex points z_j = u_{2j} + i u_{2j+1}.  From the half spectrum X_0 .. X_M
// of u (and X_{M+k} = conj X_{M-k}):
//   Z_k = (X_k + conj X_{M-k}) + i e^{2 pi i k/N} (X_k - conj X_{M-k}),  k < M,
//   z = unnormalised inverse DFT_M of Z.
// After s = sin u, the forward DFT_M W of w_j = s_{2j} + i s_{2j+1} gives
//   A_k = (W_k + conj W_{M-k}) / 2,   B_k = -i (W_k - conj W_{M-k}) / 2,
//   S_k = A_k + e^{-2 pi i k/N} B_k  (k < M),   S_M = A_0 - B_0,
// where A and B are the DFTs of the even and odd samples of s.  The column
// pass is the complex one of k_sg.cu applied to the sx columns.
// The same row work without the sine, in either direction alone, turns real
// fields into half spectra and back (HalfRow).
#pragma once
#include "launch.cuh"
#include "sg_sin.cuh"

namespace pss {

template <class Rl, int M, bool SMALL> struct R2cCfg {
    static constexpr int P = Shape<Rl>::rowP(M, SMALL);
    static constexpr int T = M / P;
    // short rows: smaller CTAs, so that few rows still spread over the SMs; FP64
    // as in RowCfg (SG 1024^2 x 2 451 -> 413 us per step, 256^2 x 2 44 -> 40)
    static constexpr int RT = sizeof(Rl) == 8 ? (M <= 256 ? 32 : 64) : M <= 256 ? 128 : 256;
    static constexpr int ROWS = T >= RT ? 1 : RT / T;
    static constexpr int THREADS = ROWS * T;
    // barrier of one row's threads (fft_sync): a warp (T <= 32: the rows are
    // warp-local), the CTA, or the row's own named barrier
    static constexpr int BLOCK = T <= 32 ? 0 : (ROWS > 1 ? T : 1);
    static constexpr int PADLOG = pad_log(P);
    static constexpr int LINE = M + (M >> PADLOG) + 2;  // the padded line plus X_M
    static constexpr size_t SMEM = size_t(ROWS) * LINE * sizeof(V2<Rl>);
    static constexpr int MIN_CTAS = sizeof(Rl) == 4 ? imin(imax(512 / THREADS, 1), 16) : 1;
};

// What a row pass does with its rows:
//   STEP   half spectrum H -> half spectrum of sin u, in place;
//   SPLIT  real row a -> half spectrum of a;
//   START  real rows a = u, b = v (may be null) -> half spectrum of dt v + (dt^2/2) sin u;
//   JOIN   half spectrum -> real row (unnormalised inverse transform).
// START's sum is the part of the sine-Gordon start-up that one transform can
// carry for both terms.
enum class HalfRow { STEP, SPLIT, START, JOIN };
template <class Rl> struct HalfRowArgs {
    V2<Rl> *h;              // half spectra, rows of sx (in: STEP, JOIN; out: all but JOIN)
    const V2<Rl> *a, *b;    // real rows of 2 M points, read as M pairs
    V2<Rl> *out;            // JOIN: real rows
    int64_t sx;
    Rl dt, dt_lo, dt2_2, dt2_2_lo;  // START: dt and dt^2/2 (FP32: and the rests of their rounding)
};

// dt v + (dt^2/2) sin u: the rests of the constants enter inside the fused
// multiply-adds, so that their rounding does not scale the whole field
template <class Rl> __device__ __forceinline__ Rl half_start(const HalfRowArgs<Rl> &g, Rl u, Rl v)
{
    const Rl s = sg_sin(u);
    return g.dt * v + (g.dt2_2 * s + (g.dt_lo * v + g.dt2_2_lo * s));
}

// rows_total = batch * ny; twm: length-M transform twiddles, twn: length-N
// twiddles (e^{-2 pi i e / N}, e < N = 2 M)
template <class Rl, int M, bool SMALL, HalfRow MODE>
__global__ void __launch_bounds__(R2cCfg<Rl, M, SMALL>::THREADS, R2cCfg<Rl, M, SMALL>::MIN_CTAS)
    k_half_row(const HalfRowArgs<Rl> g, int64_t rows_total, const TW<Rl> *__restrict__ twm,
               const TW<Rl> *__restrict__ twn)
{
    using C = R2cCfg<Rl, M, SMALL>;
    using V = V2<Rl>;
    using Sm = SmemLine<V, C::PADLOG>;
    constexpr int P = C::P, T = C::T;
    constexpr bool FROM_HALF = MODE == HalfRow::STEP || MODE == HalfRow::JOIN;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int rl = threadIdx.x / T, t = threadIdx.x % T;
    const Sm sm{reinterpret_cast<V *>(smem_raw) + rl * C::LINE};
    fill_stage_tw<M, P>(twm);
    grid_wait();
    grid_trigger((rows_total + C::ROWS - 1) / C::ROWS);
    __syncthreads();
    for (int64_t r0 = int64_t(blockIdx.x) * C::ROWS; r0 < rows_total; r0 += int64_t(gridDim.x) * C::ROWS) {
        const int64_t row = r0 + rl;
        const bool ok = row < rows_total;
        V *const p = g.h + (ok ? row : int64_t(0)) * g.sx;
        fft_sync<C::BLOCK>();  // the previous row's last readers are done
        V v[P];
        const TW<Rl> *tn;
        if constexpr (FROM_HALF) {
            // stage X_0 .. X_M of the row (every thread reads two of them below)
            if (ok) {
#pragma unroll
                for (int m = 0; m < P; ++m) cp_async<sizeof(V)>(&sm[t + T * m], p + t + T * m);
                if (t == 0) cp_async<sizeof(V)>(&sm[M], p + M);
            }
            cp_async_commit();
            cp_async_wait<0>();
            fft_sync<C::BLOCK>();
            tn = launder(twn);
#pragma unroll
            for (int m = 0; m < P; ++m) {
                const int k = t + T * m;
                const V x = sm[k], xp = sm[M - k];
                const V e{x.x + xp.x, x.y - xp.y};                           // X_k + conj X_{M-k}
                const V o = twmul<+1>(V{x.x - xp.x, x.y + xp.y}, __ldg(tn + k));  // e^{2 pi i k/N} (X_k - conj X_{M-k})
                // conj Z_k: the inverse transform runs as conj(F conj Z)
                v[m] = V{e.x - o.y, -(e.y + o.x)};
            }
        } else {
            const int64_t at = (ok ? row : int64_t(0)) * M + t;
#pragma unroll
            for (int m = 0; m < P; ++m) {
                v[m] = g.a[at + T * m];
                if constexpr (MODE == HalfRow::START) {
                    const V w = g.b ? g.b[at + T * m] : V{Rl(0), Rl(0)};
                    v[m] = V{half_start(g, v[m].x, w.x), half_start(g, v[m].y, w.y)};
                }
            }
        }
#pragma unroll 1
        for (int pass = MODE == HalfRow::STEP ? 0 : 1; pass < 2; ++pass) {
            block_fft<M, P, -1, C::BLOCK>(v, sm, t, twm);
            if (MODE == HalfRow::STEP && pass == 0) {
                // z = conj(F conj Z): u_{2j} = Re z, u_{2j+1} = Im z = -Im(F conj Z)
                if (sg_all_small(v, true)) {
#pragma unroll
                    for (int m = 0; m < P; ++m) v[m] = V{sg_sin_poly(v[m].x), sg_sin_poly(-v[m].y)};
                } else {
#pragma unroll
                    for (int m = 0; m < P; ++m) v[m] = V{sg_sin(v[m].x), sg_sin(-v[m].y)};
                }
            }
        }
        if constexpr (MODE == HalfRow::JOIN) {
            if (ok)
#pragma unroll
                for (int m = 0; m < P; ++m) g.out[row * M + t + T * m] = V{v[m].x, -v[m].y};
            continue;
        }
        // W_k in registers (k = t + T m); the partner W_{M-k} through shared memory
        fft_sync<C::BLOCK>();
#pragma unroll
        for (int m = 0; m < P; ++m) sm[t + T * m] = v[m];
        fft_sync<C::BLOCK>();
        tn = launder(twn);
        const Rl half = Rl(0.5);
#pragma unroll
        for (int m = 0; m < P; ++m) {
            const int k = t + T * m;
            const V w = v[m], wp = sm[(M - k) & (M - 1)];
            const V a{half * (w.x + wp.x), half * (w.y - wp.y)};  // (W_k + conj W_{M-k}) / 2
            const V b{half * (w.y + wp.y), half * (wp.x - w.x)};  // -i (W_k - conj W_{M-k}) / 2
            const V tb = twmul<-1>(b, __ldg(tn + k));
            if (ok) p[k] = V{a.x + tb.x, a.y + tb.y};
            if (ok && k == 0) p[M] = V{a.x - b.x, a.y - b.y};
        }
        // new half spectra: the columns beyond N/2 hold zeros
        if (MODE != HalfRow::STEP && ok)
            for (int64_t x = M + 1 + t; x < g.sx; x += T) p[x] = V{Rl(0), Rl(0)};
    }
    cp_async_wait<0>();
}

template <class Rl, int M, bool SMALL, HalfRow MODE>
cudaError_t launch_half_row(const HalfRowArgs<Rl> &g, int64_t rows_total, const TW<Rl> *twm, const TW<Rl> *twn,
                            cudaStream_t s)
{
    using C = R2cCfg<Rl, M, SMALL>;
    auto k = k_half_row<Rl, M, SMALL, MODE>;
    static std::atomic<unsigned> done{0};
    static int ctas[32] = {};
    cudaError_t e = allow_smem(k, C::SMEM, done);
    if (e != cudaSuccess) return e;
    const int64_t tiles = (rows_total + C::ROWS - 1) / C::ROWS;
    if (tiles <= 0) return cudaSuccess;
    int grid = 0;
    if ((e = resident_ctas(k, C::THREADS, C::SMEM, ctas, &grid)) != cudaSuccess) return e;
    if (tiles < grid) grid = int(tiles);
    return launch_chain(k, unsigned(grid), C::THREADS, C::SMEM, s, g, rows_total, twm, twn);
}

// rows of nx real points, nx/2 = M
template <class Rl, HalfRow MODE>
cudaError_t half_rows(const HalfRowArgs<Rl> &g, int64_t nx, int64_t ny, int64_t batch, const TW<Rl> *twm,
                      const TW<Rl> *twn, cudaStream_t s)
{
    const int64_t rows_total = batch * ny;
    [[maybe_unused]] const bool small = nx * ny <= SMALL_FIELD;
    switch (nx / 2) {
#define PSS_CASE(N)                                                                                  \
    case N:                                                                                          \
        if constexpr (short_variant<Rl>(N))                                                          \
            if (small) return launch_half_row<Rl, N, true, MODE>(g, rows_total, twm, twn, s);        \
        return launch_half_row<Rl, N, false, MODE>(g, rows_total, twm, twn, s);
        PSS_CASE(8) PSS_CASE(16) PSS_CASE(32) PSS_CASE(64) PSS_CASE(128) PSS_CASE(256) PSS_CASE(512)
        PSS_CASE(1024) PSS_CASE(2048) PSS_CASE(4096)
#undef PSS_CASE
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace pss
