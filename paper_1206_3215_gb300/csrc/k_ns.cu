// Navier-Stokes passes: loop control, row pass, derivative pass and the
// Crank-Nicolson column pass (the kernels are defined in k_ns.cuh).
#include "k_ns.cuh"

namespace pss {

// One block per field: fold the partials of its update in a fixed order (a
// strided sum per thread, then a tree), decide, count.  A field whose step is
// done goes on with its next one in the next update, whatever the batch's
// other fields do; with `restart_at_end` (midpoint: a step starts with the
// derivatives of w^n, formed once per loop body) it pauses until the body's
// last update (`last`).  The block that finishes last resets the control
// words for the next column pass and, inside a captured loop, sets the WHILE
// node's condition: some field is active.  Every field stops at max_iter at
// the latest, so the loop always ends; after a lost tile copy it ends at once.
constexpr int NS_DECIDE_THREADS = 256;
__global__ void __launch_bounds__(NS_DECIDE_THREADS)
    k_ns_decide(NsField *fs, const double *partials, int64_t groups, int64_t batch, int *ctl, double parseval,
                double tol, int max_iter, int restart_at_end, int last, int use_graph, cudaGraphConditionalHandle h)
{
    __shared__ double red[NS_DECIDE_THREADS];
    grid_wait();
    grid_trigger(1);
    // one thread reads the record and the loop's state for the block: it writes
    // the record below, and the block that finishes last writes the state
    __shared__ NsField rec;
    __shared__ int over;
    const int64_t f = blockIdx.x;
    if (threadIdx.x == 0) {
        rec = fs[f];
        over = ctl[NS_CTL_MORE] == 0;
    }
    __syncthreads();
    const bool idle = over != 0;
    NsField s = rec;
    if (!idle && s.active) {  // the same for every thread of the block
        double sum = 0.0;
        for (int64_t g = threadIdx.x; g < groups; g += NS_DECIDE_THREADS) sum += partials[f * groups + g];
        red[threadIdx.x] = sum;
        __syncthreads();
        for (int w = NS_DECIDE_THREADS / 2; w > 0; w >>= 1) {
            if (int(threadIdx.x) < w) red[threadIdx.x] += red[threadIdx.x + w];
            __syncthreads();
        }
    }
    if (threadIdx.x != 0) return;
    if (!idle) {
        if (s.active) {
            const double norm = parseval * red[0];
            s.updates += 1;
            const bool done = norm < tol;
            if (done || s.k + 1 >= max_iter) {
                if (!done) s.nonconv = 1;
                s.idx = ns_buf(s.idx, s.k + 1);
                s.k = 0;
                s.left -= 1;
                s.active = s.left > 0 && !restart_at_end;
            } else {
                s.k += 1;
            }
        }
        if (restart_at_end && last && !s.active && s.left > 0) s.active = 1;
        fs[f] = s;
        const int any = (s.left > 0 ? 1 : 0) | (s.active && s.k == 0 ? 2 : 0) | (s.active ? 4 : 0);
        if (any) atomicOr(ctl + NS_CTL_ANY, any);
    }
    __threadfence();
    if (atomicAdd(ctl + NS_CTL_TICKET, 1) + 1 < int(gridDim.x)) return;
    __threadfence();
    const int any = atomicExch(ctl + NS_CTL_ANY, 0);
    const int more = (any & 1) && ctl[FLAG_SLOT_PASS_STATUS] == 0;
    ctl[NS_CTL_TICKET] = 0;
    ctl[NS_CTL_MORE] = more;
    ctl[NS_CTL_START] = (any & 2) != 0;
    ctl[NS_CTL_ACTIVE] = more && (any & 4) != 0;
    ctl[FLAG_SLOT_SPLIT_CLAIM] = 0;  // the next column pass claims its items from 0
    ctl[FLAG_SLOT_EPOCH] += 1;       // and publishes its tiles under a new value
    if (use_graph) cudaGraphSetConditional(h, more ? 1u : 0u);
}

// start of a call of n steps
__global__ void k_ns_begin(NsField *fs, int64_t batch, int *ctl, int n)
{
    const int64_t f = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (f == 0) {
        ctl[NS_CTL_ANY] = 0;
        ctl[NS_CTL_TICKET] = 0;
        ctl[NS_CTL_MORE] = 1;
        ctl[NS_CTL_START] = 1;
        ctl[NS_CTL_ACTIVE] = 1;
        ctl[FLAG_SLOT_SPLIT_CLAIM] = 0;
    }
    if (f < batch) {
        fs[f].active = 1;
        fs[f].k = 0;
        fs[f].left = n;
    }
}

// Row pass of one update for FP32 rows of up to 2048 points: row inverse
// transforms of C1 and C2, J = Re C1 Re C2 + Im C1 Im C2, row forward
// transform into c1.
//
// All three run through one forward-transform body (F^-1 x = conj(F conj x),
// exact), and a thread holds one array of P points (at most 128 registers, 16
// warps per SM; with both arrays in registers 215 and 8): C1's result waits
// in the second shared-memory line of the row, at the thread's own points,
// where C2 was staged.  That line is read and written at own points only, so
// it needs no barrier; its next copy is issued once J is formed, the first
// line's from the start of the last stage.  NS per step, both arrays in
// registers -> this: 1024^2 x 4 half spectra 256 -> 234 us, 512^2 x 8
// 157 -> 152, 512 x 256 x 5 midpoint 89 -> 86; 2048^2 the same.  80 registers
// (24 warps) spill: 1024^2 x 4 267 us.  Two halves of a CTA carrying C1 and C2
// side by side: 246 us, 4096^2 940 (64 registers: 280, 1067).
//
// Dealiasing (2/3 rule): the columns with 3 |mx| >= nx hold zeros in C1 and C2
// and are not read (zero_in; a restored state may have them filled), and J is
// not written there (the column pass skips them, the mask discards J); half
// spectra: J is written for columns 0 .. nx/2.
constexpr int NS_ROW_MAX = 2048;
template <int N> struct NsRowCfg {
    static constexpr int P = imin(Shape<float>::rowP(N), 16);
    static constexpr int T = N / P;
    static constexpr int RT = N <= 256 ? 64 : 256;
    static constexpr int ROWS = T >= RT ? 1 : RT / T;
    static constexpr int THREADS = ROWS * T;
    static constexpr int BLOCK = T <= 32 ? 0 : (ROWS > 1 ? T : 1);  // the barrier of one row's threads
    static constexpr int PADLOG = pad_log(P);
    static constexpr int LINE = N + (N >> PADLOG);
    static constexpr size_t SMEM = size_t(2) * ROWS * LINE * sizeof(float2);
    static constexpr int MIN_CTAS = imin(imax(512 / THREADS, 1), 16);
};

template <int N>
__global__ void __launch_bounds__(NsRowCfg<N>::THREADS, NsRowCfg<N>::MIN_CTAS)
    k_ns_row(float2 *c1, const float2 *c2, const NsField *fs, int lgy, int dealias, int zero_in, int half,
             const int *ctl, const float4 *__restrict__ tw, int64_t rows_total)
{
    using C = NsRowCfg<N>;
    using V = float2;
    using Sm = SmemLine<V, C::PADLOG>;
    constexpr int P = C::P, T = C::T;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    V *const lines = reinterpret_cast<V *>(smem_raw);
    const int lr = threadIdx.x / T, t = threadIdx.x % T;
    const Sm sm{lines + lr * C::LINE}, park{lines + (C::ROWS + lr) * C::LINE};
    const int64_t tiles = (rows_total + C::ROWS - 1) / C::ROWS;
    auto kept_col = [&](int x) { return 3 * (x < N / 2 ? x : N - x) < N; };
    // column x of C1, C2 is not known to be zero
    auto live_col = [&](int x) { return !zero_in || kept_col(x); };
    auto issue = [&](int64_t tile, const V *in, const Sm &line) {
        const int64_t row = tile * C::ROWS + lr;
        if (tile < tiles && row < rows_total) {
            const V *p = in + row * N + t;
#pragma unroll
            for (int m = 0; m < P; ++m)
                if (live_col(t + T * m)) cp_async<sizeof(V)>(&line[t + T * m], p + T * m);
        }
        cp_async_commit();
    };
    fill_stage_tw<N, P>(tw);
    grid_wait();
    grid_trigger(tiles);
    if (ctl[NS_CTL_ACTIVE] == 0) return;
    int64_t tile = blockIdx.x;
    issue(tile, c2, park);
    issue(tile, c1, sm);
    __syncthreads();
    for (; tile < tiles; tile += gridDim.x) {
        const int64_t row = tile * C::ROWS + lr, next = tile + gridDim.x;
        cp_async_wait<0>();
        V v[P];
#pragma unroll
        for (int m = 0; m < P; ++m) {
            const V x = sm[t + T * m];
            v[m] = live_col(t + T * m) ? V{x.x, -x.y} : V{0.0f, 0.0f};
        }
        // pass 0: C1, pass 1: C2 (each as F of the conjugate, which leaves the
        // conjugate of the inverse transform), pass 2: J
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            block_fft<N, P, -1, C::BLOCK>(v, sm, t, tw, [&]() {
                if (pass == 2) {
                    fft_sync<C::BLOCK>();  // the row's last shared-memory reads are done
                    issue(next, c1, sm);
                }
            });
            if (pass == 0) {
#pragma unroll
                for (int m = 0; m < P; ++m) {
                    const V w = park[t + T * m];
                    park[t + T * m] = v[m];
                    v[m] = live_col(t + T * m) ? V{w.x, -w.y} : V{0.0f, 0.0f};
                }
            } else if (pass == 1) {
#pragma unroll
                for (int m = 0; m < P; ++m) {
                    const V w = park[t + T * m];
                    v[m] = V{fma_rn(w.x, v[m].x, mul_rn(w.y, v[m].y)), 0.0f};
                }
                issue(next, c2, park);
            }
        }
        if (row < rows_total && fs[row >> lgy].active) {
            V *p = c1 + row * N + t;
#pragma unroll
            for (int m = 0; m < P; ++m) {
                const int x = t + T * m;
                if ((!dealias || kept_col(x)) && (!half || x <= N / 2)) p[T * m] = v[m];
            }
        }
    }
    cp_async_wait<0>();
}

template <class Rl>
cudaError_t ns_row_pass(V2<Rl> *c1, V2<Rl> *c2, const void *fs, int64_t nx, int64_t ny, int64_t batch,
                        const int *ctl, const TW<Rl> *twx, cudaStream_t s, bool dealias, bool zero_in, bool half)
{
    const NsField *f = static_cast<const NsField *>(fs);
    int lgy = 0;
    while ((int64_t(1) << lgy) < ny) ++lgy;  // ny is a power of two: row r belongs to field r >> lgy
    auto short_rows = [&](auto n) -> cudaError_t {
        constexpr int N = decltype(n)::value;
        using C = NsRowCfg<N>;
        auto k = k_ns_row<N>;
        static std::atomic<unsigned> done{0};
        static int ctas[32] = {};
        cudaError_t e = allow_smem(k, C::SMEM, done);
        if (e != cudaSuccess) return e;
        const int64_t rows_total = batch * ny, tiles = (rows_total + C::ROWS - 1) / C::ROWS;
        int grid = 0;
        if ((e = resident_ctas(k, C::THREADS, C::SMEM, ctas, &grid)) != cudaSuccess) return e;
        if (tiles < grid) grid = int(tiles);
        return launch_chain(k, unsigned(grid), C::THREADS, C::SMEM, s, reinterpret_cast<float2 *>(c1),
                            reinterpret_cast<const float2 *>(c2), f, lgy, dealias ? 1 : 0, zero_in ? 1 : 0, half ? 1 : 0,
                            ctl, reinterpret_cast<const float4 *>(twx), rows_total);
    };
    const NsRow<Rl> op{c1, c2, f, lgy, dealias ? 1 : 0, zero_in ? 1 : 0, half ? 1 : 0, ctl};
    switch (nx) {
#define PSS_CASE(N)                                                                                       \
    case N:                                                                                               \
        if constexpr (sizeof(Rl) == 4 && N <= NS_ROW_MAX) return short_rows(std::integral_constant<int, N>{}); \
        else return launch_row_n<Rl, N>(op, twx, ny, batch, s);
        PSS_FOR_EACH_N(PSS_CASE)
#undef PSS_CASE
    default: return cudaErrorInvalidValue;
    }
}

template <class Rl>
cudaError_t ns_col_pass(V2<Rl> *c1, V2<Rl> *c2, V2<Rl> *const w[3], V2<Rl> *jn, void *fs, double *partials,
                        const Rl *kxo, const Rl *kyo, const Rl *kx2, const Rl *ky2, const Rl *keepx,
                        const Rl *keepy, double dt, double nu, int64_t nx, int64_t ny, int64_t batch,
                        const int *ctl, int midpoint, const TW<Rl> *twy, int *groups_out, cudaStream_t s,
                        bool dealias, int64_t sx)
{
    if (sx > 0)
        return ns_col_half<Rl>(c1, c2, w, jn, fs, partials, kxo, kyo, kx2, ky2, keepx, keepy, dt, nu, nx, sx, ny,
                               batch, ctl, midpoint, twy, groups_out, s, dealias);
    return midpoint ? ns_col_mid<Rl>(c1, c2, w, jn, fs, partials, kxo, kyo, kx2, ky2, keepx, keepy, dt, nu, nx, ny,
                                     batch, ctl, twy, groups_out, s, dealias)
                    : ns_col_run<Rl, false, false>(c1, c2, w, jn, fs, partials, kxo, kyo, kx2, ky2, keepx, keepy, dt,
                                                   nu, nx, nx, ny, batch, ctl, twy, groups_out, s, dealias);
}

template <class Rl>
cudaError_t ns_prep_pass(V2<Rl> *const w[3], const void *fs, V2<Rl> *c1, V2<Rl> *c2, const Rl *kxo, const Rl *kyo,
                         const Rl *kx2, const Rl *ky2, int64_t nx, int64_t ny, int64_t batch,
                         const int *ctl, const TW<Rl> *twy, cudaStream_t s, int64_t sx)
{
    if (sx > 0) return ns_prep_half<Rl>(w, fs, c1, c2, kxo, kyo, kx2, ky2, nx, sx, ny, batch, ctl, twy, s);
    NsPrep<Rl> op{w[0], w[1], w[2], static_cast<const NsField *>(fs), c1, c2, kxo, kyo, kx2, ky2,
                  Rl(1.0 / (double(nx) * double(ny))), nx, nx, ctl};
    return launch_col<Rl>(ny, nx, op, twy, batch, s);
}

cudaError_t ns_begin(void *fs, int64_t batch, int *ctl, int n, cudaStream_t s)
{
    k_ns_begin<<<unsigned((batch + 255) / 256), 256, 0, s>>>(static_cast<NsField *>(fs), batch, ctl, n);
    return cudaGetLastError();
}

cudaError_t ns_decide(void *fs, const double *partials, int64_t groups, int64_t batch, int *ctl, double parseval,
                      double tol, int max_iter, bool restart_at_end, bool last, bool use_graph,
                      cudaGraphConditionalHandle h, cudaStream_t s)
{
    return launch_chain(k_ns_decide, unsigned(batch), NS_DECIDE_THREADS, 0, s, static_cast<NsField *>(fs), partials,
                        groups, batch, ctl, parseval, tol, max_iter, restart_at_end ? 1 : 0, last ? 1 : 0,
                        use_graph ? 1 : 0, h);
}

size_t ns_field_bytes() { return sizeof(NsField); }

#define PSS_INST(Rl)                                                                                         \
    template cudaError_t ns_row_pass<Rl>(V2<Rl> *, V2<Rl> *, const void *, int64_t, int64_t, int64_t,       \
                                         const int *, const TW<Rl> *, cudaStream_t, bool, bool, bool);       \
    template cudaError_t ns_col_pass<Rl>(V2<Rl> *, V2<Rl> *, V2<Rl> *const[3], V2<Rl> *, void *, double *,  \
                                         const Rl *, const Rl *, const Rl *, const Rl *, const Rl *,         \
                                         const Rl *, double, double, int64_t, int64_t, int64_t,             \
                                         const int *, int, const TW<Rl> *, int *, cudaStream_t, bool,       \
                                         int64_t);                                                           \
    template cudaError_t ns_prep_pass<Rl>(V2<Rl> *const[3], const void *, V2<Rl> *, V2<Rl> *, const Rl *,     \
                                          const Rl *,                                                         \
                                          const Rl *, const Rl *, int64_t, int64_t, int64_t, const int *,    \
                                          const TW<Rl> *, cudaStream_t, int64_t);
PSS_INST(float)
PSS_INST(double)

}  // namespace pss
