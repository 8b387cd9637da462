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
    const bool idle = ctl[NS_CTL_MORE] == 0;
    const int64_t f = blockIdx.x;
    NsField s = fs[f];
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

template <class Rl>
cudaError_t ns_row_pass(V2<Rl> *c1, V2<Rl> *c2, const void *fs, int64_t nx, int64_t ny, int64_t batch,
                        const int *ctl, const TW<Rl> *twx, cudaStream_t s, bool dealias, bool half)
{
    int lgy = 0;
    while ((int64_t(1) << lgy) < ny) ++lgy;  // ny is a power of two
    return launch_row<Rl>(nx, ny, NsRow<Rl>{c1, c2, static_cast<const NsField *>(fs), lgy, dealias ? 1 : 0, half ? 1 : 0,
                                            ctl},
                          twx, batch, s);
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
                                         const int *, const TW<Rl> *, cudaStream_t, bool, bool);             \
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
