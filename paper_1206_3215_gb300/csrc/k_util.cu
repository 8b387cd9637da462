// Elementwise helpers for state set-up and read-back (off the stepping path).
#include "fft_core.cuh"

namespace pss {

// copy every field's current vorticity (buffer fs[f].idx) into dst
struct NsFieldView {
    int idx, active, nonconv, k;
    long long updates;
    int left, pad;
};
template <class Rl>
__global__ void k_ns_gather(const NsFieldView *fs, const V2<Rl> *w0, const V2<Rl> *w1, const V2<Rl> *w2,
                            V2<Rl> *dst, int64_t per_field, int64_t n)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const int b = fs[i / per_field].idx;
        dst[i] = (b == 0 ? w0 : b == 1 ? w1 : w2)[i];
    }
}

// dst = a - c b (complex)
template <class Rl> __global__ void k_axpy(const V2<Rl> *a, const V2<Rl> *b, Rl c, V2<Rl> *dst, int64_t n)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        dst[i] = V2<Rl>{a[i].x - c * b[i].x, a[i].y - c * b[i].y};
}

// spectrum *= keepx[x] keepy[y] (the 2/3 rule mask, 0 or 1)
template <class Rl>
__global__ void k_mask(V2<Rl> *a, const Rl *keepx, const Rl *keepy, int64_t nx, int64_t ny, int64_t n)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
        const Rl m = keepx[i % nx] * keepy[(i / nx) % ny];
        a[i] = V2<Rl>{a[i].x * m, a[i].y * m};
    }
}

template <class Rl> __global__ void k_masked_columns(const V2<Rl> *a, const Rl *keepx, int64_t nx, int64_t n, int *found)
{
    bool any = false;  // (NaN counts)
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
        if (keepx[i % nx] == Rl(0)) any = any || a[i].x != Rl(0) || a[i].y != Rl(0);
    if (any) atomicOr(found, 1);
}

static unsigned blocks_for(int64_t n) { return unsigned(n / 256 + 1 < 4096 ? n / 256 + 1 : 4096); }

template <class Rl>
cudaError_t ns_gather(const void *fs, V2<Rl> *const w[3], V2<Rl> *dst, int64_t per_field, int64_t batch,
                      cudaStream_t s)
{
    const int64_t n = per_field * batch;
    k_ns_gather<Rl><<<blocks_for(n), 256, 0, s>>>(static_cast<const NsFieldView *>(fs), w[0], w[1], w[2], dst,
                                                 per_field, n);
    return cudaGetLastError();
}

template <class Rl> cudaError_t cplx_axpy(const V2<Rl> *a, const V2<Rl> *b, Rl c, V2<Rl> *dst, int64_t n, cudaStream_t s)
{
    k_axpy<Rl><<<blocks_for(n), 256, 0, s>>>(a, b, c, dst, n);
    return cudaGetLastError();
}
template <class Rl>
cudaError_t apply_mask(V2<Rl> *a, const Rl *keepx, const Rl *keepy, int64_t nx, int64_t ny, int64_t batch, cudaStream_t s)
{
    const int64_t n = nx * ny * batch;
    k_mask<Rl><<<blocks_for(n), 256, 0, s>>>(a, keepx, keepy, nx, ny, n);
    return cudaGetLastError();
}

template <class Rl>
cudaError_t masked_columns(const V2<Rl> *a, const Rl *keepx, int64_t nx, int64_t n, int *found, cudaStream_t s)
{
    k_masked_columns<Rl><<<blocks_for(n), 256, 0, s>>>(a, keepx, nx, n, found);
    return cudaGetLastError();
}

#define PSS_INST(Rl)                                                                                      \
    template cudaError_t cplx_axpy<Rl>(const V2<Rl> *, const V2<Rl> *, Rl, V2<Rl> *, int64_t, cudaStream_t); \
    template cudaError_t masked_columns<Rl>(const V2<Rl> *, const Rl *, int64_t, int64_t, int *, cudaStream_t); \
    template cudaError_t apply_mask<Rl>(V2<Rl> *, const Rl *, const Rl *, int64_t, int64_t, int64_t, cudaStream_t); \
    template cudaError_t ns_gather<Rl>(const void *, V2<Rl> *const[3], V2<Rl> *, int64_t, int64_t, cudaStream_t);
PSS_INST(float)
PSS_INST(double)

}  // namespace pss
