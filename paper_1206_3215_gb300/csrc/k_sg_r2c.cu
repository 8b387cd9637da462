// Sine-Gordon step on half spectra (kernel in k_sg_r2c.cuh), and the copies
// between half and full spectra.
#include <algorithm>

#include "k_sg_r2c.cuh"

namespace pss {

namespace {

// half spectrum <-> full spectrum of real fields ([ny][n] <-> [ny][sx])
template <class Rl>
__global__ void k_pack_half(const V2<Rl> *__restrict__ full, V2<Rl> *__restrict__ half, int64_t n, int64_t ny,
                            int64_t sx, int64_t total)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t x = i % sx, r = i / sx;  // r = field * ny + y
        half[i] = x <= n / 2 ? full[r * n + x] : V2<Rl>{Rl(0), Rl(0)};
    }
}

// full(y, x) = half(y, x) for x <= n/2, conj half(-y mod ny, n - x) otherwise
template <class Rl>
__global__ void k_unpack_half(const V2<Rl> *__restrict__ half, V2<Rl> *__restrict__ full, int64_t n, int64_t ny,
                              int64_t sx, int64_t total)
{
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += int64_t(gridDim.x) * blockDim.x) {
        const int64_t x = i % n, r = i / n, y = r % ny, f = r / ny;
        if (x <= n / 2) {
            full[i] = half[r * sx + x];
        } else {
            const V2<Rl> c = half[(f * ny + (ny - y) % ny) * sx + (n - x)];
            full[i] = V2<Rl>{c.x, -c.y};
        }
    }
}

}  // namespace

template <class Rl>
cudaError_t sg_row_pass_r2c(V2<Rl> *h, int64_t nx, int64_t sx, int64_t ny, int64_t batch, const TW<Rl> *twm,
                            const TW<Rl> *twn, cudaStream_t s)
{
    return half_rows<Rl, HalfRow::STEP>({h, nullptr, nullptr, nullptr, sx, Rl(0), Rl(0), Rl(0), Rl(0)}, nx, ny, batch, twm, twn, s);
}

template <class Rl>
cudaError_t pack_half(const V2<Rl> *full, V2<Rl> *half, int64_t nx, int64_t ny, int64_t sx, int64_t batch,
                      cudaStream_t s)
{
    const int64_t total = sx * ny * batch;
    const unsigned blocks = unsigned(std::min<int64_t>((total + 255) / 256, 4096));
    k_pack_half<Rl><<<blocks, 256, 0, s>>>(full, half, nx, ny, sx, total);
    return cudaGetLastError();
}

template <class Rl>
cudaError_t unpack_half(const V2<Rl> *half, V2<Rl> *full, int64_t nx, int64_t ny, int64_t sx, int64_t batch,
                        cudaStream_t s)
{
    const int64_t total = nx * ny * batch;
    const unsigned blocks = unsigned(std::min<int64_t>((total + 255) / 256, 4096));
    k_unpack_half<Rl><<<blocks, 256, 0, s>>>(half, full, nx, ny, sx, total);
    return cudaGetLastError();
}

#define PSS_INST(Rl)                                                                                        \
    template cudaError_t sg_row_pass_r2c<Rl>(V2<Rl> *, int64_t, int64_t, int64_t, int64_t, const TW<Rl> *, \
                                             const TW<Rl> *, cudaStream_t);                                 \
    template cudaError_t pack_half<Rl>(const V2<Rl> *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,        \
                                       cudaStream_t);                                                       \
    template cudaError_t unpack_half<Rl>(const V2<Rl> *, V2<Rl> *, int64_t, int64_t, int64_t, int64_t,      \
                                         cudaStream_t);
PSS_INST(float)
PSS_INST(double)

}  // namespace pss
