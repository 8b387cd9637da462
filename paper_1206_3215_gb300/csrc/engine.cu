// Stepping drivers: which passes run, in which order, on which buffers.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "engine.h"
#include "plan.h"
#include "tables.h"

using namespace pss;

namespace {
// the device status word pass kernels report a lost tile copy in
int *pass_status(pss_grid *g) { return reinterpret_cast<int *>(g->flags) + FLAG_SLOT_PASS_STATUS; }
}  // namespace

namespace {

template <class Rl> V2<Rl> *B(pss_grid *g, int i) { return static_cast<V2<Rl> *>(g->buf[i]); }
template <class Rl> const V2<Rl> *C(const void *p) { return static_cast<const V2<Rl> *>(p); }
template <class Rl> const TW<Rl> *Tw(const void *p) { return static_cast<const TW<Rl> *>(p); }

cudaMemcpyKind kind_in(int where) { return where == PSS_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice; }
cudaMemcpyKind kind_out(int where) { return where == PSS_HOST ? cudaMemcpyDeviceToHost : cudaMemcpyDeviceToDevice; }

// The range [base, base + size) of the device allocation (or mapping) that holds
// p, by the driver's cuMemGetAddressRange (looked up once through the runtime:
// the library does not link the driver library); false where it has none.
bool address_range(const void *p, uintptr_t *base, size_t *size)
{
    using Range = CUresult (*)(CUdeviceptr *, size_t *, CUdeviceptr);
    static const Range range = []() -> Range {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q{};
        const cudaError_t e = cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &fn, 12000, cudaEnableDefault, &q);
        if (e != cudaSuccess) cudaGetLastError();
        return (e == cudaSuccess && q == cudaDriverEntryPointSuccess) ? reinterpret_cast<Range>(fn) : nullptr;
    }();
    CUdeviceptr b = 0;
    if (!range || range(&b, size, reinterpret_cast<CUdeviceptr>(p)) != CUDA_SUCCESS) return false;
    *base = uintptr_t(b);
    return true;
}

// How the library reaches `bytes` bytes of a caller's device array.  DIRECT: a
// kernel may read or write it: memory of the current device (or managed), inside
// one allocation, aligned for the kernel's widest access.  SHORT: no memory
// follows where the array would go on; the call is refused, as a copy of that
// size would be (a kernel would fault).  COPY: anything else goes through a
// copy, which reports what it cannot do.
enum class Access { DIRECT, COPY, SHORT };
Access kernel_access(const void *p, size_t align, size_t bytes)
{
    auto on_device = [](uintptr_t q) {
        cudaPointerAttributes at;
        if (cudaPointerGetAttributes(&at, reinterpret_cast<const void *>(q)) != cudaSuccess) {
            cudaGetLastError();
            return false;
        }
        int dev = -1;
        return cudaGetDevice(&dev) == cudaSuccess && at.device == dev &&
               (at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged);
    };
    const uintptr_t a = reinterpret_cast<uintptr_t>(p);
    uintptr_t base = 0;
    size_t size = 0;
    if (!on_device(a) || !address_range(p, &base, &size)) return Access::COPY;
    if (bytes <= base + size - a) return a % align ? Access::COPY : Access::DIRECT;
    for (uintptr_t q = base + size; q - a < bytes; q = base + size)
        if (!on_device(q) || !address_range(reinterpret_cast<const void *>(q), &base, &size)) return Access::SHORT;
    return Access::COPY;
}

int short_array(pss_grid *g, const char *what, size_t bytes)
{
    return g->fail(PSS_E_CUDA, "%s: the device array is shorter than %zu bytes", what, bytes);
}

// Upload a per-axis table of n complex values given by f(m) -> (re, im) in FP64,
// in the twiddle layout of the grid's precision (FP32: hi + lo quadruples).
template <class F> int upload_cplx_table(pss_grid *g, int64_t n, F f, void **dst)
{
    if (g->p.precision == PSS_FP32) {
        std::vector<float> t(4 * n);
        for (int64_t m = 0; m < n; ++m) {
            double re, im;
            f(m, &re, &im);
            hilo_f32(re, im, &t[4 * m]);
        }
        return g->upload(dst, t.data(), t.size() * 4);
    }
    std::vector<double> t(2 * n);
    for (int64_t m = 0; m < n; ++m) f(m, &t[2 * m], &t[2 * m + 1]);
    return g->upload(dst, t.data(), t.size() * 8);
}

int upload_twiddles(pss_grid *g, int64_t n, void **dst)
{
    if (g->p.precision == PSS_FP32) {
        auto t = twiddles_f32(n);
        return g->upload(dst, t.data(), t.size() * 4);
    }
    auto t = twiddles_f64(n);
    return g->upload(dst, t.data(), t.size() * 8);
}

template <class Rl> int upload_real(pss_grid *g, const std::vector<double> &v, void **dst)
{
    std::vector<Rl> r(v.begin(), v.end());
    return g->upload(dst, r.data(), r.size() * sizeof(Rl));
}

}  // namespace

// ----------------------------------------------------------------------------

int pss_grid::init()
{
    nx = p.nx;
    ny = p.ny;
    batch = p.batch;
    npts = nx * ny;
    ntot = npts * batch;
    esz = p.precision == PSS_FP32 ? 8 : 16;
    int rc;
    if ((rc = cuda(cudaGetDevice(&dev), "cudaGetDevice"))) return rc;
    if (p.stream) {
        stream = static_cast<cudaStream_t>(p.stream);
    } else {
        if ((rc = cuda(cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking), "stream"))) return rc;
        own_stream = true;
    }
    {
        const char *gr = getenv("PSS_GRAPHS");
        use_graphs = !(gr && gr[0] == '0');
    }
    // work arrays
    nbuf = p.eq == PSS_EQ_NLS ? 3 : p.eq == PSS_EQ_SG ? 5 : 7;
    for (int i = 0; i < nbuf; ++i) {
        if ((rc = alloc(&buf[i], field_bytes()))) return rc;
        if ((rc = cuda(cudaMemset(buf[i], 0, field_bytes()), "memset"))) return rc;
    }
    // tables
    if ((rc = upload_twiddles(this, nx, &twx))) return rc;
    if ((rc = upload_twiddles(this, ny, &twy))) return rc;
    std::vector<double> kx2v(nx), ky2v(ny), kxov(nx), kyov(ny), kpx(nx), kpy(ny);
    for (int64_t m = 0; m < nx; ++m) {
        const double k = wavenumber(m, nx, p.lx);
        kx2v[m] = k * k;
        kxov[m] = (m == nx / 2) ? 0.0 : k;
        kpx[m] = (!p.dealias || 3 * std::llabs(m < nx / 2 ? m : m - nx) < nx) ? 1.0 : 0.0;
    }
    for (int64_t m = 0; m < ny; ++m) {
        const double k = wavenumber(m, ny, p.ly);
        ky2v[m] = k * k;
        kyov[m] = (m == ny / 2) ? 0.0 : k;
        kpy[m] = (!p.dealias || 3 * std::llabs(m < ny / 2 ? m : m - ny) < ny) ? 1.0 : 0.0;
    }
    if ((rc = upload((void **)&kx2d, kx2v.data(), nx * 8))) return rc;
    if ((rc = upload((void **)&ky2d, ky2v.data(), ny * 8))) return rc;
    if (p.precision == PSS_FP32) {
        if ((rc = upload_real<float>(this, kx2v, &kx2)) || (rc = upload_real<float>(this, ky2v, &ky2)) ||
            (rc = upload_real<float>(this, kxov, &kxo)) || (rc = upload_real<float>(this, kyov, &kyo)) ||
            (rc = upload_real<float>(this, kpx, &keepx)) || (rc = upload_real<float>(this, kpy, &keepy)))
            return rc;
    } else {
        if ((rc = upload_real<double>(this, kx2v, &kx2)) || (rc = upload_real<double>(this, ky2v, &ky2)) ||
            (rc = upload_real<double>(this, kxov, &kxo)) || (rc = upload_real<double>(this, kyov, &kyo)) ||
            (rc = upload_real<double>(this, kpx, &keepx)) || (rc = upload_real<double>(this, kpy, &keepy)))
            return rc;
    }
    if (p.eq == PSS_EQ_NS && p.rfft) {
        ns_half = true;
        nsx = nx / 2 + 8;  // a multiple of every column-tile width
    }
    if (p.eq == PSS_EQ_SG && p.rfft) {
        half = true;
        sx = nx / 2 + 8;  // a multiple of every column-tile width
        const size_t hb = size_t(sx) * size_t(ny) * size_t(batch) * esz;
        for (int i = 0; i < 3; ++i) {
            if ((rc = alloc(&hbuf[i], hb))) return rc;
            if ((rc = cuda(cudaMemset(hbuf[i], 0, hb), "memset"))) return rc;
        }
        if ((rc = upload_twiddles(this, nx / 2, &twm))) return rc;
        std::vector<double> kh(sx, 0.0);
        for (int64_t m = 0; m <= nx / 2; ++m) kh[m] = kx2v[m];
        if ((rc = p.precision == PSS_FP32 ? upload_real<float>(this, kh, &kx2h) : upload_real<double>(this, kh, &kx2h)))
            return rc;
    }
    if (p.eq == PSS_EQ_SG && p.precision == PSS_FP32) {
        // (dt^2/2) k^2 per axis as {hi, lo} (start-up)
        auto halves = [&](const std::vector<double> &k2, void **dst) {
            std::vector<float> t(2 * k2.size());
            for (size_t m = 0; m < k2.size(); ++m) {
                const double c = 0.5 * p.dt * p.dt * k2[m];
                t[2 * m] = float(c);
                t[2 * m + 1] = float(c - double(float(c)));
            }
            return upload(dst, t.data(), t.size() * 4);
        };
        if ((rc = halves(kx2v, &sgcx)) || (rc = halves(ky2v, &sgcy))) return rc;
    }
    if (p.eq == PSS_EQ_NLS) {
        // exp(-i k^2 tau) - 1 = (-2 sin^2(k^2 tau / 2), -sin(k^2 tau)) per axis,
        // tau = dt/2 (index 0) and dt (index 1); no cancellation for small k
        for (int h = 0; h < 2; ++h) {
            const double tau = h == 0 ? 0.5 * p.dt : p.dt;
            auto km1 = [](double ph, double *re, double *im) {
                const double sh = std::sin(0.5 * ph);
                *re = -2.0 * sh * sh;
                *im = -std::sin(ph);
            };
            auto fx = [&](int64_t m, double *re, double *im) { km1(kx2v[m] * tau, re, im); };
            auto fy = [&](int64_t m, double *re, double *im) { km1(ky2v[m] * tau, re, im); };
            if ((rc = upload_cplx_table(this, nx, fx, &ax[h]))) return rc;
            if ((rc = upload_cplx_table(this, ny, fy, &by[h]))) return rc;
        }
    }
    if ((rc = upload_tables())) return rc;
    // reductions
    const size_t parts = size_t(batch) * 3 * std::max<int64_t>(RED_BLOCKS, nx);
    if ((rc = alloc((void **)&partials, parts * 8))) return rc;
    if ((rc = alloc((void **)&sums, size_t(batch) * 3 * 8))) return rc;
    // NS: the per-tile words of the split column pass follow the 64-byte block
    const size_t flag_bytes = 64 + (p.eq == PSS_EQ_NS ? size_t(batch) * size_t(nx) * 4 : 0);
    if ((rc = alloc((void **)&flags, flag_bytes))) return rc;
    if ((rc = cuda(cudaMemset(flags, 0, flag_bytes), "memset"))) return rc;
    void *hp = nullptr;
    if ((rc = cuda(cudaMallocHost(&hp, size_t(batch) * 3 * 8 + 64), "cudaMallocHost"))) return rc;
    owned_host.push_back(hp);
    host_sums = static_cast<double *>(hp);
    host_flags = reinterpret_cast<unsigned *>(static_cast<char *>(hp) + size_t(batch) * 3 * 8);
    if (p.eq == PSS_EQ_NS) {
        if ((rc = alloc(&ns_field, size_t(batch) * ns_field_bytes()))) return rc;
        if ((rc = cuda(cudaMemset(ns_field, 0, size_t(batch) * ns_field_bytes()), "memset"))) return rc;
        if ((rc = cuda(cudaMallocHost(&hp, size_t(batch) * ns_field_bytes()), "cudaMallocHost"))) return rc;
        owned_host.push_back(hp);
        host_fields = hp;
    }
    return cuda(cudaDeviceSynchronize(), "init sync");
}

int pss_grid::sync()
{
    int rc = cuda(cudaStreamSynchronize(stream), "stream sync");
    if (rc) return rc;
    if ((rc = check_pass_status())) return rc;
    if ((rc = check_ns_nonconv())) return rc;
    if (nonconv_pending) {
        nonconv_pending = false;
        return fail(PSS_E_NOT_CONVERGED, "NS fixed point reached max_iter=%d", p.max_iter);
    }
    return PSS_OK;
}

namespace pss {
PlanTuning *plan_tuning()
{
    thread_local PlanTuning t;
    return &t;
}
std::atomic<int> &plan_epoch()
{
    static std::atomic<int> e{0};
    return e;
}
}  // namespace pss

int pss_grid::pass_begin(int kind)
{
    ++launches;
    plan_tuning()->open_kind = kind;
    if (!profiling) return PSS_OK;
    prof_open = sampled(prof_pass++);
    if (!prof_open) return PSS_OK;
    if (capturing) {
        // a profiling graph: an event pair around each timed pass; the graph
        // owns its events
        cudaEvent_t e;
        int rc = cuda(cudaEventCreate(&e), "event create");
        if (rc) return rc;
        capturing->evs.push_back(e);
        capturing->kinds.push_back(kind);
        // External: a node of the graph that records the event when it runs
        // (a plain record during capture only orders the captured work)
        return cuda(cudaEventRecordWithFlags(e, stream, cudaEventRecordExternal), "event record");
    }
    while (ev_pool.size() < ev_used + 2) {
        cudaEvent_t e;
        int rc = cuda(cudaEventCreate(&e), "event create");
        if (rc) return rc;
        ev_pool.push_back(e);
    }
    ev_kind.push_back(kind);
    return cuda(cudaEventRecord(ev_pool[ev_used++], stream), "event record");
}

int pss_grid::pass_end()
{
    plan_tuning()->open_kind = -1;
    if (!profiling || !prof_open) return PSS_OK;
    prof_open = false;
    if (capturing) {
        cudaEvent_t e;
        int rc = cuda(cudaEventCreate(&e), "event create");
        if (rc) return rc;
        capturing->evs.push_back(e);
        return cuda(cudaEventRecordWithFlags(e, stream, cudaEventRecordExternal), "event record");
    }
    return cuda(cudaEventRecord(ev_pool[ev_used++], stream), "event record");
}

int pss_grid::profile_resolve()
{
    int rc = cuda(cudaStreamSynchronize(stream), "profile sync");
    if (rc) return rc;
    if (prof_pending) {
        // timed pass i of the graph ran between its events 2i and 2i + 1
        const StepGraph &g = *prof_pending;
        prof_pending = nullptr;
        for (size_t i = 0; i < g.kinds.size() && 2 * i + 1 < g.evs.size(); ++i) {
            float ms = 0.f;
            if ((rc = cuda(cudaEventElapsedTime(&ms, g.evs[2 * i], g.evs[2 * i + 1]), "elapsed"))) return rc;
            prof_ms[g.kinds[i]] += ms;
            prof_n[g.kinds[i]] += 1;
        }
    }
    for (size_t i = 0; i < ev_kind.size(); ++i) {
        float ms = 0.f;
        if ((rc = cuda(cudaEventElapsedTime(&ms, ev_pool[2 * i], ev_pool[2 * i + 1]), "elapsed"))) return rc;
        prof_ms[ev_kind[i]] += ms;
        prof_n[ev_kind[i]] += 1;
    }
    ev_kind.clear();
    ev_used = 0;
    return PSS_OK;
}

// per-field fixed-point record as written by the NS kernels
struct NsFieldHost {
    int idx, active, nonconv, k;
    long long updates;
    int left, pad;
};

int pss_grid::ns_update_count(int64_t *n)
{
    *n = 0;
    if (p.eq != PSS_EQ_NS || !has_state) return PSS_OK;
    int rc = cuda(cudaMemcpyAsync(host_fields, ns_field, size_t(batch) * ns_field_bytes(), cudaMemcpyDeviceToHost,
                                  stream), "fields copy");
    if (rc || (rc = cuda(cudaStreamSynchronize(stream), "sync"))) return rc;
    const NsFieldHost *f = static_cast<const NsFieldHost *>(host_fields);
    for (int64_t i = 0; i < batch; ++i) *n += f[i].updates;
    return PSS_OK;
}

// Report (and clear) fields that reached max_iter since the last check.
// a pass kernel that gave up waiting for a tile copy left its tiles
// unfinished: the state is no longer valid
int pss_grid::check_pass_status()
{
    int *dev_slot = reinterpret_cast<int *>(flags) + pss::FLAG_SLOT_PASS_STATUS;
    int *host_slot = reinterpret_cast<int *>(host_flags) + pss::FLAG_SLOT_PASS_STATUS;
    int rc = cuda(cudaMemcpyAsync(host_slot, dev_slot, sizeof(int), cudaMemcpyDeviceToHost, stream), "status copy");
    if (rc || (rc = cuda(cudaStreamSynchronize(stream), "sync"))) return rc;
    if (*host_slot == 0) return PSS_OK;
    *host_slot = 0;
    if ((rc = cuda(cudaMemsetAsync(dev_slot, 0, sizeof(int), stream), "status reset"))) return rc;
    has_state = false;
    drop_graphs();  // captured launches are rebuilt by the next step
    return fail(PSS_E_CUDA, "a column-pass tile copy did not arrive in time; the state is lost (set it again)");
}

int pss_grid::check_ns_nonconv()
{
    if (p.eq != PSS_EQ_NS || !has_state) return PSS_OK;
    const size_t bytes = size_t(batch) * ns_field_bytes();
    int rc = cuda(cudaMemcpyAsync(host_fields, ns_field, bytes, cudaMemcpyDeviceToHost, stream), "fields copy");
    if (rc || (rc = cuda(cudaStreamSynchronize(stream), "sync"))) return rc;
    NsFieldHost *h = static_cast<NsFieldHost *>(host_fields);
    bool nc = false;
    for (int64_t i = 0; i < batch; ++i) {
        nc = nc || h[i].nonconv;
        h[i].nonconv = 0;
    }
    if (!nc) return PSS_OK;
    if ((rc = cuda(cudaMemcpyAsync(ns_field, h, bytes, cudaMemcpyHostToDevice, stream), "fields copy")) ||
        (rc = cuda(cudaStreamSynchronize(stream), "sync")))
        return rc;
    return fail(PSS_E_NOT_CONVERGED, "NS fixed point reached max_iter=%d", p.max_iter);
}

// ----------------------------------------------------------------------------
// NLS: state buf[0] = row transform of psi (unnormalised); buf[1], buf[2] scratch.

namespace {

// fields f .. f + nb - 1 from the caller's array: straight through the row
// transform where a kernel can read it, else copied first
template <class Rl> int nls_set(pss_grid *g, int64_t f, int64_t nb, const void *a, int where)
{
    V2<Rl> *dst = B<Rl>(g, 0) + f * g->npts;
    const V2<Rl> *src = dst;
    const size_t bytes = size_t(nb * g->npts) * g->esz;
    const Access ac = where == PSS_DEVICE ? kernel_access(a, sizeof(V2<Rl>), bytes) : Access::COPY;
    int rc;
    if (ac == Access::SHORT) return short_array(g, "set_state", bytes);
    if (ac == Access::DIRECT)
        src = C<Rl>(a);
    else if ((rc = g->cuda(cudaMemcpyAsync(dst, a, bytes, kind_in(where), g->stream), "set_state copy")))
        return rc;
    rc = g->cuda(fft_rows<Rl>(src, dst, g->nx, g->ny, nb, -1, Rl(1), Tw<Rl>(g->twx), g->stream), "set_state row fft");
    if (rc) return rc;
    if (where == PSS_HOST) return g->cuda(cudaStreamSynchronize(g->stream), "set_state sync");
    return PSS_OK;
}

template <class Rl> int nls_step(pss_grid *g, int64_t n)
{
    const Rl s_mid = Rl(1.0 / (double(g->nx) * double(g->ny)));  // exact: powers of two
    const Rl s_end = Rl(1.0 / double(g->ny));
    const Rl sdt = Rl(g->p.sigma * g->p.dt);
    auto col = [&](int full, Rl scale) {
        return nls_col_pass<Rl>(B<Rl>(g, 0), g->nx, g->ny, g->batch, scale, Tw<Rl>(g->ax[full]),
                                Tw<Rl>(g->by[full]), Tw<Rl>(g->twy), pass_status(g), g->stream);
    };
    if (n == 0) return PSS_OK;
    int rc;
    if ((rc = g->pass_begin(1))) return rc;
    cudaError_t e = col(0, s_mid);
    if ((rc = g->pass_end())) return rc;
    for (int64_t i = 0; i < n && e == cudaSuccess; ++i) {
        if ((rc = g->pass_begin(0))) return rc;
        e = nls_row_pass<Rl>(B<Rl>(g, 0), g->nx, g->ny, g->batch, sdt, Tw<Rl>(g->twx), g->stream);
        if ((rc = g->pass_end())) return rc;
        if (e != cudaSuccess) break;
        const bool last = (i + 1 == n);
        if ((rc = g->pass_begin(1))) return rc;
        e = col(last ? 0 : 1, last ? s_end : s_mid);
        if ((rc = g->pass_end())) return rc;
    }
    return g->cuda(e, "nls step");
}

// psi (physical) of fields f .. f + nb - 1 into dst
template <class Rl> int nls_physical(pss_grid *g, int64_t f, int64_t nb, V2<Rl> *dst)
{
    return g->cuda(fft_rows<Rl>(B<Rl>(g, 0) + f * g->npts, dst, g->nx, g->ny, nb, +1, Rl(1.0 / double(g->nx)),
                                Tw<Rl>(g->twx), g->stream),
                   "row inverse");
}

template <class Rl> int nls_get(pss_grid *g, int64_t f, int64_t nb, void *a, int where)
{
    const size_t bytes = size_t(nb * g->npts) * g->esz;
    const Access ac = where == PSS_DEVICE ? kernel_access(a, sizeof(V2<Rl>), bytes) : Access::COPY;
    if (ac == Access::SHORT) return short_array(g, "get_state", bytes);
    V2<Rl> *dst = ac == Access::DIRECT ? static_cast<V2<Rl> *>(a) : B<Rl>(g, 1) + f * g->npts;
    int rc = nls_physical<Rl>(g, f, nb, dst);
    if (!rc && ac == Access::COPY)
        rc = g->cuda(cudaMemcpyAsync(a, dst, bytes, kind_out(where), g->stream), "get_state copy");
    return rc ? rc : g->sync();
}

template <class Rl> int nls_conserved(pss_grid *g, double *out)
{
    int rc = nls_physical<Rl>(g, 0, g->batch, B<Rl>(g, 1));
    if (rc) return rc;
    rc = g->cuda(fft_cols<Rl>(B<Rl>(g, 0), B<Rl>(g, 2), g->nx, g->ny, g->batch, -1, Rl(1), Tw<Rl>(g->twy), g->stream),
                 "col fft");
    if (rc) return rc;
    rc = g->cuda(nls_sums<Rl>(B<Rl>(g, 1), B<Rl>(g, 2), g->nx, g->ny, g->batch, g->kx2d, g->ky2d, g->partials,
                              g->sums, g->stream),
                 "nls sums");
    if (rc) return rc;
    rc = g->cuda(cudaMemcpyAsync(g->host_sums, g->sums, size_t(g->batch) * 3 * 8, cudaMemcpyDeviceToHost, g->stream),
                 "sums copy");
    if (rc) return rc;
    if ((rc = g->sync())) return rc;
    const double dA = g->dA(), inv_n = 1.0 / (double(g->nx) * double(g->ny));
    bool finite = true;
    for (int64_t f = 0; f < g->batch; ++f) {
        const double *s = g->host_sums + 3 * f;
        out[2 * f] = dA * s[0];
        out[2 * f + 1] = dA * (0.5 * s[2] * inv_n + 0.25 * g->p.sigma * s[1]);
        finite = finite && std::isfinite(out[2 * f]) && std::isfinite(out[2 * f + 1]);
    }
    return finite ? PSS_OK : g->fail(PSS_E_NONFINITE, "non-finite NLS invariant");
}

}  // namespace

// ----------------------------------------------------------------------------
// shared helpers

namespace {

template <class Rl> const Rl *Rt(const void *p) { return static_cast<const Rl *>(p); }

int finish_sums(pss_grid *g)
{
    int rc = g->cuda(cudaMemcpyAsync(g->host_sums, g->sums, size_t(g->batch) * 3 * 8, cudaMemcpyDeviceToHost,
                                     g->stream), "sums copy");
    return rc ? rc : g->sync();
}

}  // namespace

// ----------------------------------------------------------------------------
// Sine-Gordon: buf[0] = uhat^n, buf[1] = d^n = uhat^n - uhat^{n-1},
// buf[2] = H (column inverse transform of uhat^n / (nx ny)); buf[3], buf[4] scratch.

namespace {

// The state arrays of fields f .. f + nb - 1: the half spectra where the grid
// steps those, else the full ones; w columns per row.
template <class Rl> struct SgState {
    V2<Rl> *u, *d, *h;
    int64_t w, f, nb;
};
template <class Rl> SgState<Rl> sg_state(pss_grid *g, int64_t f, int64_t nb)
{
    const int64_t w = g->half ? g->sx : g->nx, o = f * w * g->ny;
    void *const *b = g->half ? g->hbuf : g->buf;
    return {static_cast<V2<Rl> *>(b[0]) + o, static_cast<V2<Rl> *>(b[1]) + o, static_cast<V2<Rl> *>(b[2]) + o, w, f,
            nb};
}
// scratch array i (3 or 4) of the fields, nb * npts complex points
template <class Rl> V2<Rl> *sg_scratch(pss_grid *g, const SgState<Rl> &st, int i) { return B<Rl>(g, i) + st.f * g->npts; }

template <class Rl> Rl sg_scale(pss_grid *g) { return Rl(1.0 / (double(g->nx) * double(g->ny))); }

// H from uhat: the same scaling and transform as the step's column pass
template <class Rl> int sg_make_h(pss_grid *g, const SgState<Rl> &st)
{
    return g->cuda(sg_level_cols<Rl>(st.u, st.h, sg_scale<Rl>(g), st.w, g->ny, st.nb, Tw<Rl>(g->twy), g->stream), "H");
}

// A caller's real array as a kernel reads it: the array itself where it can be,
// else a copy in `tmp`.
template <class Rl> int real_in(pss_grid *g, const void *src, int where, Rl *tmp, int64_t n, const Rl **out)
{
    const size_t bytes = size_t(n) * sizeof(Rl);
    const Access ac = where == PSS_DEVICE ? kernel_access(src, sizeof(Rl), bytes) : Access::COPY;
    if (ac == Access::SHORT) return short_array(g, "state", bytes);
    *out = ac == Access::DIRECT ? static_cast<const Rl *>(src) : tmp;
    if (ac == Access::DIRECT) return PSS_OK;
    return g->cuda(cudaMemcpyAsync(tmp, src, bytes, kind_in(where), g->stream), "state copy");
}

// row transform of the real fields `a` into dst (rows of st.w)
template <class Rl> cudaError_t sg_split(pss_grid *g, const SgState<Rl> &st, const Rl *a, V2<Rl> *dst)
{
    return rows_from_real<Rl>(a, dst, g->nx, g->half ? g->sx : 0, g->ny, st.nb, Tw<Rl>(g->twx), g->stream);
}

template <class Rl> int sg_set_fields(pss_grid *g, int64_t f, int64_t nb, const void *u0, const void *v0, int where)
{
    const SgState<Rl> st = sg_state<Rl>(g, f, nb);
    const int64_t n = nb * g->npts;
    // scratch: copies of u and v in array 3; sin u, then the transform of v, in array 4
    Rl *copies = reinterpret_cast<Rl *>(sg_scratch<Rl>(g, st, 3)), *sine = reinterpret_cast<Rl *>(sg_scratch<Rl>(g, st, 4));
    V2<Rl> *vh = v0 ? sg_scratch<Rl>(g, st, 4) : nullptr;
    const Rl *u = nullptr, *v = nullptr;
    auto cols = [&](V2<Rl> *a) {
        return fft_cols<Rl>(a, a, st.w, g->ny, nb, -1, Rl(1), Tw<Rl>(g->twy), g->stream);
    };
    int rc;
    if ((rc = real_in<Rl>(g, u0, where, copies, n, &u)) || (v0 && (rc = real_in<Rl>(g, v0, where, copies + n, n, &v))))
        return rc;
    if ((rc = g->cuda(sg_sine<Rl>(u, sine, n, g->stream), "sin u")) ||
        (rc = g->cuda(sg_split<Rl>(g, st, sine, st.d), "forward rows")) ||
        (rc = g->cuda(sg_split<Rl>(g, st, u, st.u), "forward rows")) || (rc = g->cuda(cols(st.u), "forward columns")) ||
        (vh && (rc = g->cuda(sg_split<Rl>(g, st, v, vh), "forward rows"))) ||
        (vh && (rc = g->cuda(cols(vh), "forward columns"))) ||
        (rc = g->cuda(sg_start_cols<Rl>(st.d, st.u, vh, g->p.dt, C<Rl>(g->sgcx), C<Rl>(g->sgcy), g->kx2d, g->ky2d, st.w,
                                        g->ny, nb, Tw<Rl>(g->twy), g->stream), "start-up columns")) ||
        (rc = sg_make_h<Rl>(g, st)))
        return rc;
    return where == PSS_HOST ? g->cuda(cudaStreamSynchronize(g->stream), "set_state sync") : PSS_OK;
}

// both levels from u^n, u^{n-1}: uhat^n = F u^n, d = uhat^n - F u^{n-1}
template <class Rl> int sg_set_levels(pss_grid *g, const void *un, const void *unm1, int where)
{
    const SgState<Rl> st = sg_state<Rl>(g, 0, g->batch);
    const Rl *a = nullptr, *b = nullptr;
    int rc;
    if ((rc = real_in<Rl>(g, un, where, reinterpret_cast<Rl *>(sg_scratch<Rl>(g, st, 3)), g->ntot, &a)) ||
        (rc = real_in<Rl>(g, unm1, where, reinterpret_cast<Rl *>(sg_scratch<Rl>(g, st, 4)), g->ntot, &b)) ||
        (rc = g->cuda(sg_split<Rl>(g, st, a, st.u), "forward rows")) ||
        (rc = g->cuda(sg_split<Rl>(g, st, b, st.d), "forward rows")) ||
        (rc = g->cuda(fft_cols<Rl>(st.u, st.u, st.w, g->ny, st.nb, -1, Rl(1), Tw<Rl>(g->twy), g->stream), "forward columns")) ||
        (rc = g->cuda(fft_cols<Rl>(st.d, st.d, st.w, g->ny, st.nb, -1, Rl(1), Tw<Rl>(g->twy), g->stream), "forward columns")) ||
        (rc = g->cuda(cplx_axpy<Rl>(st.u, st.d, Rl(1), st.d, st.w * g->ny * st.nb, g->stream), "d")) ||
        (rc = sg_make_h<Rl>(g, st)))
        return rc;
    return where == PSS_HOST ? g->cuda(cudaStreamSynchronize(g->stream), "sync") : PSS_OK;
}

// half spectra <-> full spectra of the sine-Gordon state
template <class Rl> int sg_half_sync(pss_grid *g, bool to_half)
{
    int rc;
    const SgState<Rl> st = sg_state<Rl>(g, 0, g->batch);
    if (to_half) {
        if ((rc = g->cuda(pack_half<Rl>(B<Rl>(g, 0), st.u, g->nx, g->ny, g->sx, g->batch, g->stream), "pack")) ||
            (rc = g->cuda(pack_half<Rl>(B<Rl>(g, 1), st.d, g->nx, g->ny, g->sx, g->batch, g->stream), "pack")))
            return rc;
        return sg_make_h<Rl>(g, st);
    }
    if ((rc = g->cuda(unpack_half<Rl>(st.u, B<Rl>(g, 0), g->nx, g->ny, g->sx, g->batch, g->stream), "unpack")) ||
        (rc = g->cuda(unpack_half<Rl>(st.d, B<Rl>(g, 1), g->nx, g->ny, g->sx, g->batch, g->stream), "unpack")))
        return rc;
    return PSS_OK;
}

template <class Rl> int sg_step(pss_grid *g, int64_t n)
{
    int rc;
    if (g->half) {
        V2<Rl> *u = static_cast<V2<Rl> *>(g->hbuf[0]), *d = static_cast<V2<Rl> *>(g->hbuf[1]),
               *h = static_cast<V2<Rl> *>(g->hbuf[2]);
        for (int64_t i = 0; i < n; ++i) {
            if ((rc = g->pass_begin(0))) return rc;
            cudaError_t e = sg_row_pass_r2c<Rl>(h, g->nx, g->sx, g->ny, g->batch, Tw<Rl>(g->twm), Tw<Rl>(g->twx),
                                                g->stream);
            if ((rc = g->pass_end()) || (rc = g->cuda(e, "sg row pass (half spectrum)"))) return rc;
            if ((rc = g->pass_begin(1))) return rc;
            e = sg_col_pass<Rl>(h, u, d, g->sx, g->ny, g->batch, Rt<Rl>(g->kx2h), Rt<Rl>(g->ky2), Rl(g->p.dt),
                                Tw<Rl>(g->twy), pass_status(g), g->stream, g->nx);
            if ((rc = g->pass_end()) || (rc = g->cuda(e, "sg column pass (half spectrum)"))) return rc;
        }
        return PSS_OK;
    }
    for (int64_t i = 0; i < n; ++i) {
        if ((rc = g->pass_begin(0))) return rc;
        cudaError_t e = sg_row_pass<Rl>(B<Rl>(g, 2), g->nx, g->ny, g->batch, Tw<Rl>(g->twx), g->stream);
        if ((rc = g->pass_end()) || (rc = g->cuda(e, "sg row pass"))) return rc;
        if ((rc = g->pass_begin(1))) return rc;
        e = sg_col_pass<Rl>(B<Rl>(g, 2), B<Rl>(g, 0), B<Rl>(g, 1), g->nx, g->ny, g->batch, Rt<Rl>(g->kx2),
                            Rt<Rl>(g->ky2), Rl(g->p.dt), Tw<Rl>(g->twy), pass_status(g), g->stream);
        if ((rc = g->pass_end()) || (rc = g->cuda(e, "sg column pass"))) return rc;
    }
    return PSS_OK;
}

// real fields of the spectra a - b (b may be null) into dst: row pass into
// scratch array 4, column pass into the real array
template <class Rl> int sg_real_of(pss_grid *g, const SgState<Rl> &st, V2<Rl> *a, const V2<Rl> *b, Rl *dst)
{
    V2<Rl> *t = sg_scratch<Rl>(g, st, 4), *const src[3] = {a, a, a};
    int rc = g->cuda(rows_inverse<Rl>(src, nullptr, 0, b, t, g->nx, g->half ? g->sx : 0, g->ny, st.nb, Tw<Rl>(g->twx),
                                      g->stream), "inverse rows");
    if (rc) return rc;
    return g->cuda(cols_to_real<Rl>(t, dst, sg_scale<Rl>(g), g->nx, g->ny, st.nb, Tw<Rl>(g->twy), g->stream),
                   "inverse columns");
}

// u^n -> a, u^{n-1} = F^-1 (uhat - d) -> b (may be null) of fields f .. f + nb - 1
template <class Rl> int sg_get_fields(pss_grid *g, int64_t f, int64_t nb, void *a, void *b, int where)
{
    const SgState<Rl> st = sg_state<Rl>(g, f, nb);
    void *const dst[2] = {a, b};
    const size_t bytes = size_t(nb * g->npts) * sizeof(Rl);
    for (int k = 0; k < 2; ++k) {
        if (!dst[k]) continue;
        const Access ac = where == PSS_DEVICE ? kernel_access(dst[k], sizeof(Rl), bytes) : Access::COPY;
        if (ac == Access::SHORT) return short_array(g, "get_state", bytes);
        Rl *r = ac == Access::DIRECT ? static_cast<Rl *>(dst[k]) : reinterpret_cast<Rl *>(sg_scratch<Rl>(g, st, 3));
        int rc = sg_real_of<Rl>(g, st, st.u, k ? st.d : nullptr, r);
        if (!rc && ac == Access::COPY)
            rc = g->cuda(cudaMemcpyAsync(dst[k], r, bytes, kind_out(where), g->stream), "state copy");
        if (rc) return rc;
    }
    return g->sync();
}

template <class Rl> int sg_conserved(pss_grid *g, double *out)
{
    const SgState<Rl> st = sg_state<Rl>(g, 0, g->batch);
    Rl *X = reinterpret_cast<Rl *>(g->buf[3]), *Y = X + g->ntot;  // u^n, u^n - u^{n-1}
    int rc;
    if ((rc = sg_real_of<Rl>(g, st, st.u, nullptr, X)) || (rc = sg_real_of<Rl>(g, st, st.d, nullptr, Y))) return rc;
    if ((rc = g->cuda(sg_sums<Rl>(X, Y, st.u, st.d, g->nx, g->ny, st.w, g->half, g->batch, g->kx2d, g->ky2d,
                                  g->p.dt, g->partials, g->sums, g->stream), "sg sums")) ||
        (rc = finish_sums(g)))
        return rc;
    const double dA = g->dA(), inv_n = 1.0 / (double(g->nx) * double(g->ny));
    bool finite = true;
    for (int64_t f = 0; f < g->batch; ++f) {
        const double *s = g->host_sums + 3 * f;
        out[f] = dA * (s[0] + s[1]) + 0.5 * dA * s[2] * inv_n;
        finite = finite && std::isfinite(out[f]);
    }
    return finite ? PSS_OK : g->fail(PSS_E_NONFINITE, "non-finite SG Hamiltonian");
}

}  // namespace

// ----------------------------------------------------------------------------
// Navier-Stokes: buf[0..2] vorticity iterates (per-field index in ns_field),
// buf[3] = J_hat^n, buf[4] = C1, buf[5] = C2, buf[6] scratch.

namespace {

// buffer i of field f
template <class Rl> V2<Rl> *Bf(pss_grid *g, int i, int64_t f) { return B<Rl>(g, i) + f * g->npts; }

template <class Rl> void ns_w(pss_grid *g, V2<Rl> *w[3])
{
    for (int i = 0; i < 3; ++i) w[i] = B<Rl>(g, i);
}

// derivatives of w^n into C1, C2 (per_step: w^n of each field in its own
// buffer idx; otherwise in buffer 0, as after set_state)
template <class Rl> int ns_prep(pss_grid *g, bool per_step = false)
{
    V2<Rl> *w[3];
    ns_w<Rl>(g, w);
    return g->cuda(ns_prep_pass<Rl>(w, per_step ? g->ns_field : nullptr, B<Rl>(g, 4), B<Rl>(g, 5), Rt<Rl>(g->kxo),
                                    Rt<Rl>(g->kyo), Rt<Rl>(g->kx2), Rt<Rl>(g->ky2), g->nx, g->ny, g->batch,
                                    reinterpret_cast<int *>(g->flags), Tw<Rl>(g->twy), g->stream,
                                    g->ns_half ? g->nsx : 0), "ns derivatives");
}

// offset of field f in a vorticity buffer (half spectra: rows of nsx)
inline int64_t ns_off(const pss_grid *g, int64_t f) { return f * g->ny * (g->ns_half ? g->nsx : g->nx); }

// derivatives of field f alone (its w^n in buffer 0)
template <class Rl> int ns_prep_one(pss_grid *g, int64_t f)
{
    V2<Rl> *w[3] = {B<Rl>(g, 0) + ns_off(g, f), B<Rl>(g, 1) + ns_off(g, f), B<Rl>(g, 2) + ns_off(g, f)};
    return g->cuda(ns_prep_pass<Rl>(w, nullptr, Bf<Rl>(g, 4, f), Bf<Rl>(g, 5, f), Rt<Rl>(g->kxo), Rt<Rl>(g->kyo),
                                    Rt<Rl>(g->kx2), Rt<Rl>(g->ky2), g->nx, g->ny, 1,
                                    reinterpret_cast<int *>(g->flags), Tw<Rl>(g->twy), g->stream,
                                    g->ns_half ? g->nsx : 0),
                   "ns derivatives");
}

// half spectra: the full spectra of `batch` fields at src into the vorticity
// layout at dst (through buf[6] when src is buf[0] itself)
template <class Rl> int ns_to_half(pss_grid *g, V2<Rl> *src, V2<Rl> *dst, int64_t batch)
{
    if (src == dst) {
        const size_t hb = size_t(g->nsx) * size_t(g->ny) * size_t(batch) * g->esz;
        int rc = g->cuda(pack_half<Rl>(src, B<Rl>(g, 6), g->nx, g->ny, g->nsx, batch, g->stream), "pack");
        if (rc) return rc;
        return g->cuda(cudaMemcpyAsync(dst, B<Rl>(g, 6), hb, cudaMemcpyDeviceToDevice, g->stream), "copy");
    }
    return g->cuda(pack_half<Rl>(src, dst, g->nx, g->ny, g->nsx, batch, g->stream), "pack");
}

// vorticity of fields f .. f + nb - 1: masked spectra into buffer 0, their
// records cleared, derivatives formed
template <class Rl> int ns_set(pss_grid *g, int64_t f, int64_t nb, const void *w0, int where)
{
    const int64_t width = g->ns_half ? g->nsx : g->nx;
    V2<Rl> *w = B<Rl>(g, 0) + ns_off(g, f);
    const Rl *src = nullptr;
    int rc;
    if ((rc = real_in<Rl>(g, w0, where, reinterpret_cast<Rl *>(Bf<Rl>(g, 6, f)), nb * g->npts, &src)) ||
        (rc = g->cuda(rows_from_real<Rl>(src, w, g->nx, g->ns_half ? g->nsx : 0, g->ny, nb, Tw<Rl>(g->twx), g->stream),
                      "forward rows")) ||
        (rc = g->cuda(fft_cols<Rl>(w, w, width, g->ny, nb, -1, Rl(1), Tw<Rl>(g->twy), g->stream), "forward columns")) ||
        (rc = g->cuda(apply_mask<Rl>(w, Rt<Rl>(g->keepx), Rt<Rl>(g->keepy), width, g->ny, nb, g->stream), "mask")) ||
        (rc = g->cuda(cudaMemsetAsync(static_cast<char *>(g->ns_field) + f * ns_field_bytes(), 0,
                                      size_t(nb) * ns_field_bytes(), g->stream), "memset")))
        return rc;
    for (int64_t i = f; i < f + nb && nb < g->batch; ++i)
        if ((rc = ns_prep_one<Rl>(g, i))) return rc;
    if (nb == g->batch && (rc = ns_prep<Rl>(g))) return rc;
    return where == PSS_HOST ? g->cuda(cudaStreamSynchronize(g->stream), "sync") : PSS_OK;
}

// Updates in one body of the captured loop: an iteration of the WHILE node
// costs about 5 us beside its kernels, so a body holds the two updates most
// steps take (four gain another 1 % on long calls and leave up to three
// updates to run empty at the end of a call, 3 kernels of 2 us each).
constexpr int NS_BODY = 2;

// one loop body: (midpoint) the derivatives of w^n of the fields that start a
// step, then `updates` times row pass, column pass and decision
template <class Rl> int ns_body(pss_grid *g, int updates, bool in_graph)
{
    V2<Rl> *w[3];
    ns_w<Rl>(g, w);
    int *ctl = reinterpret_cast<int *>(g->flags);
    const bool mid = g->p.scheme == PSS_NS_MIDPOINT;
    const double parseval = g->p.lx * g->p.ly / (double(g->npts) * double(g->npts));
    int rc;
    if (mid && (rc = ns_prep<Rl>(g, true))) return rc;
    for (int u = 0; u < updates; ++u) {
        if (!in_graph && (rc = g->pass_begin(0))) return rc;
        cudaError_t e = ns_row_pass<Rl>(B<Rl>(g, 4), B<Rl>(g, 5), g->ns_field, g->nx, g->ny, g->batch, ctl,
                                        Tw<Rl>(g->twx), g->stream, g->p.dealias != 0,
                                        g->p.dealias != 0 && !g->ns_masked_modes, g->ns_half);
        if ((!in_graph && (rc = g->pass_end())) || (rc = g->cuda(e, "ns row pass"))) return rc;
        int groups = 0;
        if (!in_graph && (rc = g->pass_begin(1))) return rc;
        e = ns_col_pass<Rl>(B<Rl>(g, 4), B<Rl>(g, 5), w, B<Rl>(g, 3), g->ns_field, g->partials, Rt<Rl>(g->kxo),
                            Rt<Rl>(g->kyo), Rt<Rl>(g->kx2), Rt<Rl>(g->ky2), Rt<Rl>(g->keepx), Rt<Rl>(g->keepy),
                            g->p.dt, g->p.nu, g->nx, g->ny, g->batch, ctl, mid ? 1 : 0, Tw<Rl>(g->twy), &groups,
                            g->stream, g->p.dealias != 0, g->ns_half ? g->nsx : 0);
        if ((!in_graph && (rc = g->pass_end())) || (rc = g->cuda(e, "ns column pass"))) return rc;
        if (!in_graph && (rc = g->pass_begin(2))) return rc;
        e = ns_decide(g->ns_field, g->partials, groups, g->batch, ctl, parseval, g->p.tol, g->p.max_iter, mid,
                      u + 1 == updates, in_graph, g->ns_cond, g->stream);
        if ((!in_graph && (rc = g->pass_end())) || (rc = g->cuda(e, "ns decide"))) return rc;
    }
    return PSS_OK;
}

// the steps of a call as a graph: WHILE(some field has steps left) { body }
template <class Rl> int ns_build_graph(pss_grid *g)
{
    cudaGraph_t graph = nullptr;
    int rc;
    if ((rc = g->cuda(cudaGraphCreate(&graph, 0), "graph create"))) return rc;
    g->ns_graph = graph;
    if ((rc = g->cuda(cudaGraphConditionalHandleCreate(&g->ns_cond, graph, 1, cudaGraphCondAssignDefault),
                      "conditional handle")))
        return rc;
    // zero-initialised node parameters (the struct's union has no default constructor)
    alignas(cudaGraphNodeParams) unsigned char raw[sizeof(cudaGraphNodeParams)] = {};
    cudaGraphNodeParams &cp = *reinterpret_cast<cudaGraphNodeParams *>(raw);
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = g->ns_cond;
    cp.conditional.type = cudaGraphCondTypeWhile;
    cp.conditional.size = 1;
    cudaGraphNode_t cnode = nullptr;
    if ((rc = g->cuda(cudaGraphAddNode(&cnode, graph, nullptr, nullptr, 0, &cp), "conditional node"))) return rc;
    cudaGraph_t body = cp.conditional.phGraph_out[0];
    if ((rc = g->cuda(cudaStreamBeginCaptureToGraph(g->stream, body, nullptr, nullptr, 0,
                                                    cudaStreamCaptureModeRelaxed), "capture body")))
        return rc;
    rc = ns_body<Rl>(g, NS_BODY, true);
    cudaGraph_t out = nullptr;
    const cudaError_t e = cudaStreamEndCapture(g->stream, &out);
    if (rc) return rc;
    if ((rc = g->cuda(e, "capture body end"))) return rc;
    return g->cuda(cudaGraphInstantiate(&g->ns_exec, graph, 0), "graph instantiate");
}

template <class Rl> int ns_step(pss_grid *g, int64_t n)
{
    int *ctl = reinterpret_cast<int *>(g->flags);
    int *hctl = reinterpret_cast<int *>(g->host_flags);
    int rc;
    if (g->use_graphs && !g->profiling && !g->ns_exec && ns_build_graph<Rl>(g) != PSS_OK) {
        // capture is not available here: keep stepping with direct launches
        g->use_graphs = false;
        cudaGetLastError();
        g->err.clear();
    }
    const int64_t most = 1 << 30;  // steps per launch of the loop (the records count in 32 bits)
    for (int64_t done = 0; done < n; done += most) {
        const int part = int(std::min(most, n - done));
        if ((rc = g->cuda(ns_begin(g->ns_field, g->batch, ctl, part, g->stream), "ns begin"))) return rc;
        if (g->use_graphs && !g->profiling) {
            if ((rc = g->cuda(cudaGraphLaunch(g->ns_exec, g->stream), "graph launch"))) return rc;
            continue;
        }
        do {
            if ((rc = ns_body<Rl>(g, 1, false))) return rc;
            if ((rc = g->cuda(cudaMemcpyAsync(hctl, ctl, 4 * sizeof(int), cudaMemcpyDeviceToHost, g->stream),
                              "ctl copy")) ||
                (rc = g->cuda(cudaStreamSynchronize(g->stream), "ns sync")))
                return rc;
        } while (hctl[2] != 0);
    }
    if (g->use_graphs && !g->profiling) return PSS_OK;  // a field that reached max_iter: the next synchronising call
    rc = g->check_ns_nonconv();
    if (rc == PSS_E_NOT_CONVERGED) g->steps += n;  // the steps were taken; pss_grid::step_n adds n only on success
    return rc;
}

// current vorticity of every field into buf[6] (full spectra); half
// spectra gather into buf[3] (J_hat^n, rebuilt at the start of every step)
// and are extended to full width
template <class Rl> int ns_current(pss_grid *g)
{
    V2<Rl> *w[3];
    ns_w<Rl>(g, w);
    if (!g->ns_half)
        return g->cuda(ns_gather<Rl>(g->ns_field, w, B<Rl>(g, 6), g->npts, g->batch, g->stream), "gather");
    int rc = g->cuda(ns_gather<Rl>(g->ns_field, w, B<Rl>(g, 3), g->ny * g->nsx, g->batch, g->stream), "gather");
    if (rc) return rc;
    return g->cuda(unpack_half<Rl>(B<Rl>(g, 3), B<Rl>(g, 6), g->nx, g->ny, g->nsx, g->batch, g->stream), "unpack");
}

// vorticity of fields f .. f + nb - 1 into a: row pass into buf[6], column pass
// into the real array
template <class Rl> int ns_get(pss_grid *g, int64_t f, int64_t nb, void *a, int where)
{
    V2<Rl> *w[3];
    for (int i = 0; i < 3; ++i) w[i] = B<Rl>(g, i) + ns_off(g, f);
    const size_t bytes = size_t(nb * g->npts) * sizeof(Rl);
    const Access ac = where == PSS_DEVICE ? kernel_access(a, sizeof(Rl), bytes) : Access::COPY;
    if (ac == Access::SHORT) return short_array(g, "get_state", bytes);
    // (J_hat^n in buf[3] is rebuilt at the start of every step)
    Rl *dst = ac == Access::DIRECT ? static_cast<Rl *>(a) : reinterpret_cast<Rl *>(g->buf[3]) + f * g->npts;
    V2<Rl> *t = Bf<Rl>(g, 6, f);
    const Rl s = Rl(1.0 / (double(g->nx) * double(g->ny)));
    int rc;
    const int *rec = reinterpret_cast<const int *>(static_cast<char *>(g->ns_field) + f * ns_field_bytes());
    if ((rc = g->cuda(rows_inverse<Rl>(w, rec, int64_t(ns_field_bytes() / sizeof(int)), nullptr, t, g->nx,
                                       g->ns_half ? g->nsx : 0, g->ny, nb, Tw<Rl>(g->twx), g->stream),
                      "inverse rows")) ||
        (rc = g->cuda(cols_to_real<Rl>(t, dst, s, g->nx, g->ny, nb, Tw<Rl>(g->twy), g->stream), "inverse columns")) ||
        (ac == Access::COPY &&
         (rc = g->cuda(cudaMemcpyAsync(a, dst, bytes, kind_out(where), g->stream), "state copy"))))
        return rc;
    return g->sync();
}

template <class Rl> int ns_conserved(pss_grid *g, double *out)
{
    V2<Rl> *w[3];
    ns_w<Rl>(g, w);
    int rc;
    if (g->ns_half) {  // sums over the full spectra of buf[6]
        if ((rc = ns_current<Rl>(g))) return rc;
        w[0] = w[1] = w[2] = B<Rl>(g, 6);
    }
    if ((rc = g->cuda(ns_sums<Rl>(g->ns_field, w, g->nx, g->ny, g->batch, g->kx2d, g->ky2d, g->partials, g->sums,
                                  g->stream), "ns sums")) ||
        (rc = finish_sums(g)))
        return rc;
    const double dA = g->dA(), inv_n = 1.0 / (double(g->nx) * double(g->ny));
    bool finite = true;
    for (int64_t f = 0; f < g->batch; ++f) {
        const double *s = g->host_sums + 3 * f;
        out[3 * f] = dA * s[0];
        out[3 * f + 1] = 0.5 * dA * s[1] * inv_n;
        out[3 * f + 2] = 0.5 * dA * s[2] * inv_n;
        for (int k = 0; k < 3; ++k) finite = finite && std::isfinite(out[3 * f + k]);
    }
    return finite ? PSS_OK : g->fail(PSS_E_NONFINITE, "non-finite NS invariant");
}

}  // namespace

// ----------------------------------------------------------------------------
// One field of the batch (slot f): the set-up and read-back of the equation on
// the sub-arrays of field f, with batch 1.

namespace {

template <class Rl> int field_set(pss_grid *g, int64_t f, const void *a, const void *b, int where)
{
    if (g->p.eq == PSS_EQ_NLS) return nls_set<Rl>(g, f, 1, a, where);
    if (g->p.eq == PSS_EQ_SG) return sg_set_fields<Rl>(g, f, 1, a, b, where);
    return ns_set<Rl>(g, f, 1, a, where);
}

template <class Rl> int field_get(pss_grid *g, int64_t f, void *a, void *b, int where)
{
    if (g->p.eq == PSS_EQ_NLS) return nls_get<Rl>(g, f, 1, a, where);
    if (g->p.eq == PSS_EQ_SG) return sg_get_fields<Rl>(g, f, 1, a, b, where);
    return ns_get<Rl>(g, f, 1, a, where);
}

}  // namespace

// ----------------------------------------------------------------------------
// dispatch by equation and precision

#define PSS_BY_PRECISION(CALL) (p.precision == PSS_FP32 ? CALL(float) : CALL(double))

// Whether a masked mode of the state may be non-zero (a dealiased grid that
// restored another grid's checkpoint); the captured loop is rebuilt when that changes.
void pss_grid::set_masked_modes(bool any)
{
    if (any == ns_masked_modes) return;
    ns_masked_modes = any;
    drop_graphs();
}

int pss_grid::find_masked_modes(bool *any)
{
    int *dev = reinterpret_cast<int *>(flags) + FLAG_SLOT_MASKED;
    int *host = reinterpret_cast<int *>(host_flags) + FLAG_SLOT_MASKED;
    int rc = cuda(cudaMemsetAsync(dev, 0, sizeof(int), stream), "masked modes");
    if (rc) return rc;
    const cudaError_t e = p.precision == PSS_FP32
                              ? masked_columns<float>(B<float>(this, 0), Rt<float>(keepx), nx, ntot, dev, stream)
                              : masked_columns<double>(B<double>(this, 0), Rt<double>(keepx), nx, ntot, dev, stream);
    if ((rc = cuda(e, "masked modes")) ||
        (rc = cuda(cudaMemcpyAsync(host, dev, sizeof(int), cudaMemcpyDeviceToHost, stream), "masked modes")) ||
        (rc = cuda(cudaStreamSynchronize(stream), "masked modes")))
        return rc;
    *any = *host != 0;
    return PSS_OK;
}

int pss_grid::set_state(const void *a, const void *b, int where)
{
    steps = 0;
    nonconv_pending = false;
    int rc;
#define NLS(R) nls_set<R>(this, 0, batch, a, where)
#define SG(R) sg_set_fields<R>(this, 0, batch, a, b, where)
#define NS(R) ns_set<R>(this, 0, batch, a, where)
    rc = p.eq == PSS_EQ_NLS ? PSS_BY_PRECISION(NLS) : p.eq == PSS_EQ_SG ? PSS_BY_PRECISION(SG) : PSS_BY_PRECISION(NS);
#undef NLS
#undef SG
#undef NS
    if (!rc) {
        has_state = true;
        full_valid = !half;
        half_valid = half;
        set_masked_modes(false);
    }
    return rc;
}

int pss_grid::set_sg_levels(const void *u_n, const void *u_nm1, int where)
{
    int rc = p.precision == PSS_FP32 ? sg_set_levels<float>(this, u_n, u_nm1, where)
                                     : sg_set_levels<double>(this, u_n, u_nm1, where);
    if (rc) return rc;
    steps = 0;
    has_state = true;
    full_valid = !half;
    half_valid = half;
    return PSS_OK;
}

int pss_grid::half_sync(bool to_half)
{
    if (!half || (to_half ? half_valid : full_valid)) return PSS_OK;
    int rc = p.precision == PSS_FP32 ? sg_half_sync<float>(this, to_half) : sg_half_sync<double>(this, to_half);
    if (rc) return rc;
    (to_half ? half_valid : full_valid) = true;
    return PSS_OK;
}

int pss_grid::step_n(int64_t n)
{
    if (n == 0) return PSS_OK;
    int rc;
    prof_pass = 0;
    if (graph_epoch != plan_epoch().load()) {  // a plan changed: recapture
        drop_graphs();
        graph_epoch = plan_epoch().load();
    }
    if ((rc = half_sync(true))) return rc;
    if (half) full_valid = false;
#define NLS(R) nls_step<R>(this, n)
#define SG(R) sg_step<R>(this, n)
#define NS(R) ns_step<R>(this, n)
    if (p.eq != PSS_EQ_NS && use_graphs) {
        // the whole launch sequence of step_n(n) as one graph, cached by
        // (n, profiling); a profiling graph's own events time its passes
        const int prof_key = profiling ? prof_stride : 0;
        StepGraph *sg = nullptr;
        for (auto &e : step_graphs)
            if (e.n == n && e.prof == prof_key) sg = &e;
        if (sg && sg == prof_pending && (rc = profile_resolve())) return rc;  // its events are reused
        if (!sg) {
            StepGraph fresh;
            fresh.n = n;
            fresh.prof = prof_key;
            rc = cuda(cudaStreamBeginCapture(stream, cudaStreamCaptureModeRelaxed), "capture");
            if (!rc) {
                const int64_t saved = launches;
                if (profiling) capturing = &fresh;
                prof_pass = 0;
                int inner = p.eq == PSS_EQ_NLS ? PSS_BY_PRECISION(NLS) : PSS_BY_PRECISION(SG);
                capturing = nullptr;
                fresh.passes = launches - saved;
                launches = saved;
                cudaGraph_t graph = nullptr;
                cudaError_t e = cudaStreamEndCapture(stream, &graph);
                if (inner) rc = inner;
                else if ((rc = cuda(e, "capture end")) == PSS_OK)
                    rc = cuda(cudaGraphInstantiate(&fresh.exec, graph, 0), "graph instantiate");
                if (graph) cudaGraphDestroy(graph);
            }
            if (rc) {
                // capture is not available here: direct launches from now on
                free_step_graph(fresh);
                use_graphs = false;
                cudaGetLastError();
                err.clear();
                rc = p.eq == PSS_EQ_NLS ? PSS_BY_PRECISION(NLS) : PSS_BY_PRECISION(SG);
                if (!rc) steps += n;
                return rc;
            }
            if (step_graphs.size() >= 4) {
                if (prof_pending) {  // resolve before the list (and the pending entry) moves
                    if ((rc = profile_resolve())) {
                        free_step_graph(fresh);
                        return rc;
                    }
                }
                free_step_graph(step_graphs.front());
                step_graphs.erase(step_graphs.begin());
            }
            if (prof_pending) {  // the vector may reallocate below
                if ((rc = profile_resolve())) {
                    free_step_graph(fresh);
                    return rc;
                }
            }
            step_graphs.push_back(std::move(fresh));
            sg = &step_graphs.back();
        }
        rc = cuda(cudaGraphLaunch(sg->exec, stream), "graph launch");
        if (!rc) {
            launches += sg->passes;
            if (sg->prof) prof_pending = sg;
        }
    } else {
        rc = p.eq == PSS_EQ_NLS ? PSS_BY_PRECISION(NLS) : p.eq == PSS_EQ_SG ? PSS_BY_PRECISION(SG) : PSS_BY_PRECISION(NS);
    }
#undef NLS
#undef SG
#undef NS
    if (!rc) steps += n;
    return rc;
}

int pss_grid::get_state(void *a, void *b, int where)
{
    int rc = half_sync(true);
    if (rc) return rc;
#define NLS(R) nls_get<R>(this, 0, batch, a, where)
#define SG(R) sg_get_fields<R>(this, 0, batch, a, b, where)
#define NS(R) ns_get<R>(this, 0, batch, a, where)
    return p.eq == PSS_EQ_NLS ? PSS_BY_PRECISION(NLS) : p.eq == PSS_EQ_SG ? PSS_BY_PRECISION(SG) : PSS_BY_PRECISION(NS);
#undef NLS
#undef SG
#undef NS
}

int pss_grid::set_field(int64_t f, const void *a, const void *b, int where)
{
    int rc = half_sync(true);  // the other fields' state must be current
    if (rc) return rc;
    if (half) full_valid = false;
    rc = p.precision == PSS_FP32 ? field_set<float>(this, f, a, b, where) : field_set<double>(this, f, a, b, where);
    if (!rc) has_state = true;
    return rc;
}

int pss_grid::get_field(int64_t f, void *a, void *b, int where)
{
    int rc = half_sync(true);
    if (rc) return rc;
    return p.precision == PSS_FP32 ? field_get<float>(this, f, a, b, where) : field_get<double>(this, f, a, b, where);
}

int pss_grid::conserved(double *out)
{
    int rc = half_sync(true);
    if (rc) return rc;
#define NLS(R) nls_conserved<R>(this, out)
#define SG(R) sg_conserved<R>(this, out)
#define NS(R) ns_conserved<R>(this, out)
    return p.eq == PSS_EQ_NLS ? PSS_BY_PRECISION(NLS) : p.eq == PSS_EQ_SG ? PSS_BY_PRECISION(SG) : PSS_BY_PRECISION(NS);
#undef NLS
#undef SG
#undef NS
}

// Checkpoint layout: the exact state buffers (NLS: row transform of psi;
// SG: uhat^n, d^n; NS: w_hat^n of every field), then {steps, NS updates}.
size_t pss_grid::checkpoint_bytes() const
{
    const int nstate = p.eq == PSS_EQ_SG ? 2 : 1;
    return size_t(nstate) * size_t(ntot) * esz + 16;
}

int pss_grid::checkpoint(void *buf_, int where, bool save)
{
    const int nstate = p.eq == PSS_EQ_SG ? 2 : 1;
    char *b = static_cast<char *>(buf_);
    int rc;
    if (save && (rc = half_sync(false))) return rc;
    int src_of[2] = {0, 1};
    if (save && p.eq == PSS_EQ_NS) {
        rc = p.precision == PSS_FP32 ? ns_current<float>(this) : ns_current<double>(this);
        if (rc) return rc;
        src_of[0] = 6;
    }
    for (int i = 0; i < nstate; ++i) {
        if (save)
            rc = cuda(cudaMemcpyAsync(b + i * field_bytes(), this->buf[src_of[i]], field_bytes(), kind_out(where), stream),
                      "checkpoint");
        else
            rc = cuda(cudaMemcpyAsync(this->buf[i], b + i * field_bytes(), field_bytes(), kind_in(where), stream),
                      "checkpoint");
        if (rc) return rc;
    }
    int64_t meta[2] = {steps, 0};
    if (save && (rc = ns_update_count(&meta[1]))) return rc;
    char *mb = b + nstate * field_bytes();
    if (save)
        rc = cuda(cudaMemcpyAsync(mb, meta, 16, where == PSS_HOST ? cudaMemcpyHostToHost : cudaMemcpyHostToDevice, stream),
                  "checkpoint meta");
    else
        rc = cuda(cudaMemcpyAsync(meta, mb, 16, where == PSS_HOST ? cudaMemcpyHostToHost : cudaMemcpyDeviceToHost, stream),
                  "checkpoint meta");
    if (rc || (rc = cuda(cudaStreamSynchronize(stream), "checkpoint sync"))) return rc;
    if (!save) {
        steps = meta[0];
        if (p.eq == PSS_EQ_SG) {
            if (!half)  // half spectra: the next use packs them and makes H
                rc = p.precision == PSS_FP32 ? sg_make_h<float>(this, sg_state<float>(this, 0, batch))
                                             : sg_make_h<double>(this, sg_state<double>(this, 0, batch));
        } else if (p.eq == PSS_EQ_NS) {
            // all fields restart from buffer 0 with their update count
            NsFieldHost *h = static_cast<NsFieldHost *>(host_fields);
            for (int64_t i = 0; i < batch; ++i) h[i] = NsFieldHost{0, 0, 0, 0, i == 0 ? meta[1] : 0, 0, 0};
            rc = cuda(cudaMemcpyAsync(ns_field, h, size_t(batch) * ns_field_bytes(), cudaMemcpyHostToDevice, stream),
                      "fields");
            bool masked = false;
            if (!rc && p.dealias) rc = find_masked_modes(&masked);
            if (!rc) set_masked_modes(masked);
            if (!rc && ns_half)
                rc = p.precision == PSS_FP32 ? ns_to_half<float>(this, B<float>(this, 0), B<float>(this, 0), batch)
                                             : ns_to_half<double>(this, B<double>(this, 0), B<double>(this, 0), batch);
            if (!rc) rc = p.precision == PSS_FP32 ? ns_prep<float>(this) : ns_prep<double>(this);
        }
        if (rc || (rc = cuda(cudaStreamSynchronize(stream), "restore sync"))) return rc;
        has_state = true;
        full_valid = true;
        half_valid = false;
    }
    return PSS_OK;
}

// ----------------------------------------------------------------------------
// Autotuner: time `steps` steps of this grid in each launch-shape variant
// (on its own state, restored afterwards; a one-step round of each first, then
// two alternating timed rounds, best of the two) and keep, per row and per
// column pass kernel, the faster variant (variant 1 must win by more than 2 %).

int pss_grid::autotune(int k, int *changed)
{
    *changed = 0;
    if (p.precision != PSS_FP32 || p.eq == PSS_EQ_NS) return PSS_OK;  // nothing tunable
    if (!has_state) return fail(PSS_E_STATE, "autotune before set_state");
    void *save = nullptr;
    const size_t bytes = checkpoint_bytes();
    if (cudaMalloc(&save, bytes) != cudaSuccess) {
        cudaGetLastError();
        return fail(PSS_E_OOM, "autotune: no room for a copy of the state");
    }
    int rc = checkpoint(save, PSS_DEVICE, true);
    const bool prof = profiling;
    const int stride = prof_stride;
    prof_stride = 1;  // every pass of the tuning steps is timed
    // per variant and pass kind, the best mean pass time over the rounds; round
    // 0 (one step of each variant) only loads the kernels and warms the clocks
    double t[2][2] = {{1e30, 1e30}, {1e30, 1e30}};
    PlanTuning *pt = plan_tuning();
    PlanSlot *used[2][8] = {};
    int nused[2] = {0, 0};
    for (int round = 0; round < 3 && rc == PSS_OK; ++round)
        for (int v = 0; v < 2 && rc == PSS_OK; ++v) {
            *pt = PlanTuning{};
            pt->force = v;
            drop_graphs();
            if ((rc = profile_resolve())) break;
            profiling = true;
            for (int i = 0; i < 3; ++i) prof_ms[i] = 0, prof_n[i] = 0;
            rc = step_n(round == 0 ? 1 : k);
            if (!rc) rc = profile_resolve();
            for (int kind = 0; kind < 2 && !rc && round > 0; ++kind)
                if (prof_n[kind]) t[v][kind] = std::min(t[v][kind], prof_ms[kind] / prof_n[kind]);
            if (v == 0 && round == 0)
                for (int kind = 0; kind < 2; ++kind) {
                    nused[kind] = pt->nused[kind];
                    for (int i = 0; i < nused[kind]; ++i) used[kind][i] = pt->used[kind][i];
                }
            const int rrc = checkpoint(save, PSS_DEVICE, false);
            if (!rc) rc = rrc;
        }
    *pt = PlanTuning{};
    profiling = prof;
    prof_stride = stride;
    for (int i = 0; i < 3; ++i) prof_ms[i] = 0, prof_n[i] = 0;
    cudaFree(save);
    if (rc) return rc;
    for (int kind = 0; kind < 2; ++kind)
        for (int i = 0; i < nused[kind]; ++i) {
            const int pick = t[1][kind] < 0.98 * t[0][kind] ? 1 : 0;
            const int old = used[kind][i]->var.exchange(pick);
            if ((old < 0 ? 0 : old) != pick) ++*changed;  // an unset slot ran variant 0
        }
    if (*changed) plan_epoch().fetch_add(1);
    drop_graphs();
    graph_epoch = plan_epoch().load();
    return PSS_OK;
}

// ----------------------------------------------------------------------------
// standalone 2D transform

namespace {
std::mutex g_tw_mutex;
std::map<std::tuple<int, int, int64_t>, void *> g_tw_cache;  // (device, precision, n)

void *cached_twiddles(int dev, int precision, int64_t n, int *rc)
{
    std::lock_guard<std::mutex> lk(g_tw_mutex);
    auto key = std::make_tuple(dev, precision, n);
    auto it = g_tw_cache.find(key);
    if (it != g_tw_cache.end()) return it->second;
    void *d = nullptr;
    size_t bytes;
    std::vector<float> tf;
    std::vector<double> td;
    const void *src;
    if (precision == PSS_FP32) {
        tf = twiddles_f32(n);
        src = tf.data();
        bytes = tf.size() * 4;
    } else {
        td = twiddles_f64(n);
        src = td.data();
        bytes = td.size() * 8;
    }
    if (cudaMalloc(&d, bytes) != cudaSuccess) {
        cudaGetLastError();
        *rc = PSS_E_OOM;
        return nullptr;
    }
    if (cudaMemcpy(d, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaFree(d);
        *rc = PSS_E_CUDA;
        return nullptr;
    }
    g_tw_cache[key] = d;
    return d;
}
}  // namespace

extern "C" int pss_fft2d(void *data, int64_t nx, int64_t ny, int64_t batch, int precision, int direction,
                         void *stream)
{
    if (!data || batch < 1 || batch > 65535 || (direction != 1 && direction != -1) ||
        (precision != PSS_FP32 && precision != PSS_FP64))
        return PSS_E_ARG;
    auto ok = [](int64_t n) { return n >= 16 && n <= 8192 && (n & (n - 1)) == 0; };
    if (!ok(nx) || !ok(ny)) return PSS_E_ARG;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return PSS_E_CUDA;
    int rc = PSS_OK;
    void *twx = cached_twiddles(dev, precision, nx, &rc);
    if (!twx) return rc;
    void *twy = cached_twiddles(dev, precision, ny, &rc);
    if (!twy) return rc;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    cudaError_t e;
    const double inv = direction > 0 ? 1.0 / (double(nx) * double(ny)) : 1.0;
    if (precision == PSS_FP32) {
        e = fft_rows<float>(static_cast<float2 *>(data), static_cast<float2 *>(data), nx, ny, batch, direction, 1.0f, static_cast<float4 *>(twx), s);
        if (e == cudaSuccess)
            e = fft_cols<float>(static_cast<float2 *>(data), static_cast<float2 *>(data), nx, ny, batch, direction, float(inv), static_cast<float4 *>(twy), s);
    } else {
        e = fft_rows<double>(static_cast<double2 *>(data), static_cast<double2 *>(data), nx, ny, batch, direction, 1.0, static_cast<double2 *>(twx), s);
        if (e == cudaSuccess)
            e = fft_cols<double>(static_cast<double2 *>(data), static_cast<double2 *>(data), nx, ny, batch, direction, inv, static_cast<double2 *>(twy), s);
    }
    return e == cudaSuccess ? PSS_OK : PSS_E_CUDA;
}
