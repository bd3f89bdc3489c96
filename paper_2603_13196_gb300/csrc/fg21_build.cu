// Region building on the GPU: the per-pixel importance weights (Sec. 4.2,
// eq. w_beam_dynamic and its sky / horizon / uniform variants) and the
// chromatic response functions of the partition (Sec. 2.2, eq.
// chromatic_function), the O(Npix F T) parts of fg21_build_regions.  The
// partition itself (sorting by the field and Algorithms 1 / 2) stays on the
// host: it is O(Npix log Npix).
//
// The arithmetic is the host's, in FP64: ln c = ln(z_t . v) per (pixel, LST),
// the beam D = 2(p+1) exp(p ln c) above the horizon, T_sky of eq.
// skyapproximation.  Only the summation order differs (fixed-order block
// trees over pixels, then over channels), so the results agree with the host
// to FP64 rounding; every sum is deterministic.
//
//   pass 1, one block per (f, t):   den[f,t] = sum_q num(q,f,t),  Bsum[f,t] = sum_q D(q,f,t)
//           (B comes of it whatever the weighting)
//   pass 2, one thread per (q, f):  pw[f,q]  = sum_t num(q,f,t) / den[f,t];
//           one thread per q:       w[q]     = (1/(F T)) sum_f pw[f,q]
//   pass 3, one block per (f, t):   A[c,f,t] = (1/Npix) sum_{q in component c} (T230_q - T_CMB) D(q,f,t)
//           over the pixels sorted by component (contiguous segments).
//
// What bounds it is the FP64 exponential of D (this part's FP64 rate is 1/64 of
// FP32's), needed by every pass: pass 1 keeps D [F][T][Npix] in device memory
// where a quarter of what is free holds it (0.3 GB at 12288 pixels, 151 channels, 20
// bins; 11.8 GB at 49152, 301, 100) and the others read it; without the room, or
// when another allocation of the build needs it, they evaluate it again.  The tables of one build serve both its halves.
// 12288 pixels, 9 regions, 151 channels, 20 bins: 4.06 ms a build from 8.00 (four
// evaluations of D, and the tables made twice).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <vector>

#include "fg21_internal.h"

namespace fg21 {
namespace {

constexpr int BUILD_THREADS = 256;

struct DevObs {
    const double *lognu;   // [F] ln(nu_f / nu0)
    const double *beam_p;  // [F]
    const double *logcT;   // [T][npix] ln(z_t . v_q), -inf below the horizon
    const double *tskyT;   // [F][npix] T_sky(q, f) (sky and beam weightings)
    const double *D;       // [F][T][npix] the beam where pass 1 kept it, else null
    int64_t npix;
    int F, T;
    double t_cmb;
};

__device__ __forceinline__ double beam_d(double lc, double p) {
    if (lc == -INFINITY) return 0.0;
    return 2.0 * (p + 1.0) * (p == 0.0 ? 1.0 : exp(p * lc));
}

// D of pixel q at (f, t) = row ft
__device__ __forceinline__ double beam_at(const DevObs &o, int ft, int64_t q, double lc, double p) {
    return o.D ? o.D[(size_t)ft * o.npix + q] : beam_d(lc, p);
}

__device__ __forceinline__ double importance_num(const DevObs &o, int weighting, int64_t q, int f, double lc,
                                                 double d) {
    switch (weighting) {
        case FG21_WEIGHT_BEAM: return o.tskyT[(size_t)f * o.npix + q] * d;
        case FG21_WEIGHT_SKY: return lc == -INFINITY ? 0.0 : o.tskyT[(size_t)f * o.npix + q];
        case FG21_WEIGHT_HORIZON: return lc == -INFINITY ? 0.0 : 1.0;
        default: return 1.0;
    }
}

// fixed-order tree over the block (BUILD_THREADS doubles in shared memory)
__device__ __forceinline__ double block_sum(double v, double *sh) {
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int w = BUILD_THREADS / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    const double r = sh[0];
    __syncthreads();
    return r;
}

__global__ void logc_kernel(const double *__restrict__ dirs, const double *__restrict__ zen, int64_t npix, int T,
                            double *__restrict__ logcT) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npix * T) return;
    const int t = (int)(i / npix);
    const int64_t q = i - (int64_t)t * npix;
    const double *v = dirs + 3 * q, *z = zen + 3 * t;
    const double c = v[0] * z[0] + v[1] * z[1] + v[2] * z[2];
    logcT[i] = c > 0.0 ? log(c) : -INFINITY;
}

__global__ void tsky_kernel(const double *__restrict__ t230, const double *__restrict__ beta,
                            const double *__restrict__ lognu, double t_cmb, int64_t npix, int F,
                            double *__restrict__ tskyT) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= npix * F) return;
    const int f = (int)(i / npix);
    const int64_t q = i - (int64_t)f * npix;
    tskyT[i] = (t230[q] - t_cmb) * exp(-beta[q] * lognu[f]) + t_cmb;
}

// inv_den = 1 / den (0 for an empty sum); keep (optional): where to put D.
__global__ void __launch_bounds__(BUILD_THREADS) den_kernel(DevObs o, int weighting, double *__restrict__ inv_den,
                                                            double *__restrict__ bsum, double *__restrict__ keep) {
    __shared__ double sh[BUILD_THREADS];
    const int ft = blockIdx.x, f = ft / o.T, t = ft % o.T;
    const double p = o.beam_p[f];
    const double *lc_row = o.logcT + (size_t)t * o.npix;
    double a = 0.0, b = 0.0;
    for (int64_t q = threadIdx.x; q < o.npix; q += BUILD_THREADS) {
        const double lc = lc_row[q];
        const double d = beam_at(o, ft, q, lc, p);
        if (keep) keep[(size_t)ft * o.npix + q] = d;
        a += importance_num(o, weighting, q, f, lc, d);
        b += d;
    }
    a = block_sum(a, sh);
    b = block_sum(b, sh);
    if (threadIdx.x == 0) {
        inv_den[ft] = a > 0.0 ? 1.0 / a : 0.0;
        bsum[ft] = b;
    }
}

__global__ void __launch_bounds__(BUILD_THREADS) pw_kernel(DevObs o, int weighting,
                                                           const double *__restrict__ inv_den,
                                                           double *__restrict__ pw) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int f = blockIdx.y;
    if (q >= o.npix) return;
    const double p = o.beam_p[f];
    double acc = 0.0;
    for (int t = 0; t < o.T; ++t) {
        const double lc = o.logcT[(size_t)t * o.npix + q];
        acc += importance_num(o, weighting, q, f, lc, beam_at(o, f * o.T + t, q, lc, p)) * inv_den[(size_t)f * o.T + t];
    }
    pw[(size_t)f * o.npix + q] = acc;
}

__global__ void w_kernel(const double *__restrict__ pw, int64_t npix, int F, double inv_ft, double *__restrict__ w) {
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= npix) return;
    double acc = 0.0;
    for (int f = 0; f < F; ++f) acc += pw[(size_t)f * npix + q];
    w[q] = acc * inv_ft;
}

__global__ void __launch_bounds__(BUILD_THREADS) resp_kernel(DevObs o, const double *__restrict__ t230,
                                                             const int64_t *__restrict__ perm,
                                                             const int64_t *__restrict__ seg, int N,
                                                             double *__restrict__ A) {
    __shared__ double sh[BUILD_THREADS];
    const int ft = blockIdx.x, f = ft / o.T, t = ft % o.T;
    const double p = o.beam_p[f];
    const double *lc_row = o.logcT + (size_t)t * o.npix;
    const double inv = 1.0 / (double)o.npix;
    for (int c = 0; c < N; ++c) {
        double a = 0.0;
        for (int64_t k = seg[c] + threadIdx.x; k < seg[c + 1]; k += BUILD_THREADS) {
            const int64_t q = perm[k];
            a += (t230[q] - o.t_cmb) * beam_at(o, ft, q, lc_row[q], p);
        }
        a = block_sum(a, sh);
        if (threadIdx.x == 0) A[((size_t)c * o.F + f) * o.T + t] = a * inv;
    }
}

int fail(cudaError_t e, const char *what) {
    cudaGetLastError();
    if (e == cudaErrorMemoryAllocation) return set_error(FG21_E_NOMEM, "%s: device allocation failed", what);
    return cuda_error(e, what);
}

}  // namespace

// Device copies of the inputs, the geometry tables and the beam of one build,
// freed on destruction.  What the build can do without, the beam, and, for its
// second half, the tables of the importance weights, is given back when another
// allocation fails for lack of memory.
struct DeviceBuild {
    const fg21_sky *s;
    const fg21_obs *o;
    size_t limit;            // most device bytes the build may hold (0: as many as there are)
    size_t held = 0;
    DevObs g{};
    double *t230 = nullptr, *beta = nullptr, *lognu = nullptr, *tsky = nullptr, *beam = nullptr;
    double *inv_den = nullptr, *bsum = nullptr, *pw = nullptr, *w = nullptr;
    bool ready = false, summed = false;      // tables made; bsum (and beam) written
    bool weighted = false;                   // no importance weights are needed any more
    int beam_use = 0;                        // 0: the beam had no room, 1: kept, 2: given back
    std::vector<std::pair<void *, size_t>> own;
    ~DeviceBuild() {
        for (auto &p : own) cudaFree(p.first);
    }
    template <typename T>
    cudaError_t try_alloc(T **p, size_t n) {
        *p = nullptr;
        const size_t bytes = sizeof(T) * n;
        if (limit && held + bytes > limit) return cudaErrorMemoryAllocation;
        cudaError_t e = cudaMalloc((void **)p, bytes);
        if (e == cudaErrorMemoryAllocation) cudaGetLastError();
        if (e != cudaSuccess) return e;
        own.emplace_back(*p, bytes);
        held += bytes;
        return e;
    }
    // Frees what the rest of the build can do without (cudaFree waits for the
    // kernels that use it); true if there was any.
    bool shed() {
        const size_t before = own.size();
        if (beam) {
            drop(beam);
            beam_use = 2;
        }
        g.D = nullptr;
        if (weighted) {
            drop(pw);
            drop(w);
            drop(tsky);
            g.tskyT = nullptr;
        }
        return own.size() < before;
    }
    void drop(double *&p) {
        for (size_t k = 0; p && k < own.size(); ++k)
            if (own[k].first == p) {
                cudaFree(p);
                held -= own[k].second;
                own.erase(own.begin() + k);
                p = nullptr;
            }
    }
    template <typename T>
    cudaError_t alloc(T **p, size_t n) {
        cudaError_t e = try_alloc(p, n);
        if (e == cudaErrorMemoryAllocation && shed()) e = try_alloc(p, n);
        return e;
    }
    cudaError_t upload(double **dst, const double *src, size_t n) {
        const cudaError_t e = alloc(dst, n);
        return e != cudaSuccess ? e : cudaMemcpy(*dst, src, sizeof(double) * n, cudaMemcpyHostToDevice);
    }
    cudaError_t prepare(bool need_tsky);
    cudaError_t pass1(int weighting);
};

// inputs, ln c per (t, q) and (when needed) T_sky per (f, q)
cudaError_t DeviceBuild::prepare(bool need_tsky) {
    const int64_t npix = s->npix;
    const int F = o->F, T = o->T, th = BUILD_THREADS;
    cudaError_t e = cudaSuccess;
    if (!ready) {
        std::vector<double> ln(F);
        for (int f = 0; f < F; ++f) ln[f] = std::log(o->nu[f] / o->nu0);
        double *dirs = nullptr, *zen = nullptr, *beam_p = nullptr, *logcT = nullptr;
        e = upload(&dirs, s->dirs, 3 * (size_t)npix);
        if (e == cudaSuccess) e = upload(&t230, s->t230, npix);
        if (e == cudaSuccess) e = upload(&beta, s->beta, npix);
        if (e == cudaSuccess) e = upload(&lognu, ln.data(), F);
        if (e == cudaSuccess) e = upload(&beam_p, o->beam_p, F);
        if (e == cudaSuccess) e = upload(&zen, o->zenith, 3 * (size_t)T);
        if (e == cudaSuccess) e = alloc(&logcT, (size_t)npix * T);
        if (e == cudaSuccess) e = alloc(&inv_den, (size_t)F * T);
        if (e == cudaSuccess) e = alloc(&bsum, (size_t)F * T);
        if (e != cudaSuccess) return e;
        logc_kernel<<<(unsigned)((npix * T + th - 1) / th), th>>>(dirs, zen, npix, T, logcT);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        g.lognu = lognu;
        g.beam_p = beam_p;
        g.logcT = logcT;
        g.npix = npix;
        g.F = F;
        g.T = T;
        g.t_cmb = o->t_cmb;
        // room for the beam: at most a quarter of the free memory, and no error without it
        const size_t need = sizeof(double) * (size_t)npix * F * T;
        size_t room = 0, total = 0;
        if (cudaMemGetInfo(&room, &total) != cudaSuccess) {
            cudaGetLastError();
            room = 0;
        }
        if (limit) room = std::min(room, limit);
        if (need <= room / 4 && try_alloc(&beam, (size_t)npix * F * T) == cudaSuccess) beam_use = 1;
        ready = true;
    }
    if (need_tsky && !tsky) {
        e = alloc(&tsky, (size_t)npix * F);
        if (e != cudaSuccess) return e;
        tsky_kernel<<<(unsigned)((npix * F + th - 1) / th), th>>>(t230, beta, lognu, o->t_cmb, npix, F, tsky);
        e = cudaGetLastError();
        g.tskyT = tsky;
    }
    return e;
}

cudaError_t DeviceBuild::pass1(int weighting) {
    den_kernel<<<(unsigned)(g.F * g.T), BUILD_THREADS>>>(g, weighting, inv_den, bsum, summed ? nullptr : beam);
    const cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && !summed) {
        g.D = beam;
        summed = true;
    }
    return e;
}

DeviceBuild *device_build_begin(const fg21_sky *s, const fg21_obs *o, size_t limit) {
    DeviceBuild *b = new DeviceBuild;
    b->s = s;
    b->o = o;
    b->limit = limit;
    return b;
}
void device_build_end(DeviceBuild *b) { delete b; }
int device_build_beam(const DeviceBuild *b) { return b->beam_use; }

int device_importance(DeviceBuild *b, int weighting, std::vector<double> &w) {
    const bool need_tsky = weighting == FG21_WEIGHT_BEAM || weighting == FG21_WEIGHT_SKY;
    cudaError_t e = b->prepare(need_tsky);
    if (e != cudaSuccess) return fail(e, "region building (inputs)");
    const int64_t npix = b->g.npix;
    const int F = b->g.F, T = b->g.T, th = BUILD_THREADS;
    // (kept for the build's other weighting, if it has one)
    if (!b->pw) e = b->alloc(&b->pw, (size_t)F * npix);
    if (e == cudaSuccess && !b->w) e = b->alloc(&b->w, (size_t)npix);
    if (e != cudaSuccess) return fail(e, "region building (importance)");
    if ((e = b->pass1(weighting)) != cudaSuccess) return fail(e, "den_kernel");
    pw_kernel<<<dim3((unsigned)((npix + th - 1) / th), (unsigned)F), th>>>(b->g, weighting, b->inv_den, b->pw);
    w_kernel<<<(unsigned)((npix + th - 1) / th), th>>>(b->pw, npix, F, 1.0 / ((double)F * (double)T), b->w);
    if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "w_kernel");
    w.resize(npix);
    if ((e = cudaMemcpy(w.data(), b->w, sizeof(double) * npix, cudaMemcpyDeviceToHost)) != cudaSuccess)
        return fail(e, "region building (w)");
    return FG21_OK;
}

int device_precompute(DeviceBuild *b, const std::vector<int32_t> &lab, int N, std::vector<double> &A,
                      std::vector<double> &B) {
    b->weighted = true;
    cudaError_t e = b->prepare(false);
    if (e != cudaSuccess) return fail(e, "region building (inputs)");
    const int64_t npix = b->g.npix;
    const int F = b->g.F, T = b->g.T;
    // pixels of each component contiguous, in index order within a component
    std::vector<int64_t> seg(N + 1, 0), perm(npix);
    for (int64_t q = 0; q < npix; ++q) seg[lab[q] + 1]++;
    for (int c = 0; c < N; ++c) seg[c + 1] += seg[c];
    {
        std::vector<int64_t> pos(seg.begin(), seg.end() - 1);
        for (int64_t q = 0; q < npix; ++q) perm[pos[lab[q]]++] = q;
    }
    int64_t *dperm = nullptr, *dseg = nullptr;
    double *dA = nullptr;
    e = b->alloc(&dperm, (size_t)npix);
    if (e == cudaSuccess) e = b->alloc(&dseg, (size_t)N + 1);
    if (e == cudaSuccess) e = b->alloc(&dA, (size_t)N * F * T);
    if (e == cudaSuccess) e = cudaMemcpy(dperm, perm.data(), sizeof(int64_t) * npix, cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(dseg, seg.data(), sizeof(int64_t) * (N + 1), cudaMemcpyHostToDevice);
    // B = (1/Npix) sum_q D: pass 1 of the importance gave it
    if (e == cudaSuccess && !b->summed) e = b->pass1(FG21_WEIGHT_UNIFORM);
    if (e != cudaSuccess) return fail(e, "region building (precompute)");
    resp_kernel<<<(unsigned)(F * T), BUILD_THREADS>>>(b->g, b->t230, dperm, dseg, N, dA);
    if ((e = cudaGetLastError()) != cudaSuccess) return fail(e, "resp_kernel");
    A.resize((size_t)N * F * T);
    B.resize((size_t)F * T);
    if ((e = cudaMemcpy(A.data(), dA, sizeof(double) * A.size(), cudaMemcpyDeviceToHost)) != cudaSuccess ||
        (e = cudaMemcpy(B.data(), b->bsum, sizeof(double) * B.size(), cudaMemcpyDeviceToHost)) != cudaSuccess)
        return fail(e, "region building (A, B)");
    for (auto &x : B) x /= (double)npix;
    return FG21_OK;
}

}  // namespace fg21
