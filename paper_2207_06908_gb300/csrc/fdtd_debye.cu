// fdtd_debye.cu -- dispersive (multi-term Debye) media: the part of the E
// update the step kernels leave out (Kuklin, arXiv 2207.06908, "Dispersive
// media": Debye permittivity by the auxiliary differential equation method
// of its references).
//
// For an edge with poles p the E half step is
//   E^{n+1} = ca E^n + cb curl H^{n+1/2} + sum_p cj_p J_p^n
// and the polarisation currents then advance by the trapezoidal rule
//   J_p^{n+1} = k_p J_p^n + be_p (E^{n+1} - E^n).
// The step kernels compute ca E + cb curl (ca, cb of dispersive edges
// already carry the poles); this kernel, launched after them and before the
// source / probe kernel, adds the current terms and advances the currents.
// It streams the planes that hold dispersive edges: per cell a record byte,
// E^n and E^{n+1} of the dispersive components and their currents.
#include <algorithm>

#include "fdtd_internal.h"

namespace fdtd {
namespace {

// V consecutive floats (V = 2, 4) as one access
template <int V>
struct __align__(4 * V) Vec {
    float v[V];
};

// Each thread takes V consecutive elements of the box (aligned to them: the
// plane is a multiple of 16 elements), issues every load of its dispersive
// components first (E^n, E^{n+1}, the currents), then updates and stores
// them.  Bound by DRAM.  With two to four poles V = 4 holds 96 to 167
// registers and leaves few threads per SM; V = 2 takes 64 to 96 (256^3 with
// half of it soil and four poles, whole step: 331.9 us against 343.5; 128^3
// 54.7 against 57.4, with two poles 43.8 against 45.5).  With one pole the
// wider accesses win (236.2 us against 237.8; 100x100x80 24.1 against 24.6).
template <int NP, int V>
__global__ void __launch_bounds__(256) debye_kernel(const DebyeArgs a)
{
    extern __shared__ float tab[];          // [n_rec][kDebyeRec], then a component mask per record
    int *mask = reinterpret_cast<int *>(tab + a.n_rec * kDebyeRec);
    for (int q = threadIdx.x; q < a.n_rec * kDebyeRec; q += blockDim.x) tab[q] = __ldg(a.table + q);
    __syncthreads();
    constexpr int np = NP;
    for (int r = threadIdx.x; r < a.n_rec; r += blockDim.x) {
        int m = 0;
        for (int c = 0; c < 3; ++c)
            for (int p = 0; p < np; ++p)
                if (tab[r * kDebyeRec + c * kMaxPoles * 3 + 3 * p + 2] != 0.f) m |= 1 << c;
        mask[r] = m;
    }
    step_chain();
    __syncthreads();
    using F = Vec<V>;
    struct __align__(V) Recs {
        uint8_t r[V];
    };
    const Recs *__restrict__ dcls = reinterpret_cast<const Recs *>(a.dcls);
    const long long nv = a.jstride / V;
    for (long long qv = (long long)blockIdx.x * blockDim.x + threadIdx.x; qv < nv;
         qv += (long long)gridDim.x * blockDim.x) {
        const Recs rec = dcls[qv];
        int comps = 0;
#pragma unroll
        for (int t = 0; t < V; ++t) comps |= mask[rec.r[t]];
        if (!comps) continue;
        const long long q = V * qv, g = a.off + q;
        F e0[3], e1[3], jv[3][NP];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (!(comps >> c & 1)) continue;
            e0[c] = *reinterpret_cast<const F *>(a.Ein[c] + g);
            e1[c] = *reinterpret_cast<const F *>(a.Eout[c] + g);
#pragma unroll
            for (int p = 0; p < np; ++p)
                jv[c][p] = *reinterpret_cast<const F *>(a.J + (long long)(c * np + p) * a.jstride + q);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            if (!(comps >> c & 1)) continue;
            F e = e1[c];
#pragma unroll
            for (int t = 0; t < V; ++t) {
                const float *rc = tab + rec.r[t] * kDebyeRec + c * kMaxPoles * 3;
                float v = e.v[t];
#pragma unroll
                for (int p = 0; p < np; ++p) v += rc[3 * p] * jv[c][p].v[t];
#pragma unroll
                for (int p = 0; p < np; ++p)
                    jv[c][p].v[t] = rc[3 * p + 1] * jv[c][p].v[t] + rc[3 * p + 2] * (v - e0[c].v[t]);
                e.v[t] = v;
            }
#pragma unroll
            for (int p = 0; p < np; ++p)
                *reinterpret_cast<F *>(a.J + (long long)(c * np + p) * a.jstride + q) = jv[c][p];
            *reinterpret_cast<F *>(a.Eout[c] + g) = e;
        }
    }
}

template <int NP, int V>
cudaError_t run_debye(const DebyeArgs &a, int sms, cudaStream_t s)
{
    const long long blocks = std::min<long long>((a.jstride / V + 255) / 256, 8LL * sms);
    const size_t smem = (size_t)a.n_rec * (kDebyeRec * sizeof(float) + sizeof(int));
    debye_kernel<NP, V><<<(unsigned)std::max<long long>(blocks, 1), 256, smem, s>>>(a);
    return cudaGetLastError();
}

template <int NP>
cudaError_t run_debye(const DebyeArgs &a, int sms, cudaStream_t s)
{
    return run_debye<NP, (NP >= 2 ? 2 : 4)>(a, sms, s);
}

}  // namespace

cudaError_t launch_debye(const DebyeArgs &a, cudaStream_t s)
{
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            sms = 148;
    }
    switch (a.npoles) {
    case 1: return run_debye<1>(a, sms, s);
    case 2: return run_debye<2>(a, sms, s);
    case 3: return run_debye<3>(a, sms, s);
    case 4: return run_debye<4>(a, sms, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace fdtd
