// Set-up, normalisation, misfit, gradient and adjoint-basis kernels.
#include <cooperative_groups.h>

#include <algorithm>

#include "csem_internal.cuh"
#include "csem_td.cuh"
#include "csem_es.cuh"

namespace csem {

// ---------------------------------------------------------------------------
// Pairs of FP32 values (hi + lo, |lo| <= ulp(hi)/2) for the once-per-run FP32 kernels: Knuth's TwoSum
// and the FMA TwoProduct (Ogita, Rump and Oishi 2005) carry about 48 bits.  FP64 (conversions included)
// issues at 1/64 of the FP32 rate here and bounded these kernels; the pairs leave them to DRAM, and a
// result that is rounded to FP32 at the end is the one FP64 gives but for ties at 2^-48.  Where a pair
// result is not finite (an overflow on the way, an infinity in the input) the entry is computed in FP64.
// ---------------------------------------------------------------------------
struct F2 { float h, l; };
__device__ __forceinline__ F2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
    return F2{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ F2 two_prod(float a, float b) {
    const float p = __fmul_rn(a, b);
    return F2{p, __fmaf_rn(a, b, -p)};
}
// s + a b, the error terms gathered in l
__device__ __forceinline__ void dot_add(F2 &s, float a, float b) {
    const F2 p = two_prod(a, b), t = two_sum(s.h, p.h);
    s.h = t.h;
    s.l = __fadd_rn(s.l, __fadd_rn(t.l, p.l));
}
__device__ __forceinline__ void sum_add(F2 &s, float a) {
    const F2 t = two_sum(s.h, a);
    s.h = t.h;
    s.l = __fadd_rn(s.l, t.l);
}
__device__ __forceinline__ F2 norm2(F2 a) {              // renormalised, |h| >= |l|
    const float s = __fadd_rn(a.h, a.l);
    return F2{s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 p = two_prod(a.h, b.h);
    p.l = __fmaf_rn(a.h, b.l, __fmaf_rn(a.l, b.h, p.l));
    return norm2(p);
}
__device__ __forceinline__ F2 div2(F2 a, float b) {      // one correction of the FP32 quotient
    const float q = __fdiv_rn(a.h, b);
    const float r = __fadd_rn(__fmaf_rn(-q, b, a.h), a.l);
    return norm2(F2{q, __fdiv_rn(r, b)});
}
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }
__device__ __forceinline__ F2 split2(double a) {
    const float h = (float)a;
    return F2{h, (float)(a - (double)h)};
}

// ---------------------------------------------------------------------------
// rho (cells) -> dt/eps on every E edge, eps = sigma_e / (2 w0)  (Sec. 2, Eq. 2)
// sigma_e = sum_c V_c / rho_c / sum_c V_c over the (up to four) cells sharing e.
// ---------------------------------------------------------------------------
// the general evaluation of one edge (component c at lattice node i, j, k), in FP64
template <typename R>
__device__ R edge_coef(const GeoD &g, const R *__restrict__ rho, const R *__restrict__ rho_z, int c, int i, int j,
                       int k, double two_w0_dt, int *bad) {
    double num = 0.0, den = 0.0;
    // cell offsets for each component: Ex spans (j-1..j, k-1..k) at cell column i, etc.
    int i0 = i, i1 = i, j0 = j, j1 = j, k0 = k, k1 = k;
    bool on = false;
    if (c == 0) { on = (i < g.nx); j0 = j - 1; k0 = k - 1; }
    if (c == 1) { on = (j < g.ny); i0 = i - 1; k0 = k - 1; }
    if (c == 2) { on = (k < g.nz); i0 = i - 1; j0 = j - 1; }
    if (!on || i >= g.NX) return R(0);
    for (int kk = k0; kk <= k1; ++kk)
        for (int jj = j0; jj <= j1; ++jj)
            for (int ii = i0; ii <= i1; ++ii) {
                if (ii < 0 || jj < 0 || kk < 0 || ii >= g.nx || jj >= g.ny || kk >= g.nz) continue;
                const double V = g.hx[ii] * g.hy[jj] * g.hz[kk];
                const double rc = (double)(c == 2 ? rho_z : rho)[((long long)kk * g.ny + jj) * g.nx + ii];
                if (!(rc > 0.0) || !isfinite(rc)) atomicOr(bad, 1);
                num += V / rc;
                den += V;
            }
    return (den > 0.0 && num > 0.0) ? (R)(two_w0_dt * den / num) : R(0);
}

template <typename R>
__global__ void k_coef_init(const GeoD g, const R *__restrict__ rho, const R *__restrict__ rho_z,
                            R *__restrict__ cE, double two_w0_dt, int *bad) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (t >= g.vol) return;
    const int i = (int)(t % g.pitch);
    const long long r = t / g.pitch;
    cE[(long long)c * g.vol + t] = edge_coef<R>(g, rho, rho_z, c, i, (int)(r % g.NY), (int)(r / g.NY), two_w0_dt, bad);
}

// FP32 contexts: dt/eps of a node's three edges, and its copy cEm with the PEC edges zeroed (Ex needs
// 1 <= j < ny, 1 <= k < nz; Ey 1 <= i < nx, 1 <= k < nz; Ez 1 <= i < nx, 1 <= j < ny; cEm may be NULL), from
// V/rho as pairs of the seven cells that the edges share.  FP64 divisions bounded the general kernel (four
// per edge); a resistivity that is bad or outside the range of pairs sends its node's edges to it.  Towline:
// 3.1 ms (with a second kernel for the masked copy), 0.30 ms now.
template <bool VTI>
__global__ void __launch_bounds__(128) k_coef_init32(const GeoD g, const float *__restrict__ rho,
                                                     const float *__restrict__ rho_z, float *__restrict__ cE,
                                                     float *__restrict__ cEm, double two_w0_dt, int *bad) {
    __shared__ F2 yz[4], scale;          // hy hz of the cells (j-1+b, k-1+c) at b + 2c, zero off the grid; 2 w0 dt
    const int i = blockIdx.x * 128 + threadIdx.x, j = blockIdx.y, k = blockIdx.z;
    if (threadIdx.x < 4) {
        const int jj = j - 1 + (threadIdx.x & 1), kk = k - 1 + (threadIdx.x >> 1);
        yz[threadIdx.x] = (jj >= 0 && jj < g.ny && kk >= 0 && kk < g.nz) ? split2(g.hy[jj] * g.hz[kk]) : F2{0.f, 0.f};
    }
    if (threadIdx.x == 4) scale = split2(two_w0_dt);
    __syncthreads();
    if (i >= g.pitch) return;
    const bool x0 = i >= 1 && i <= g.nx, x1 = i < g.nx;       // cells i-1, i are on the grid
    const F2 hx[2] = {x0 ? split2(g.hx[i - 1]) : F2{0.f, 0.f}, x1 ? split2(g.hx[i]) : F2{0.f, 0.f}};
    // volume and V/rho of the cell (i-1+a, j-1+b, k-1+c) at a + 2b + 4c, zero off the grid
    F2 V[8], q[8], qz[VTI ? 8 : 1];
    bool plain = true;
#pragma unroll
    for (int u = 1; u < 8; ++u) {
        const int a = u & 1, b = (u >> 1) & 1, c = u >> 2;
        const F2 w = yz[b + 2 * c];
        V[u] = q[u] = F2{0.f, 0.f};
        if (VTI) qz[u] = F2{0.f, 0.f};
        if ((a ? x1 : x0) && w.h > 0.f) {
            const long long o = ((long long)(k - 1 + c) * g.ny + (j - 1 + b)) * g.nx + (i - 1 + a);
            V[u] = mul2(hx[a], w);
            const float r = __ldg(rho + o);
            plain = plain && r > 1e-12f && r < 1e12f && V[u].h > 1e-18f && V[u].h < 1e24f;
            q[u] = div2(V[u], r);
            if (VTI && c == 1) {         // the z edge lies between cells of plane k
                const float rz = __ldg(rho_z + o);
                plain = plain && rz > 1e-12f && rz < 1e12f;
                qz[u] = div2(V[u], rz);
            }
        }
    }
    auto edge = [&](const F2 *n, int a, int b, int c, int d) -> float {     // 2 w0 dt sum V / sum V/rho
        F2 sn = n[a], sd = V[a];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
            const int u = m == 0 ? b : (m == 1 ? c : d);
            sum_add(sn, n[u].h); sn.l += n[u].l;
            sum_add(sd, V[u].h); sd.l += V[u].l;
        }
        if (!(sn.h > 0.f)) return 0.f;
        const F2 w = mul2(norm2(sd), scale);
        sn = norm2(sn);
        const float t = __fdiv_rn(w.h, sn.h);
        const float r = __fadd_rn(__fmaf_rn(-t, sn.h, w.h), __fmaf_rn(-t, sn.l, w.l));
        return __fadd_rn(t, __fdiv_rn(r, sn.h));
    };
    float cx = edge(q, 1, 3, 5, 7), cy = edge(q, 2, 3, 6, 7), cz = edge(VTI ? qz : q, 4, 5, 6, 7);
    if (!plain || !isfinite(cx) || !isfinite(cy) || !isfinite(cz)) {
        cx = edge_coef<float>(g, rho, rho_z, 0, i, j, k, two_w0_dt, bad);
        cy = edge_coef<float>(g, rho, rho_z, 1, i, j, k, two_w0_dt, bad);
        cz = edge_coef<float>(g, rho, rho_z, 2, i, j, k, two_w0_dt, bad);
    }
    const long long t = ((long long)k * g.NY + j) * g.pitch + i;
    cE[t] = cx; cE[g.vol + t] = cy; cE[2 * g.vol + t] = cz;
    if (cEm) {
        const bool xi = i >= 1 && i < g.nx, yi = j >= 1 && j < g.ny, zi = k >= 1 && k < g.nz;
        cEm[t] = (i < g.nx && yi && zi) ? cx : 0.f;
        cEm[g.vol + t] = (xi && j < g.ny && zi) ? cy : 0.f;
        cEm[2 * g.vol + t] = (xi && yi && k < g.nz) ? cz : 0.f;
    }
}

template <typename R>
cudaError_t launch_coef_init(const GeoD &g, const R *rho, const R *rho_z, R *cE, R *cEm, bool *masked,
                             double two_w0_dt, int *bad, cudaStream_t st) {
    g_launches++;
    *masked = false;
    if constexpr (sizeof(R) == 4) {
        const double scale = two_w0_dt;
        if (g.NY <= 65535 && g.NZ <= 65535 && scale > 1e-15 && scale < 1e15) {
            const dim3 grid((unsigned)((g.pitch + 127) / 128), (unsigned)g.NY, (unsigned)g.NZ);
            if (rho_z == rho) k_coef_init32<false><<<grid, 128, 0, st>>>(g, rho, rho_z, cE, cEm, scale, bad);
            else k_coef_init32<true><<<grid, 128, 0, st>>>(g, rho, rho_z, cE, cEm, scale, bad);
            *masked = cEm != nullptr;
            return cudaGetLastError();
        }
    }
    dim3 grid((unsigned)((g.vol + 255) / 256), 3);
    k_coef_init<R><<<grid, 256, 0, st>>>(g, rho, rho_z, cE, two_w0_dt, bad);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// normalisation of volumes: out = alpha_k * (acc - comp)   (Sec. 2, Eq. 3)
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_finalize_volume(typename C2<R>::T *acc, const typename C2<R>::T *comp, long long vol, int S,
                                  int nf, const double2 *alpha) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= vol) return;
    const int sc = blockIdx.y;           // s*3 + c
    for (int f = 0; f < nf; ++f) {
        const long long o = ((long long)sc * nf + f) * vol + t;
        typename C2<R>::T a = acc[o];
        double ar = a.x, ai = a.y;
        if (comp) { ar -= comp[o].x; ai -= comp[o].y; }
        const double2 al = alpha[f];
        a.x = (R)(al.x * ar - al.y * ai);
        a.y = (R)(al.x * ai + al.y * ar);
        acc[o] = a;
    }
}

// FP32: two entries per thread, the difference acc - comp exact as a pair, the product with alpha (a pair
// per part) in pairs.  Bound by DRAM: 24 B per entry with compensation.  2 sources x 4 frequencies of the
// 256 x 256 x 128 towline: 4.3 ms in FP64, 0.76 ms now (6.6 TB/s).
template <bool COMP>
__global__ void __launch_bounds__(256) k_finalize_volume32(float4 *__restrict__ acc, const float4 *__restrict__ comp,
                                                           long long half, int nf, const double2 *__restrict__ alpha) {
    __shared__ F2 as[2];                 // alpha as pairs, split once per block (FP64)
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const double2 al = __ldg(alpha + blockIdx.y % nf);
    if (threadIdx.x < 2) as[threadIdx.x] = split2(threadIdx.x ? al.y : al.x);
    __syncthreads();
    if (t >= half) return;
    const F2 ar = as[0], ai = as[1], an = F2{-ai.h, -ai.l};
    const float big = fmaxf(fabsf(ar.h), fabsf(ai.h));
    const bool wide = !(big > 1e-20f && big < 1e20f);   // a normalisation outside the range of pairs
    const long long o = (long long)blockIdx.y * half + t;
    float4 a = acc[o];
    const float4 c = COMP ? __ldcs(comp + o) : make_float4(0.f, 0.f, 0.f, 0.f);
    auto one = [&](float re, float im, float cr, float ci) {
        const F2 x = COMP ? two_sum(re, -cr) : F2{re, 0.f}, y = COMP ? two_sum(im, -ci) : F2{im, 0.f};
        auto dot = [&](F2 u, F2 v) {     // u x + v y
            F2 s = two_prod(u.h, x.h);
            dot_add(s, v.h, y.h);
            s.l = __fadd_rn(s.l, __fadd_rn(__fmaf_rn(u.h, x.l, __fmul_rn(u.l, x.h)), __fmaf_rn(v.h, y.l, __fmul_rn(v.l, y.h))));
            return __fadd_rn(s.h, s.l);
        };
        float2 r = make_float2(dot(ar, an), dot(ai, ar));
        if (wide || !isfinite(r.x) || !isfinite(r.y)) {
            const double dr = COMP ? (double)re - (double)cr : (double)re, di = COMP ? (double)im - (double)ci : (double)im;
            r = make_float2((float)(al.x * dr - al.y * di), (float)(al.x * di + al.y * dr));
        }
        return r;
    };
    const float2 u = one(a.x, a.y, c.x, c.y), v = one(a.z, a.w, c.z, c.w);
    acc[o] = make_float4(u.x, u.y, v.x, v.y);
}

template <typename R>
cudaError_t launch_finalize_volume(typename C2<R>::T *acc, const typename C2<R>::T *comp, long long vol, int S,
                                   int nf, const double2 *alpha, cudaStream_t st) {
    if constexpr (sizeof(R) == 4) {      // vol is a multiple of the pitch, so of 8; the volumes may be on any 8 bytes
        if (aligned16(acc) && aligned16(comp) && (long long)S * 3 * nf <= 65535) {
            const long long half = vol / 2;
            const dim3 g2((unsigned)((half + 255) / 256), (unsigned)(S * 3 * nf));
            if (comp) k_finalize_volume32<true><<<g2, 256, 0, st>>>((float4 *)acc, (const float4 *)comp, half, nf, alpha);
            else k_finalize_volume32<false><<<g2, 256, 0, st>>>((float4 *)acc, nullptr, half, nf, alpha);
            g_launches++;
            return cudaGetLastError();
        }
    }
    dim3 grid((unsigned)((vol + 255) / 256), (unsigned)(S * 3));
    k_finalize_volume<R><<<grid, 256, 0, st>>>(acc, comp, vol, S, nf, alpha);
    g_launches++;
    return cudaGetLastError();
}

__global__ void k_finalize_receivers(const double2 *racc, double *out, int n, int nf, const double2 *alpha) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const double2 a = racc[t], al = alpha[t % nf];
    out[2 * t] = al.x * a.x - al.y * a.y;
    out[2 * t + 1] = al.x * a.y + al.y * a.x;
}

cudaError_t launch_finalize_receivers(const double2 *racc, double *out, int S, int n_rec, int nf,
                                      const double2 *alpha, cudaStream_t st) {
    const int n = S * n_rec * nf;
    if (n == 0) return cudaSuccess;
    k_finalize_receivers<<<(n + 255) / 256, 256, 0, st>>>(racc, out, n, nf, alpha);
    g_launches++;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// adjoint series coefficients: c_k = k_k conj(r_k) / dt -> [Re c; Im c]  (Sec. 3.2-3.3)
// ---------------------------------------------------------------------------
__global__ void k_adjoint_coef(const double *resid, double *coef, int n, int nf, const double2 *kf, double inv_dt) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;   // (s, r, f)
    if (t >= n) return;
    const int f = t % nf;
    const int sr = t / nf;
    const double rr = resid[2 * t], ri = -resid[2 * t + 1];   // conj(r)
    const double2 k = kf[f];
    coef[(long long)sr * 2 * nf + f] = (k.x * rr - k.y * ri) * inv_dt;
    coef[(long long)sr * 2 * nf + nf + f] = (k.x * ri + k.y * rr) * inv_dt;
}

cudaError_t launch_adjoint_coef(const double *resid, double *coef, int S, int n_rec, int nf, const double2 *kf,
                                double inv_dt, cudaStream_t st) {
    const int n = S * n_rec * nf;
    k_adjoint_coef<<<(n + 255) / 256, 256, 0, st>>>(resid, coef, n, nf, kf, inv_dt);
    g_launches++;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// gradient (Sec. 3.1 isotropic form, Sec. 3.5 chain rule)
//   edge:  p_e = -Re sum_s sum_k conj(v)_{e,k} E_{e,k}
//   cell:  dphi/dsigma_c = V_c / 4 * sum of p_e over the 12 edges of c
// (dV_e / sum_{c at e} V_c = 1/4 on every edge that carries a field; the
// outer-boundary edges hold E = 0.)
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_grad_edge(const typename C2<R>::T *E, const typename C2<R>::T *V, long long vol, int S, int nf,
                            R *pe) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (t >= vol) return;
    double acc = 0.0;
    for (int s = 0; s < S; ++s)
        for (int f = 0; f < nf; ++f) {
            const long long o = (((long long)s * 3 + c) * nf + f) * vol + t;
            const typename C2<R>::T e = E[o], v = V[o];
            acc += (double)v.x * (double)e.x - (double)v.y * (double)e.y;
        }
    pe[(long long)c * vol + t] = (R)(-acc);
}

// FP32: two entries per thread, the sum over sources and frequencies as a pair.  Bound by DRAM (16 B per
// entry, source and frequency).  Towline, 2 sources x 4 frequencies: 2.6 ms with FP64 sums, 0.475 ms now
// (7.1 TB/s).
__global__ void __launch_bounds__(256) k_grad_edge32(const float4 *__restrict__ E, const float4 *__restrict__ V,
                                                     long long half, int S, int nf, float2 *__restrict__ pe) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int c = blockIdx.y;
    if (t >= half) return;
    // scaled (exactly) so that the low parts of products of small fields stay normal numbers
    constexpr float kUp = 18446744073709551616.f, kDown = 1.f / kUp;
    F2 a{0.f, 0.f}, b{0.f, 0.f};
    for (int s = 0; s < S; ++s) {
        const long long o = ((long long)s * 3 + c) * nf * half + t;
#pragma unroll 4
        for (int f = 0; f < nf; ++f) {
            float4 e = __ldcs(E + o + f * half);
            const float4 v = __ldcs(V + o + f * half);
            e.x *= kUp; e.y *= kUp; e.z *= kUp; e.w *= kUp;
            dot_add(a, v.x, e.x);
            dot_add(a, -v.y, e.y);
            dot_add(b, v.z, e.z);
            dot_add(b, -v.w, e.w);
        }
    }
    auto down = [&](F2 u) {              // rounded once, also where the result is subnormal
        const float w = -__fadd_rn(u.h, u.l) * kDown;
        return fabsf(w) < 2.4e-38f ? (float)(-((double)u.h + (double)u.l) * (double)kDown) : w;
    };
    float2 r = make_float2(down(a), down(b));
    if (!isfinite(r.x) || !isfinite(r.y)) {
        double x = 0.0, y = 0.0;
        for (int s = 0; s < S; ++s)
            for (int f = 0; f < nf; ++f) {
                const long long o = (((long long)s * 3 + c) * nf + f) * half + t;
                const float4 e = E[o], v = V[o];
                x += (double)v.x * (double)e.x - (double)v.y * (double)e.y;
                y += (double)v.z * (double)e.z - (double)v.w * (double)e.w;
            }
        r = make_float2((float)-x, (float)-y);
    }
    pe[c * half + t] = r;
}

// FP32 cells: the twelve edges' sum, the volume and the quotient as pairs (grad_v as in k_grad_cell).  A
// thread takes one column of kCellK planes, so that the FP64 work is a few operations per column.  Towline:
// 690 us in FP64, 112 us now.
constexpr int kCellK = 8;
__global__ void __launch_bounds__(128) k_grad_cell32(const GeoD g, const float *__restrict__ pe,
                                                     const float *__restrict__ rho, const float *__restrict__ rho_v,
                                                     int wrt, float *grad, float *grad_v) {
    __shared__ F2 yz[kCellK];            // hy hz / 4 of the block's rows
    const int i = blockIdx.x * 128 + threadIdx.x, j = blockIdx.y, k0 = blockIdx.z * kCellK;
    const int nk = min(kCellK, g.nz - k0);
    if ((int)threadIdx.x < nk) yz[threadIdx.x] = split2(0.25 * g.hy[j] * g.hz[k0 + threadIdx.x]);
    __syncthreads();
    if (i >= g.nx) return;
    const F2 hx = split2(g.hx[i]);
    const long long dy = g.pitch, dz = g.plane;
    const float *px = pe + ((long long)k0 * g.NY + j) * g.pitch + i, *py = px + g.vol, *pz = py + g.vol;
    long long t = ((long long)k0 * g.ny + j) * g.nx + i;
    for (int m = 0; m < nk; ++m, px += dz, py += dz, pz += dz, t += (long long)g.ny * g.nx) {
        const float e[12] = {px[0], py[0], px[dy], py[1], px[dz], py[dz], px[dy + dz], py[1 + dz],
                             pz[0], pz[1], pz[dy], pz[dy + 1]};
        const F2 V = mul2(hx, yz[m]);
        auto out = [&](int lo, int hi, const float *r, float *d) {
            F2 s{e[lo], 0.f};
#pragma unroll
            for (int u = 1; u < 12; ++u)
                if (u > lo && u < hi) sum_add(s, e[u]);
            const float rc = wrt == 1 ? r[t] : 1.f;
            F2 q = mul2(norm2(s), V);
            if (wrt == 1) { q = div2(q, rc); q.h = -q.h; q.l = -q.l; }
            float v = __fadd_rn(q.h, q.l);
            if (!isfinite(v)) {
                double w = 0.0;
                for (int u = lo; u < hi; ++u) w += (double)e[u];
                w *= 0.25 * g.hx[i] * g.hy[j] * g.hz[k0 + m];
                v = (float)(wrt == 1 ? -w / (double)rc : w);
            }
            d[t] += v;
        };
        if (grad_v) {
            out(0, 8, rho, grad);
            out(8, 12, rho_v, grad_v);
        } else {
            out(0, 12, rho, grad);
        }
    }
}

// rho_v, grad_v non-null: VTI, the x and y edges feed grad (sigma_h), the z edges grad_v (sigma_v)
template <typename R>
__global__ void k_grad_cell(const GeoD g, const R *pe, const R *rho, const R *rho_v, int wrt, R *grad, R *grad_v) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long cells = (long long)g.nx * g.ny * g.nz;
    if (t >= cells) return;
    const int i = (int)(t % g.nx);
    const long long r = t / g.nx;
    const int j = (int)(r % g.ny);
    const int k = (int)(r / g.ny);
    const R *px = pe, *py = pe + g.vol, *pz = pe + 2 * g.vol;
    auto at = [&](int ii, int jj, int kk) { return ((long long)kk * g.NY + jj) * g.pitch + ii; };
    double sh = 0.0, sv = 0.0;
    for (int d1 = 0; d1 < 2; ++d1)
        for (int d0 = 0; d0 < 2; ++d0) {
            sh += (double)px[at(i, j + d0, k + d1)];
            sh += (double)py[at(i + d0, j, k + d1)];
            sv += (double)pz[at(i + d0, j + d1, k)];
        }
    const double V = g.hx[i] * g.hy[j] * g.hz[k];
    if (grad_v) {
        double gh = 0.25 * V * sh, gv = 0.25 * V * sv;   // d phi / d sigma_h, d phi / d sigma_v
        if (wrt == 1) { gh = -gh / (double)rho[t]; gv = -gv / (double)rho_v[t]; }
        grad[t] += (R)gh;
        grad_v[t] += (R)gv;
        return;
    }
    double gs = 0.25 * V * (sh + sv);           // d phi / d sigma_c
    if (wrt == 1) gs = -gs / (double)rho[t];    // d phi / d ln rho_c = -sigma_c d phi / d sigma_c
    grad[t] += (R)gs;
}

template <typename R>
cudaError_t launch_grad_cells(const GeoD &g, const R *rho, const R *pe, int wrt, bool vti, R *grad, cudaStream_t st) {
    const long long cells = (long long)g.nx * g.ny * g.nz;
    const R *rho_v = vti ? rho + cells : nullptr;
    R *grad_v = vti ? grad + cells : nullptr;
    if constexpr (sizeof(R) == 4) {
        if (g.ny <= 65535 && g.nz <= 65535) {
            const dim3 grid((unsigned)((g.nx + 127) / 128), (unsigned)g.ny, (unsigned)((g.nz + kCellK - 1) / kCellK));
            k_grad_cell32<<<grid, 128, 0, st>>>(g, pe, rho, rho_v, wrt, grad, grad_v);
            g_launches++;
            return cudaGetLastError();
        }
    }
    k_grad_cell<R><<<(unsigned)((cells + 255) / 256), 256, 0, st>>>(g, pe, rho, rho_v, wrt, grad, grad_v);
    g_launches++;
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_gradient(const GeoD &g, const R *rho, const typename C2<R>::T *E, const typename C2<R>::T *V,
                            int S, int nf, int wrt, bool vti, R *edge_scratch, R *grad, cudaStream_t st) {
    bool pairs = false;
    if constexpr (sizeof(R) == 4) {      // the volumes may be on any 8 bytes
        pairs = aligned16(E) && aligned16(V);
        const dim3 ge((unsigned)((g.vol / 2 + 255) / 256), 3);
        if (pairs)
            k_grad_edge32<<<ge, 256, 0, st>>>((const float4 *)E, (const float4 *)V, g.vol / 2, S, nf, (float2 *)edge_scratch);
    }
    if (!pairs) {
        const dim3 ge((unsigned)((g.vol + 255) / 256), 3);
        k_grad_edge<R><<<ge, 256, 0, st>>>(E, V, g.vol, S, nf, edge_scratch);
    }
    g_launches++;
    return launch_grad_cells<R>(g, rho, edge_scratch, wrt, vti, grad, st);
}

// ---------------------------------------------------------------------------
// early end of a forward data run: convergence of the running receiver transform
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_es_check(const double2 *racc, double2 *prev, double2 *fin, int n,
                                                  double tol, int chunk, int last, int steps_at, int *state) {
    __shared__ int moved;
    if (state[0]) return;                      // already ended: the kept spectra stay
    if (threadIdx.x == 0) moved = (chunk == 0) ? 1 : 0;
    __syncthreads();
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const double2 a = racc[t], b = prev[t];
        const double dr = a.x - b.x, di = a.y - b.y;
        if (sqrt(dr * dr + di * di) > tol * sqrt(a.x * a.x + a.y * a.y)) moved = 1;
    }
    __syncthreads();
    const bool done = !moved || last;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const double2 a = racc[t];
        prev[t] = a;
        if (done) fin[t] = a;
    }
    if (done && threadIdx.x == 0) {
        state[1] = steps_at;
        state[0] = 1;
    }
}

cudaError_t launch_es_check(const double2 *racc, double2 *prev, double2 *fin, int n, double tol, int chunk,
                            int last, int steps_at, int *state, cudaStream_t st) {
    k_es_check<<<1, 256, 0, st>>>(racc, prev, fin, n, tol, chunk, last, steps_at, state);
    g_launches++;
    return cudaGetLastError();
}

template <typename R>
__global__ void __launch_bounds__(256) k_es_vol_stats(const typename C2<R>::T *acc, typename C2<R>::T *prev,
                                                      long long vol, int nf, float tol, float floor_frac,
                                                      EsTail tail, unsigned *stats) {
    const int blk = blockIdx.y;                       // (s*3 + c)*nf + f
    const int f = blk % nf;
    const long long base = (long long)blk * vol;
    // entries below floor_frac of the frequency's largest magnitude at the previous check are
    // held to an absolute bound (the decision is taken in FP32)
    const float floor_a = floor_frac * __uint_as_float(stats[2 * nf + f]);
    const float tf = tail.f[f];                       // remainder per unit change (geometric tail)
    float amax = 0.f;
    unsigned viol = 0u;
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < vol; e += (long long)gridDim.x * blockDim.x) {
        const typename C2<R>::T a = acc[base + e], b = prev[base + e];
        const float am = hypotf((float)a.x, (float)a.y);
        const float dm = hypotf((float)(a.x - b.x), (float)(a.y - b.y)) * tf;
        amax = fmaxf(amax, am);
        if (dm > tol * fmaxf(am, floor_a)) viol = 1u;
        prev[base + e] = a;
    }
    for (int o = 16; o > 0; o >>= 1) {
        amax = fmaxf(amax, __shfl_down_sync(0xffffffffu, amax, o));
        viol |= __shfl_down_sync(0xffffffffu, viol, o);
    }
    __shared__ float sa[8];
    __shared__ unsigned sv[8];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { sa[wid] = amax; sv[wid] = viol; }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) { amax = fmaxf(amax, sa[k]); viol |= sv[k]; }
        atomicMax(stats + f, __float_as_uint(amax));          // non-negative floats order like their bits
        if (viol) atomicOr(stats + nf + f, 1u);
    }
}

template <typename R>
cudaError_t launch_es_vol_stats(const typename C2<R>::T *acc, typename C2<R>::T *prev, long long vol, int S, int nf,
                                double tol, double floor_frac, const EsTail &tail, unsigned *stats, cudaStream_t st) {
    const dim3 grid((unsigned)std::min<long long>((vol + 255) / 256, 64), (unsigned)(S * 3 * nf));
    k_es_vol_stats<R><<<grid, 256, 0, st>>>(acc, prev, vol, nf, (float)tol, (float)floor_frac, tail, stats);
    g_launches++;
    return cudaGetLastError();
}

__global__ void k_es_vol_decide(unsigned *stats, int nf, int chunk, int last, int steps_at, int *state) {
    if (state[0]) return;
    bool done = last != 0;
    if (!done && chunk >= 1) {
        done = true;
        for (int f = 0; f < nf; ++f)
            if (stats[nf + f]) done = false;
    }
    for (int f = 0; f < nf; ++f) stats[2 * nf + f] = stats[f];   // this check's maxima for the next one
    if (done) { state[1] = steps_at; state[0] = 1; }
}

cudaError_t launch_es_vol_decide(unsigned *stats, int nf, int chunk, int last, int steps_at, int *state,
                                 cudaStream_t st) {
    k_es_vol_decide<<<1, 1, 0, st>>>(stats, nf, chunk, last, steps_at, state);
    g_launches++;
    return cudaGetLastError();
}

template cudaError_t launch_es_vol_stats<float>(const float2 *, float2 *, long long, int, int, double, double,
                                                const EsTail &, unsigned *, cudaStream_t);
template cudaError_t launch_es_vol_stats<double>(const double2 *, double2 *, long long, int, int, double, double,
                                                 const EsTail &, unsigned *, cudaStream_t);

// ---------------------------------------------------------------------------
// misfit and weighted residual (Sec. 3.1, Eq. 7), one block
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) k_misfit(int n, const double *dobs, const double *dsyn, const double *w,
                                                 double *resid, double *phi) {
    __shared__ double red[32];
    double acc = 0.0;
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const double wt = w ? w[t] : 1.0;
        const double rr = dobs[2 * t] - dsyn[2 * t], ri = dobs[2 * t + 1] - dsyn[2 * t + 1];
        acc += wt * wt * (rr * rr + ri * ri);
        resid[2 * t] = wt * wt * rr;
        resid[2 * t + 1] = wt * wt * ri;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
        acc = (threadIdx.x < (blockDim.x >> 5)) ? red[threadIdx.x] : 0.0;
        for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
        if (threadIdx.x == 0) *phi = 0.5 * acc;
    }
}

cudaError_t launch_misfit(int n, const double *d_obs, const double *d_syn, const double *w, double *resid,
                          double *phi, cudaStream_t st) {
    k_misfit<<<1, 1024, 0, st>>>(n, d_obs, d_syn, w, resid, phi);
    g_launches++;
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Adjoint-source basis (Sec. 3.3), FP64.  The samples are cut into kBT contiguous ranges, one per
// (virtual) thread.  Within a range exp((-1+i) a_k t_n) advances by the complex factor
// exp((-1+i) a_k dt) per sample (the start of each range is evaluated directly).  Rows 0..nf-1 of B
// are the real parts, nf..2nf-1 the imaginary parts.
//
// What bounds it is the FP64 pipe (a warp instruction holds it for tens of cycles) and, between
// passes, latency.  So the phasors are evaluated once into a table that every pass of every column
// reads (k_basis_table; re-evaluating them cost two thirds of a pass's operations and two sincos and
// exp per range and pass), and a column's kBT ranges are spread over a cluster of eight SMs that
// keeps the column's CG vectors in shared memory (k_basis_cg).  Every sum is taken over the ranges
// in the order of one block of kBT threads, so the results are those of that block.  Eight
// frequencies, 19 492 steps, three solves of up to 200 iterations: 469 ms with one block per column
// and phasors advanced in every pass, 43 ms now.
// ---------------------------------------------------------------------------
constexpr int kBT = 512;                 // ranges per column
constexpr int kBC = 8;                   // SMs (CTAs of a cluster) per column
constexpr int kBW = kBT / kBC;           // ranges (threads) per CTA
constexpr int kBMaxChunk = 128;          // samples per range that fit in shared memory: 3 vectors x 64 x 128 x 8 B

struct BasisArgs {
    double dt; int nt; int nf; double a[kMaxFreq];
};

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double block_sum(double v, double *red) {
    v = warp_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    return s;
}

// z_k(n0) = exp((-1+i) a_k (n0+1/2) dt), step factor q_k = exp((-1+i) a_k dt)
__device__ __forceinline__ void phasor_start(const BasisArgs &b, int f, int n0, double &zr, double &zi, double &qr,
                                             double &qi) {
    const double t = (n0 + 0.5) * b.dt;
    double sn, cs;
    sincos(b.a[f] * t, &sn, &cs);
    const double e = exp(-b.a[f] * t);
    zr = e * cs; zi = e * sn;
    sincos(b.a[f] * b.dt, &sn, &cs);
    const double eq = exp(-b.a[f] * b.dt);
    qr = eq * cs; qi = eq * sn;
}

// Z[(m*nf + f)*kBT + t]: the phasor of frequency f at sample m of range t (zero past the last sample).
__global__ void __launch_bounds__(64) k_basis_table(BasisArgs b, int chunk, double2 *Z) {
    const int t = blockIdx.x * 64 + threadIdx.x, f = blockIdx.y;
    const int n0 = t * chunk, n1 = min(n0 + chunk, b.nt);
    double zr, zi, qr, qi;
    phasor_start(b, f, n0, zr, zi, qr, qi);
    for (int m = 0; m < chunk; ++m) {
        Z[((long long)m * b.nf + f) * kBT + t] = n0 + m < n1 ? make_double2(zr, zi) : make_double2(0.0, 0.0);
        const double u = zr * qr - zi * qi; zi = zr * qi + zi * qr; zr = u;
    }
}

// Gram matrix G = B B^T (2nf x 2nf), one block per (row, col) pair with row <= col.
__global__ void __launch_bounds__(kBT) k_basis_gram(int nt, int nf, int chunk, const double2 *__restrict__ Z, double *G) {
    __shared__ double red[kBT / 32];
    const int m = 2 * nf;
    const int r = blockIdx.x, c = blockIdx.y;
    if (r > c) return;
    const int n0 = threadIdx.x * chunk, n1 = min(n0 + chunk, nt);
    const double2 *zr = Z + (long long)(r % nf) * kBT + threadIdx.x, *zc = Z + (long long)(c % nf) * kBT + threadIdx.x;
    double acc = 0.0;
    for (int n = n0; n < n1; ++n) {
        const long long o = (long long)(n - n0) * nf * kBT;
        const double2 a = zr[o], b = zc[o];
        acc += (r < nf ? a.x : a.y) * (c < nf ? b.x : b.y);
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0) { G[r * m + c] = acc; G[c * m + r] = acc; }
}

// gamma = gamma_rel * lambda_max(G) by power iteration (G is symmetric positive semi-definite), one row
// per lane; ends early once the vector repeats exactly.
__global__ void __launch_bounds__(32) k_basis_gamma(const double *G, int m, double gamma, int rel, double *out) {
    __shared__ double v[2 * kMaxFreq], w[2 * kMaxFreq];
    const int i = threadIdx.x;
    if (!rel) {
        if (i == 0) out[0] = gamma;
        return;
    }
    double g[2 * kMaxFreq];
#pragma unroll
    for (int j = 0; j < 2 * kMaxFreq; ++j) g[j] = (i < m && j < m) ? G[i * m + j] : 0.0;
    if (i < m) v[i] = 1.0 / (1.0 + i);
    __syncwarp();
    double lam = 0.0;
    for (int it = 0; it < 500; ++it) {
        double s = 0.0;
#pragma unroll
        for (int j = 0; j < 2 * kMaxFreq; ++j)
            if (j < m) s += g[j] * v[j];
        if (i < m) w[i] = s;
        __syncwarp();
        double nrm = 0.0;
#pragma unroll
        for (int j = 0; j < 2 * kMaxFreq; ++j)
            if (j < m) nrm += w[j] * w[j];
        nrm = sqrt(nrm);
        if (nrm == 0.0) break;
        bool same = true;
        if (i < m) {
            const double u = s / nrm;
            same = u == v[i];
            v[i] = u;
        }
        lam = nrm;
        __syncwarp();
        if (__all_sync(0xffffffffu, same)) break;   // a fixed point: the remaining iterations repeat this one
    }
    if (i == 0) out[0] = gamma * lam;
}

// CGNR on (B^T B + gamma I) x = B^T e_j, one cluster of kBC CTAs per column j (Sec. 3.3); x is written
// into basis[n*2nf + j], then the fit max_i |(B x)_i - delta_ij|.  CTA r of the cluster holds the ranges
// r*kBW ..; the vectors x, p, s are in shared memory as [sample][thread].  A sum over all ranges: every
// warp writes its partial sum into the table of every CTA, one cluster barrier, and each CTA adds the
// partial sums in range order.  Two tables in turn, so one barrier per exchange is enough.
// The roundings are spelled out (which products are fused), so that they do not depend on unrolling.
__device__ __forceinline__ double add_dot2(double s, double2 z, double r, double i) {
    return __dadd_rn(s, fma(z.x, r, __dmul_rn(z.y, i)));
}
template <int NF>
__global__ void __cluster_dims__(kBC, 1, 1) __launch_bounds__(kBW)
    k_basis_cg(int nt, int chunk, const double2 *__restrict__ Z, const double *gamma_p, int max_iter, double tol,
               double *basis, int *iters, double *fit) {
    namespace cg = cooperative_groups;
    constexpr int M = 2 * NF, NWT = kBT / 32, U = NF > 5 ? 2 : 4;
    extern __shared__ double sm[];
    __shared__ double tab[2][M + 1][NWT];
    __shared__ double rvec[M], tot[M + 1];
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), col = blockIdx.x / kBC, tid = threadIdx.x;
    const int t = rank * kBW + tid;
    const int n0 = t * chunk, cnt = max(0, min(n0 + chunk, nt) - n0);
    double *X = sm + tid, *P = X + (long long)chunk * kBW, *Sv = P + (long long)chunk * kBW;
    const double2 *z = Z + t;
    const double gamma = gamma_p[0];
    // partial sums of the values v over the ranges into table b of every CTA (lane i: value i), the
    // barrier, and the totals into tot
    auto exchange = [&](int b, const auto &v) {
        constexpr int NV = (int)(sizeof(v) / sizeof(double));
        double mine = 0.0;
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const double ws = __shfl_sync(0xffffffffu, warp_sum(v[i]), 0);
            if ((tid & 31) == i) mine = ws;
        }
        if ((tid & 31) < NV)
            for (int r = 0; r < kBC; ++r) *cl.map_shared_rank(&tab[b][tid & 31][t >> 5], r) = mine;
        cl.sync();
        if (tid < NV) {
            double s = 0.0;
            for (int w = 0; w < NWT; ++w) s += tab[b][tid][w];
            tot[tid] = s;
        }
        __syncthreads();
    };
    if (tid < M) rvec[tid] = (tid == col) ? 1.0 : 0.0;
    cl.sync();                            // every CTA runs before any writes to its tables
    // s = B^T r - gamma x with x = 0, p = s
    double gl[1] = {0.0};
    for (int m = 0; m < cnt; ++m) {
        double s = 0.0;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const double2 zz = z[((long long)m * NF + f) * kBT];
            s = add_dot2(s, zz, rvec[f], rvec[NF + f]);
        }
        Sv[m * kBW] = s; P[m * kBW] = s; X[m * kBW] = 0.0;
        gl[0] = fma(s, s, gl[0]);
    }
    exchange(1, gl);
    double gam = tot[0];
    const double g0 = gam;
    int it = 0;
    for (; it < max_iter; ++it) {
        if (!(sqrt(gam) > tol * sqrt(g0))) break;
        // q = B p, pp = ||p||^2
        double ql[M + 1];
#pragma unroll
        for (int i = 0; i <= M; ++i) ql[i] = 0.0;
#pragma unroll U
        for (int m = 0; m < cnt; ++m) {
            const double pn = P[m * kBW];
            ql[M] = fma(pn, pn, ql[M]);
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const double2 zz = z[((long long)m * NF + f) * kBT];
                ql[f] = fma(zz.x, pn, ql[f]);
                ql[NF + f] = fma(zz.y, pn, ql[NF + f]);
            }
        }
        exchange(0, ql);
        double q[M], qq = 0.0;
#pragma unroll
        for (int i = 0; i < M; ++i) { q[i] = tot[i]; qq = fma(q[i], q[i], qq); }
        const double alpha = gam / fma(gamma, tot[M], qq);
        double rv[M];
#pragma unroll
        for (int i = 0; i < M; ++i) rv[i] = fma(-alpha, q[i], rvec[i]);
        __syncthreads();                  // every thread has read rvec and tot
        if (tid < M) {
#pragma unroll
            for (int i = 0; i < M; ++i)
                if (i == tid) rvec[i] = rv[i];
        }
        // x += alpha p; s = B^T r - gamma x; ||s||^2
        gl[0] = 0.0;
#pragma unroll U
        for (int m = 0; m < cnt; ++m) {
            const double x = fma(alpha, P[m * kBW], X[m * kBW]);
            X[m * kBW] = x;
            double s = __dmul_rn(-gamma, x);
#pragma unroll
            for (int f = 0; f < NF; ++f) {
                const double2 zz = z[((long long)m * NF + f) * kBT];
                s = add_dot2(s, zz, rv[f], rv[NF + f]);
            }
            Sv[m * kBW] = s;
            gl[0] = fma(s, s, gl[0]);
        }
        exchange(1, gl);              // (its barrier also orders rvec)
        const double gnew = tot[0];       // (read before the next exchange's barrier lets tot change)
        const double beta = gnew / gam;
        gam = gnew;
        for (int m = 0; m < cnt; ++m) P[m * kBW] = fma(beta, P[m * kBW], Sv[m * kBW]);
    }
    if (t == 0) iters[col] = it;
    double ql[M];
#pragma unroll
    for (int i = 0; i < M; ++i) ql[i] = 0.0;
    for (int m = 0; m < cnt; ++m) {
        const double x = X[m * kBW];
        basis[(long long)(n0 + m) * M + col] = x;
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            const double2 zz = z[((long long)m * NF + f) * kBT];
            ql[f] = fma(zz.x, x, ql[f]);
            ql[NF + f] = fma(zz.y, x, ql[NF + f]);
        }
    }
    exchange(0, ql);                   // also: no CTA ends while another may still write to it
    double worst = 0.0;
    for (int i = 0; i < M; ++i) worst = fmax(worst, fabs(tot[i] - (i == col ? 1.0 : 0.0)));
    if (t == 0) fit[col] = worst;
}

// The same for ranges too long for shared memory (more than 65 536 steps): one block per column, the CG
// vectors P and Sv in [2nf][nt] scratch rows, x in the basis, the phasors advanced in every pass.
__global__ void __launch_bounds__(kBT) k_basis_cgnr(BasisArgs b, const double *gamma_p, int max_iter, double tol,
                                                   double *basis, double *scratch, int *iters) {
    __shared__ double red[kBT / 32];
    __shared__ double rvec[2 * kMaxFreq], qvec[2 * kMaxFreq];
    const int m = 2 * b.nf, col = blockIdx.x;
    const double gamma = gamma_p[0];
    double *P = scratch + (long long)col * 2 * b.nt;
    double *Sv = P + b.nt;
    const int chunk = (b.nt + kBT - 1) / kBT;
    const int n0 = threadIdx.x * chunk, n1 = min(n0 + chunk, b.nt);
    if (threadIdx.x < m) rvec[threadIdx.x] = (threadIdx.x == col) ? 1.0 : 0.0;
    __syncthreads();

    // s = B^T r - gamma x with x = 0, p = s
    double gl = 0.0;
    double zr[kMaxFreq], zi[kMaxFreq], qr[kMaxFreq], qi[kMaxFreq];
    if (n0 < n1) {
        for (int f = 0; f < b.nf; ++f) phasor_start(b, f, n0, zr[f], zi[f], qr[f], qi[f]);
        for (int n = n0; n < n1; ++n) {
            double s = 0.0;
            for (int f = 0; f < b.nf; ++f) {
                s += zr[f] * rvec[f] + zi[f] * rvec[b.nf + f];
                double t = zr[f] * qr[f] - zi[f] * qi[f]; zi[f] = zr[f] * qi[f] + zi[f] * qr[f]; zr[f] = t;
            }
            Sv[n] = s; P[n] = s;
            basis[(long long)n * m + col] = 0.0;
            gl += s * s;
        }
    }
    double gam = block_sum(gl, red);
    const double g0 = gam;
    int it = 0;
    for (; it < max_iter; ++it) {
        if (!(sqrt(gam) > tol * sqrt(g0))) break;
        // q = B p, pp = ||p||^2
        double ql[2 * kMaxFreq];
        for (int i = 0; i < m; ++i) ql[i] = 0.0;
        double pp = 0.0;
        if (n0 < n1) {
            for (int f = 0; f < b.nf; ++f) phasor_start(b, f, n0, zr[f], zi[f], qr[f], qi[f]);
            for (int n = n0; n < n1; ++n) {
                const double pn = P[n];
                pp += pn * pn;
                for (int f = 0; f < b.nf; ++f) {
                    ql[f] += zr[f] * pn;
                    ql[b.nf + f] += zi[f] * pn;
                    double t = zr[f] * qr[f] - zi[f] * qi[f]; zi[f] = zr[f] * qi[f] + zi[f] * qr[f]; zr[f] = t;
                }
            }
        }
        for (int i = 0; i < m; ++i) {
            const double v = block_sum(ql[i], red);
            if (threadIdx.x == 0) qvec[i] = v;
        }
        pp = block_sum(pp, red);
        __syncthreads();
        double qq = 0.0;
        for (int i = 0; i < m; ++i) qq += qvec[i] * qvec[i];
        const double alpha = gam / (qq + gamma * pp);
        __syncthreads();
        if (threadIdx.x < m) rvec[threadIdx.x] -= alpha * qvec[threadIdx.x];
        __syncthreads();
        // x += alpha p; s = B^T r - gamma x; ||s||^2
        gl = 0.0;
        if (n0 < n1) {
            for (int f = 0; f < b.nf; ++f) phasor_start(b, f, n0, zr[f], zi[f], qr[f], qi[f]);
            for (int n = n0; n < n1; ++n) {
                double x = basis[(long long)n * m + col] + alpha * P[n];
                basis[(long long)n * m + col] = x;
                double s = -gamma * x;
                for (int f = 0; f < b.nf; ++f) {
                    s += zr[f] * rvec[f] + zi[f] * rvec[b.nf + f];
                    double t = zr[f] * qr[f] - zi[f] * qi[f]; zi[f] = zr[f] * qi[f] + zi[f] * qr[f]; zr[f] = t;
                }
                Sv[n] = s;
                gl += s * s;
            }
        }
        const double gnew = block_sum(gl, red);
        const double beta = gnew / gam;
        gam = gnew;
        for (int n = n0; n < n1; ++n) P[n] = Sv[n] + beta * P[n];
        __syncthreads();
    }
    if (threadIdx.x == 0) iters[col] = it;
}

// fit: max_i |(B B+)_{i,col} - delta_{i,col}|, one block per column
__global__ void __launch_bounds__(kBT) k_basis_fit(BasisArgs b, const double *basis, double *fit) {
    __shared__ double red[kBT / 32];
    const int m = 2 * b.nf, col = blockIdx.x;
    const int chunk = (b.nt + kBT - 1) / kBT;
    const int n0 = threadIdx.x * chunk, n1 = min(n0 + chunk, b.nt);
    double ql[2 * kMaxFreq];
    for (int i = 0; i < m; ++i) ql[i] = 0.0;
    if (n0 < n1) {
        double zr[kMaxFreq], zi[kMaxFreq], qr[kMaxFreq], qi[kMaxFreq];
        for (int f = 0; f < b.nf; ++f) phasor_start(b, f, n0, zr[f], zi[f], qr[f], qi[f]);
        for (int n = n0; n < n1; ++n) {
            const double x = basis[(long long)n * m + col];
            for (int f = 0; f < b.nf; ++f) {
                ql[f] += zr[f] * x;
                ql[b.nf + f] += zi[f] * x;
                double t = zr[f] * qr[f] - zi[f] * qi[f]; zi[f] = zr[f] * qi[f] + zi[f] * qr[f]; zr[f] = t;
            }
        }
    }
    double worst = 0.0;
    for (int i = 0; i < m; ++i) {
        const double v = block_sum(ql[i], red);
        worst = fmax(worst, fabs(v - (i == col ? 1.0 : 0.0)));
    }
    if (threadIdx.x == 0) fit[col] = worst;
}

namespace {
int basis_chunk(int nt) { return (nt + kBT - 1) / kBT; }
template <int NF>
cudaError_t cg_go(int nt, const double2 *Z, const double *gamma_p, int max_iter, double tol, double *basis, int *iters,
                  double *fit, cudaStream_t st) {
    const int chunk = basis_chunk(nt);
    const size_t smem = 3 * (size_t)chunk * kBW * sizeof(double);
    cudaError_t e = cudaFuncSetAttribute(k_basis_cg<NF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)(3 * (size_t)kBMaxChunk * kBW * sizeof(double)));
    if (e != cudaSuccess) return e;
    k_basis_cg<NF><<<2 * NF * kBC, kBW, smem, st>>>(nt, chunk, Z, gamma_p, max_iter, tol, basis, iters, fit);
    return cudaGetLastError();
}
}  // namespace

size_t basis_scratch_doubles(int nt, int nf) {
    const size_t table = (size_t)basis_chunk(nt) * kBT * nf * 2;
    return basis_chunk(nt) <= kBMaxChunk ? table : table + 4 * (size_t)nf * nt;
}

cudaError_t launch_basis(double dt, int nt, const double *a, int nf, double gamma, int gamma_rel, int max_iter,
                         double tol, double *basis, double *scratch, double *gram, double *out_scalars,
                         int *out_iters, cudaStream_t st) {
    BasisArgs b;
    b.dt = dt; b.nt = nt; b.nf = nf;
    for (int f = 0; f < kMaxFreq; ++f) b.a[f] = (f < nf) ? a[f] : 0.0;
    const int m = 2 * nf, chunk = basis_chunk(nt);
    double2 *Z = reinterpret_cast<double2 *>(scratch);
    k_basis_table<<<dim3(kBT / 64, nf), 64, 0, st>>>(b, chunk, Z);
    k_basis_gram<<<dim3(m, m), kBT, 0, st>>>(nt, nf, chunk, Z, gram);
    k_basis_gamma<<<1, 32, 0, st>>>(gram, m, gamma, gamma_rel, out_scalars);
    g_launches += 4;
    if (chunk > kBMaxChunk) {
        double *vec = scratch + (size_t)chunk * kBT * nf * 2;
        k_basis_cgnr<<<m, kBT, 0, st>>>(b, out_scalars, max_iter, tol, basis, vec, out_iters);
        k_basis_fit<<<m, kBT, 0, st>>>(b, basis, out_scalars + 1);
        g_launches++;
        return cudaGetLastError();
    }
    double *fit = out_scalars + 1;
    switch (nf) {
        case 1: return cg_go<1>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 2: return cg_go<2>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 3: return cg_go<3>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 4: return cg_go<4>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 5: return cg_go<5>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 6: return cg_go<6>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 7: return cg_go<7>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        case 8: return cg_go<8>(nt, Z, out_scalars, max_iter, tol, basis, out_iters, fit, st);
        default: return cudaErrorInvalidValue;
    }
}

// colmap[pos[u]] = val[u]: sets the column map of the injection taps
__global__ void k_scatter_int2(int2 *dst, const long long *pos, const int2 *val, int n) {
    const int u = blockIdx.x * blockDim.x + threadIdx.x;
    if (u < n) dst[pos[u]] = val[u];
}

cudaError_t launch_scatter_int2(int2 *dst, const long long *pos, const int2 *val, int n, cudaStream_t st) {
    if (n <= 0) return cudaSuccess;
    k_scatter_int2<<<(n + 255) / 256, 256, 0, st>>>(dst, pos, val, n);
    g_launches++;
    return cudaGetLastError();
}

template cudaError_t launch_coef_init<float>(const GeoD &, const float *, const float *, float *, float *, bool *,
                                             double, int *, cudaStream_t);
template cudaError_t launch_coef_init<double>(const GeoD &, const double *, const double *, double *, double *, bool *,
                                              double, int *, cudaStream_t);
template cudaError_t launch_finalize_volume<float>(float2 *, const float2 *, long long, int, int, const double2 *,
                                                   cudaStream_t);
template cudaError_t launch_finalize_volume<double>(double2 *, const double2 *, long long, int, int,
                                                    const double2 *, cudaStream_t);
template cudaError_t launch_gradient<float>(const GeoD &, const float *, const float2 *, const float2 *, int, int,
                                            int, bool, float *, float *, cudaStream_t);
template cudaError_t launch_gradient<double>(const GeoD &, const double *, const double2 *, const double2 *, int,
                                             int, int, bool, double *, double *, cudaStream_t);
template cudaError_t launch_grad_cells<float>(const GeoD &, const float *, const float *, int, bool, float *,
                                              cudaStream_t);
template cudaError_t launch_grad_cells<double>(const GeoD &, const double *, const double *, int, bool, double *,
                                               cudaStream_t);

}  // namespace csem
