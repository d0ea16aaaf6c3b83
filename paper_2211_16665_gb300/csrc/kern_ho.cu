// Fourth-order staggered H and E steps on the non-uniform grid (Sec. 2,
// Eq. 4 with the high-order differences of the paper's engine; the weights are
// described in csem_ho.cuh).  One thread per (i, j) column and KZ planes, the
// four-point neighbours read through the read-only cache; the CPML memory is
// touched only inside its slabs.  E lives in the same ring of snapshots as in
// the second-order kernels (E^{n+1} is written to slot n+1 from slot n), and the
// E kernel applies the source injection of its column's taps.
#include <algorithm>

#include "csem_ho.cuh"

namespace csem {

namespace {

constexpr int kHoX = 32, kHoY = 8, kHoZ = 4;

template <typename R> __device__ __forceinline__ R ld(const R *p) { return __ldg(p); }

// The roundings are spelled out: left to itself the compiler fuses one product or the other of a sum of two, and
// another one with every change of a kernel; gradients multiply such a difference by up to 10^4.  The choices are
// those of the kernels as first compiled from plain expressions, so results are what they were.
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
// a b + c d: a b fused to the rounded c d
template <typename R> __device__ __forceinline__ R dot2(R a, R b, R c, R d) { return fma_rn(a, b, mul_rn(c, d)); }


// d/da at the half node pos (of n) of a node-located field F, F[at] at node pos
template <typename R>
__device__ __forceinline__ R d_half(const R *__restrict__ F, long long at, long long s, int pos, int n,
                                    const R *__restrict__ w) {
    const R *wr = w + 4 * pos;
    R d = dot2(ld(wr + 1), ld(F + at), ld(wr + 2), ld(F + at + s));
    if (pos >= 1 && pos <= n - 2) d = fma_rn(ld(wr + 3), ld(F + at + 2 * s), fma_rn(ld(wr), ld(F + at - s), d));
    return d;
}

// d/da at the node pos (of n) of a half-node-located field F, F[at] at half node pos
template <typename R>
__device__ __forceinline__ R d_node(const R *F, long long at, long long s, int pos, int n,
                                    const R *__restrict__ w) {
    const R *wr = w + 4 * pos;
    R d = dot2(ld(wr + 1), F[at - s], ld(wr + 2), F[at]);
    if (pos >= 2 && pos <= n - 2) d = fma_rn(ld(wr + 3), F[at + s], fma_rn(ld(wr), F[at - 2 * s], d));
    return d;
}

// psi <- b psi + a d inside the slab, d + psi returned; q: psi, loaded with the others of the plane (see pml2)
template <typename R>
__device__ __forceinline__ R pml(R d, bool in, R b, R a, R q, R *ps) {
    if (!in) return d;
    const R v = dot2(a, d, b, q);
    *ps = v;
    return add_rn(d, v);
}

template <typename R>
__global__ void __launch_bounds__(kHoX *kHoY) k_h_ho(const StepParams<R> p, const HoTab<R> w, const int jstep) {
    const int i = blockIdx.x * kHoX + threadIdx.x;
    const int j = blockIdx.y * kHoY + threadIdx.y;
    const int nzb = (p.NZ + kHoZ - 1) / kHoZ;
    const int s = blockIdx.z / nzb, k0 = (blockIdx.z % nzb) * kHoZ;
    if (i >= p.NX || j >= p.NY) return;
    pdl_wait();
    const int n = *p.step + jstep;
    const long long vol = p.vol, plane = p.plane, pitch = p.pitch;
    const R *__restrict__ Ex = p.ering + (long long)s * p.ering_stride + (long long)(n % p.nslot) * 3 * vol;
    const R *__restrict__ Ey = Ex + vol;
    const R *__restrict__ Ez = Ex + 2 * vol;
    R *__restrict__ Hx = p.H + (long long)s * 3 * vol;
    R *__restrict__ Hy = Hx + vol;
    R *__restrict__ Hz = Hx + 2 * vol;
    R *__restrict__ P = p.psi + (long long)s * p.psi_stride;
    const int nx = p.nx, ny = p.ny, nz = p.nz, npml = p.npml;
    const R cH = p.cH;
    const bool xin = slab_half(i, nx, npml) >= 0, yin = slab_half(j, ny, npml) >= 0;
    const R bx = xin ? ld(p.ax.b_h + i) : R(0), ax_ = xin ? ld(p.ax.a_h + i) : R(0);
    const R by = yin ? ld(p.ay.b_h + j) : R(0), ay_ = yin ? ld(p.ay.a_h + j) : R(0);
    for (int k = k0; k < k0 + kHoZ && k < p.NZ; ++k) {
        const long long idx = (long long)k * plane + (long long)j * pitch + i;
        const bool zin = slab_half(k, nz, npml) >= 0;
        const R bz = zin ? ld(p.az.b_h + k) : R(0), az_ = zin ? ld(p.az.a_h + k) : R(0);
        R q0 = 0, q1 = 0, q2 = 0, q3 = 0, q4 = 0, q5 = 0;
        if (yin) { q0 = P[idx]; q5 = P[5 * vol + idx]; }
        if (zin) { q1 = P[1 * vol + idx]; q2 = P[2 * vol + idx]; }
        if (xin) { q3 = P[3 * vol + idx]; q4 = P[4 * vol + idx]; }
        if (j < ny && k < nz) {            // Hx at (i, j+1/2, k+1/2)
            const R a = pml(d_half(Ez, idx, pitch, j, ny, w.wyh), yin, by, ay_, q0, P + idx);
            const R b = pml(d_half(Ey, idx, plane, k, nz, w.wzh), zin, bz, az_, q1, P + vol + idx);
            Hx[idx] = fma_rn(-cH, add_rn(a, -b), Hx[idx]);
        }
        if (i < nx && k < nz) {            // Hy at (i+1/2, j, k+1/2)
            const R a = pml(d_half(Ex, idx, plane, k, nz, w.wzh), zin, bz, az_, q2, P + 2 * vol + idx);
            const R b = pml(d_half(Ez, idx, 1LL, i, nx, w.wxh), xin, bx, ax_, q3, P + 3 * vol + idx);
            Hy[idx] = fma_rn(-cH, add_rn(a, -b), Hy[idx]);
        }
        if (i < nx && j < ny) {            // Hz at (i+1/2, j+1/2, k)
            const R a = pml(d_half(Ey, idx, 1LL, i, nx, w.wxh), xin, bx, ax_, q4, P + 4 * vol + idx);
            const R b = pml(d_half(Ex, idx, pitch, j, ny, w.wyh), yin, by, ay_, q5, P + 5 * vol + idx);
            Hz[idx] = fma_rn(-cH, add_rn(a, -b), Hz[idx]);
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(kHoX *kHoY) k_e_ho(const StepParams<R> p, const HoTab<R> w, const int jstep) {
    const int i = blockIdx.x * kHoX + threadIdx.x;
    const int j = blockIdx.y * kHoY + threadIdx.y;
    const int nzb = (p.NZ + kHoZ - 1) / kHoZ;
    const int s = blockIdx.z / nzb, k0 = (blockIdx.z % nzb) * kHoZ;
    if (i >= p.NX || j >= p.NY) return;
    pdl_wait();
    const int n = *p.step + jstep;
    const long long vol = p.vol, plane = p.plane, pitch = p.pitch;
    const R *__restrict__ Eo = p.ering + (long long)s * p.ering_stride + (long long)(n % p.nslot) * 3 * vol;
    R *__restrict__ En = p.ering + (long long)s * p.ering_stride + (long long)((n + 1) % p.nslot) * 3 * vol;
    const R *Hx = p.H + (long long)s * 3 * vol;        // plain loads: see pdl_wait
    const R *Hy = Hx + vol;
    const R *Hz = Hx + 2 * vol;
    R *__restrict__ P = p.psi + (long long)s * p.psi_stride;
    const int nx = p.nx, ny = p.ny, nz = p.nz, npml = p.npml;
    const bool xin = slab_node(i, nx, npml) >= 0, yin = slab_node(j, ny, npml) >= 0;
    const R bx = xin ? ld(p.ax.b_n + i) : R(0), ax_ = xin ? ld(p.ax.a_n + i) : R(0);
    const R by = yin ? ld(p.ay.b_n + j) : R(0), ay_ = yin ? ld(p.ay.a_n + j) : R(0);
    const bool ix = (i >= 1 && i < nx), jy = (j >= 1 && j < ny);
    for (int k = k0; k < k0 + kHoZ && k < p.NZ; ++k) {
        const long long idx = (long long)k * plane + (long long)j * pitch + i;
        const bool zin = slab_node(k, nz, npml) >= 0;
        const R bz = zin ? ld(p.az.b_n + k) : R(0), az_ = zin ? ld(p.az.a_n + k) : R(0);
        const bool kz = (k >= 1 && k < nz);
        R q0 = 0, q1 = 0, q2 = 0, q3 = 0, q4 = 0, q5 = 0;
        if (yin) { q0 = P[6 * vol + idx]; q5 = P[11 * vol + idx]; }
        if (zin) { q1 = P[7 * vol + idx]; q2 = P[8 * vol + idx]; }
        if (xin) { q3 = P[9 * vol + idx]; q4 = P[10 * vol + idx]; }
        if (i < nx && jy && kz) {          // Ex at (i+1/2, j, k)
            const R a = pml(d_node(Hz, idx, pitch, j, ny, w.wyn), yin, by, ay_, q0, P + 6 * vol + idx);
            const R b = pml(d_node(Hy, idx, plane, k, nz, w.wzn), zin, bz, az_, q1, P + 7 * vol + idx);
            En[idx] = fma_rn(ld(p.cE + idx), add_rn(a, -b), ld(Eo + idx));
        }
        if (j < ny && ix && kz) {          // Ey at (i, j+1/2, k)
            const R a = pml(d_node(Hx, idx, plane, k, nz, w.wzn), zin, bz, az_, q2, P + 8 * vol + idx);
            const R b = pml(d_node(Hz, idx, 1LL, i, nx, w.wxn), xin, bx, ax_, q3, P + 9 * vol + idx);
            En[vol + idx] = fma_rn(ld(p.cE + vol + idx), add_rn(a, -b), ld(Eo + vol + idx));
        }
        if (k < nz && ix && jy) {          // Ez at (i, j, k+1/2)
            const R a = pml(d_node(Hy, idx, 1LL, i, nx, w.wxn), xin, bx, ax_, q4, P + 10 * vol + idx);
            const R b = pml(d_node(Hx, idx, pitch, j, ny, w.wyn), yin, by, ay_, q5, P + 11 * vol + idx);
            En[2 * vol + idx] = fma_rn(ld(p.cE + 2 * vol + idx), add_rn(a, -b), ld(Eo + 2 * vol + idx));
        }
    }
    // source term E^{n+1} -= dt/eps J'^{n+1/2} for the taps of this column and planes
    if (p.colmap) {
        const int2 cm = p.colmap[s * p.colmap_stride + (long long)j * pitch + i];
        for (int u = cm.x; u < cm.x + cm.y; ++u) {
            const Tap tp = p.itaps[(long long)s * p.itap_stride + u];
            const int k = (int)(tp.idx / plane);
            if (k < k0 || k >= k0 + kHoZ) continue;
            const double *cf = p.coef + ((long long)s * p.n_emit + tp.emit) * p.J;
            const double *T = p.T + (long long)n * p.J;
            double amp = 0.0;
            for (int jj = 0; jj < p.J; ++jj) amp += cf[jj] * T[jj];
            const long long o = (long long)tp.comp * vol + tp.idx;
            const double add = -(double)p.cE[o] * tp.w * amp;
            if (add != 0.0) En[o] += (R)add;
        }
    }
}

// ---------------------------------------------------------------------------
// Lean FP32 fourth-order kernels: two consecutive cells (i, i+1) of one (j, k) row
// per thread (8-byte accesses), 32 x 4-thread blocks with a register budget, KZ
// planes per thread marched along z with the four planes of the z derivatives in
// a register window (one new plane loaded per step), the x and y neighbours of a
// plane loaded together, and no branches on the boundary rows: their two-point
// weights have zero outer entries and the neighbours they would read outside the
// lattice are clamped to the cell itself.  E is advanced with dt/eps zeroed on the
// PEC edges, so every component is written unconditionally.  The CPML memory
// (12 field-layout arrays per source) is touched only in its slabs; the source
// taps come from the per-chunk increments.  The work domain is the cell range
// [0,nx) x [0,ny) x [0,nz) (H outside it never changes).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 f2g(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
__device__ __forceinline__ float2 f2w(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ void f2s(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
// at a 32-bit byte offset from a base that is the same for the whole block (one add per access)
__device__ __forceinline__ const float *at(const float *b, unsigned o) {
    return reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o);
}
__device__ __forceinline__ float2 f2g(const float *b, unsigned o) { return f2g(at(b, o)); }
__device__ __forceinline__ float2 f2w(const float *b, unsigned o) { return f2w(at(b, o)); }
// E^n in the E update, read once and by one thread: past L1, which keeps the rows of H that neighbours read again
// (512 steps of 128 x 128 x 96: 18.2 -> 17.3 ms)
__device__ __forceinline__ float2 f2e(const float *b, unsigned o) {
    float2 r;
    asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(r.x), "=f"(r.y) : "l"(at(b, o)));
    return r;
}
__device__ __forceinline__ float f1g(const float *b, unsigned o) { return __ldg(at(b, o)); }
__device__ __forceinline__ float f1w(const float *b, unsigned o) { return *at(b, o); }
__device__ __forceinline__ void f2s(float *b, unsigned o, float2 v) { f2s(const_cast<float *>(at(b, o)), v); }
__device__ __forceinline__ float4 f4g(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
// w . (a, b, c, d); SEC: the second product is fused to the rounded first one, else the first to the rounded second
template <bool SEC> __device__ __forceinline__ float dot4(const float4 &w, float a, float b, float c, float d) {
    const float p = SEC ? dot2(w.y, b, w.x, a) : dot2(w.x, a, w.y, b);
    return fma_rn(w.w, d, fma_rn(w.z, c, p));
}
// the same for both cells of the pair
template <bool SEC> __device__ __forceinline__ float2 dot4(const float4 &w, float2 a, float2 b, float2 c, float2 d) {
    return make_float2(dot4<SEC>(w, a.x, b.x, c.x, d.x), dot4<SEC>(w, a.y, b.y, c.y, d.y));
}
// x derivative of the pair from five consecutive values f0 .. f4 (cell i uses f0..f3, cell i+1 f1..f4)
template <bool SEC0, bool SEC1>
__device__ __forceinline__ float2 dx5(const float4 &w0, const float4 &w1, float f0, float f1, float f2, float f3,
                                      float f4) {
    return make_float2(dot4<SEC0>(w0, f0, f1, f2, f3), dot4<SEC1>(w1, f1, f2, f3, f4));
}
// h + c (u - v) for both cells
__device__ __forceinline__ float2 curl2(float2 h, float2 c, float2 u, float2 v) {
    return make_float2(fma_rn(c.x, add_rn(u.x, -v.x), h.x), fma_rn(c.y, add_rn(u.y, -v.y), h.y));
}
// d with its CPML memory v.  The six entries of a plane are loaded together (H: with the plane's fields; E: after
// its differences, which leaves the registers of the fields for them).  Loaded one by one, each after the store of
// the one before it (same array, so the compiler keeps their order), a thread on a slab waited for L2 up to six
// times per plane: 512 steps of 128 x 128 x 96, 25.6 -> 18.2 ms.
__device__ __forceinline__ void pml2(float2 &d, bool in, float b, float a, float2 v, float *ps, unsigned o) {
    if (!in) return;
    v.x = dot2(a, d.x, b, v.x); v.y = dot2(a, d.y, b, v.y);
    f2s(ps, o, v);
    d.x = add_rn(d.x, v.x); d.y = add_rn(d.y, v.y);
}
__device__ __forceinline__ void pml2x(float2 &d, bool in, float2 b, float2 a, float2 v, float *ps, unsigned o) {
    if (!in) return;
    v.x = dot2(a.x, d.x, b.x, v.x); v.y = dot2(a.y, d.y, b.y, v.y);
    f2s(ps, o, v);
    d.x = add_rn(d.x, v.x); d.y = add_rn(d.y, v.y);
}
__device__ __forceinline__ float3 ho_taps(const int *__restrict__ tk, const float *__restrict__ inc, int k, int2 cm) {
    float3 r = make_float3(0.f, 0.f, 0.f);
    for (int u = cm.x; u < cm.x + cm.y; ++u) {
        const int code = __ldg(tk + u);
        const float v = __ldg(inc + u);
        if ((code >> 2) != k) continue;
        if ((code & 3) == 0) r.x += v;
        else if ((code & 3) == 1) r.y += v;
        else r.z += v;
    }
    return r;
}

template <int KZ, int MINB>
__global__ void __launch_bounds__(128, MINB) k_h_ho4(const StepParams<float> p, const HoTab<float> w, const int jstep,
                                                     const unsigned S, const unsigned mS, const int nbig) {
    const int i = (blockIdx.x * 32 + threadIdx.x) * 2;
    const int j = blockIdx.y * 4 + threadIdx.y;
    const int zb = (int)div_by(blockIdx.z, mS), s = (int)(blockIdx.z - zb * S);
    const int k0 = zb < nbig ? zb * KZ : nbig * KZ + (zb - nbig), k1 = min(k0 + (zb < nbig ? KZ : 1), p.nz);   // big_blocks
    if (i >= p.nx || j >= p.ny) return;
    pdl_wait();
    const int sl = slot_of(p, *p.step + jstep);
    const int nx = p.nx, ny = p.ny, nz = p.nz, npml = p.npml;
    const long long vol = p.vol;
    const int plane = (int)p.plane, pitch = p.pitch;
    const float *__restrict__ Ex = p.ering + (long long)s * p.ering_stride + (long long)sl * 3 * p.vol;
    const float *__restrict__ Ey = Ex + vol;
    const float *__restrict__ Ez = Ex + 2 * vol;
    float *__restrict__ H = p.H + (long long)s * 3 * vol;
    float *__restrict__ P = p.psi + (long long)s * p.psi_stride;
    const float2 mc = make_float2(-p.cH, -p.cH);
    // neighbours, clamped on the lattice: column i-1; rows j-1, j+2 (column i+3 lies in the
    // lattice row or its padding, and only the last half node's zero weight meets it there)
    const unsigned im = (i > 0) ? -4 : 0;
    const unsigned jm = (j > 0) ? -4 * pitch : 0, jp = 4 * pitch, jp2 = (j + 2 <= ny) ? 8 * pitch : 4 * (ny - j) * pitch;
    const float4 wx0 = f4g(w.wxh + 4 * i), wx1 = f4g(w.wxh + 4 * (i + 1)), wy = f4g(w.wyh + 4 * j);
    const bool xs = slab_half(i, nx, npml) >= 0 || slab_half(i + 1, nx, npml) >= 0;
    const bool ys = slab_half(j, ny, npml) >= 0;
    const float2 bx = make_float2(__ldg(p.lx.b_h + i), __ldg(p.lx.b_h + i + 1));
    const float2 ax = make_float2(__ldg(p.lx.a_h + i), __ldg(p.lx.a_h + i + 1));
    const float by = __ldg(p.ly.b_h + j), ay = __ldg(p.ly.a_h + j);
    // z window of Ex, Ey at the thread's cells: planes k-1, k, k+1 (k+2 loaded per step)
    const unsigned base = 4u * (unsigned)(j * pitch + i), dz = 4u * (unsigned)plane;
    int km = (k0 > 0) ? k0 - 1 : 0;
    float2 xa = f2g(Ex, km * dz + base), xb = f2g(Ex, k0 * dz + base), xc = f2g(Ex, (k0 + 1) * dz + base);
    float2 ya = f2g(Ey, km * dz + base), yb = f2g(Ey, k0 * dz + base), yc = f2g(Ey, (k0 + 1) * dz + base);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
        const int k = k0 + kk;
        if (k >= k1) break;
        const unsigned o = k * dz + base;
        const int kp2 = (k + 2 <= nz) ? k + 2 : nz;
        const float2 xd = f2g(Ex, kp2 * dz + base), yd = f2g(Ey, kp2 * dz + base);
        const float4 wz = f4g(w.wzh + 4 * k);
        // x neighbours of Ey, Ez (plane k): values at i-1 .. i+3
        const float eym = f1g(Ey, o + im), ezm = f1g(Ez, o + im);
        const float2 ez01 = f2g(Ez, o), ey23 = f2g(Ey, o + 8), ez23 = f2g(Ez, o + 8);
        // y neighbours of Ex, Ez (plane k): rows j-1, j+1, j+2
        const float2 exm = f2g(Ex, o + jm), exp1 = f2g(Ex, o + jp), exp2 = f2g(Ex, o + jp2);
        const float2 ezm2 = f2g(Ez, o + jm), ezp1 = f2g(Ez, o + jp), ezp2 = f2g(Ez, o + jp2);
        float2 hx = f2w(H, o), hy = f2w(H + vol, o), hz = f2w(H + 2 * vol, o);
        const bool zs = slab_half(k, nz, npml) >= 0;
        float2 q0 = {}, q1 = {}, q2 = {}, q3 = {}, q4 = {}, q5 = {};
        if (ys) { q0 = f2w(P, o); q5 = f2w(P + 5 * vol, o); }
        if (zs) { q1 = f2w(P + vol, o); q2 = f2w(P + 2 * vol, o); }
        if (xs) { q3 = f2w(P + 3 * vol, o); q4 = f2w(P + 4 * vol, o); }
        float2 dEz_dy = dot4<true>(wy, ezm2, ez01, ezp1, ezp2), dEy_dz = dot4<false>(wz, ya, yb, yc, yd);
        float2 dEx_dz = dot4<false>(wz, xa, xb, xc, xd), dEz_dx = dx5<false, false>(wx0, wx1, ezm, ez01.x, ez01.y, ez23.x, ez23.y);
        float2 dEy_dx = dx5<true, false>(wx0, wx1, eym, yb.x, yb.y, ey23.x, ey23.y), dEx_dy = dot4<true>(wy, exm, xb, exp1, exp2);
        if (ys || zs || xs) {
            const float bz = __ldg(p.lz.b_h + k), az = __ldg(p.lz.a_h + k);
            pml2(dEz_dy, ys, by, ay, q0, P, o);
            pml2(dEy_dz, zs, bz, az, q1, P + vol, o);
            pml2(dEx_dz, zs, bz, az, q2, P + 2 * vol, o);
            pml2x(dEz_dx, xs, bx, ax, q3, P + 3 * vol, o);
            pml2x(dEy_dx, xs, bx, ax, q4, P + 4 * vol, o);
            pml2(dEx_dy, ys, by, ay, q5, P + 5 * vol, o);
        }
        hx = curl2(hx, mc, dEz_dy, dEy_dz);
        hy = curl2(hy, mc, dEx_dz, dEz_dx);
        hz = curl2(hz, mc, dEy_dx, dEx_dy);
        f2s(H, o, hx);
        f2s(H + vol, o, hy);
        f2s(H + 2 * vol, o, hz);
        xa = xb; xb = xc; xc = xd;
        ya = yb; yb = yc; yc = yd;
    }
}

template <int KZ, int MINB, bool FAR>
__global__ void __launch_bounds__(128, MINB) k_e_ho4(const StepParams<float> p, const HoTab<float> w, const int jstep,
                                                     const unsigned S, const unsigned mS, const int nbig) {
    const int i = (blockIdx.x * 32 + threadIdx.x) * 2;
    const int j = blockIdx.y * 4 + threadIdx.y;
    const int zb = (int)div_by(blockIdx.z, mS), s = (int)(blockIdx.z - zb * S);
    const int at = zb < nbig ? zb * KZ : nbig * KZ + (zb - nbig), len = zb < nbig ? KZ : 1;   // big_blocks
    const int k0 = FAR ? max(p.nz - at - len, 0) : at;       // downwards where FAR (kFarBytes)
    const int k1 = FAR ? p.nz - at : min(at + len, p.nz);
    if (i >= p.nx || j >= p.ny) return;
    pdl_wait();
    const int sl = slot_of(p, *p.step + jstep);
    const int nx = p.nx, ny = p.ny, nz = p.nz, npml = p.npml;
    const long long vol = p.vol;
    const int plane = (int)p.plane, pitch = p.pitch;
    const float *__restrict__ ring = p.ering + (long long)s * p.ering_stride;
    const float *__restrict__ Eo = ring + (long long)sl * 3 * p.vol;
    float *__restrict__ En = const_cast<float *>(ring) + (long long)slot_after(p, sl) * 3 * p.vol;
    const float *Hx = p.H + (long long)s * 3 * vol;        // plain loads: see pdl_wait
    const float *Hy = Hx + vol;
    const float *Hz = Hx + 2 * vol;
    float *__restrict__ P = p.psi + (long long)s * p.psi_stride + 6LL * vol;
    const float *__restrict__ cE = p.cEm;
    // neighbours, clamped on the lattice: columns i-2; rows j-2, j-1
    const unsigned im2 = (i >= 2) ? -8 : -4 * i;
    const unsigned jm2 = (j >= 2) ? -8 * pitch : -4 * j * pitch, jm1 = (j >= 1) ? -4 * pitch : 0, jp = 4 * pitch;
    const float4 wx0 = f4g(w.wxn + 4 * i), wx1 = f4g(w.wxn + 4 * (i + 1)), wy = f4g(w.wyn + 4 * j);
    const bool xs = slab_node(i, nx, npml) >= 0 || slab_node(i + 1, nx, npml) >= 0;
    const bool ys = slab_node(j, ny, npml) >= 0;
    const float2 bx = make_float2(__ldg(p.lx.b_n + i), __ldg(p.lx.b_n + i + 1));
    const float2 ax = make_float2(__ldg(p.lx.a_n + i), __ldg(p.lx.a_n + i + 1));
    const float by = __ldg(p.ly.b_n + j), ay = __ldg(p.ly.a_n + j);
    const bool taps = p.colmap && p.inc && p.tflag[s * p.tflag_stride + j * p.nseg + (i >> 5)];
    // z window of Hx, Hy at the thread's cells: planes k-2, k-1, k (k+1 loaded per step)
    const unsigned base = 4u * (unsigned)(j * pitch + i), dz = 4u * (unsigned)plane;
    const int ka = (k0 >= 2) ? k0 - 2 : 0, kb = (k0 >= 1) ? k0 - 1 : 0;
    float2 xa = f2w(Hx, ka * dz + base), xb = f2w(Hx, kb * dz + base), xc = f2w(Hx, k0 * dz + base);
    float2 ya = f2w(Hy, ka * dz + base), yb = f2w(Hy, kb * dz + base), yc = f2w(Hy, k0 * dz + base);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk) {
        const int k = k0 + kk;
        if (k >= k1) break;
        const unsigned o = k * dz + base;
        const float2 xd = f2w(Hx, o + dz), yd = f2w(Hy, o + dz);   // plane k+1 <= nz
        const float4 wz = f4g(w.wzn + 4 * k);
        // x neighbours of Hy, Hz (plane k): values at i-2 .. i+2
        const float2 hym = f2w(Hy, o + im2), hzm = f2w(Hz, o + im2);
        const float2 hz01 = f2w(Hz, o);
        const float hy2 = f1w(Hy, o + 8), hz2 = f1w(Hz, o + 8);
        // y neighbours of Hx, Hz (plane k): rows j-2, j-1, j+1
        const float2 hxm2 = f2w(Hx, o + jm2), hxm1 = f2w(Hx, o + jm1), hxp1 = f2w(Hx, o + jp);
        const float2 hzm2 = f2w(Hz, o + jm2), hzm1 = f2w(Hz, o + jm1), hzp1 = f2w(Hz, o + jp);
        const float2 e0 = f2e(Eo, o), e1 = f2e(Eo + vol, o), e2 = f2e(Eo + 2 * vol, o);
        const float2 c0 = f2g(cE, o), c1 = f2g(cE + vol, o), c2 = f2g(cE + 2 * vol, o);
        const bool zs = slab_node(k, nz, npml) >= 0;
        float2 dHz_dy = dot4<false>(wy, hzm2, hzm1, hz01, hzp1), dHy_dz = dot4<false>(wz, ya, yb, yc, yd);
        float2 dHx_dz = dot4<false>(wz, xa, xb, xc, xd);
        float2 dHz_dx = dx5<false, false>(wx0, wx1, hzm.x, hzm.y, hz01.x, hz01.y, hz2);
        float2 dHy_dx = dx5<false, true>(wx0, wx1, hym.x, hym.y, yc.x, yc.y, hy2);
        float2 dHx_dy = dot4<false>(wy, hxm2, hxm1, xc, hxp1);
        if (ys || zs || xs) {
            float2 q0 = {}, q1 = {}, q2 = {}, q3 = {}, q4 = {}, q5 = {};
            if (ys) { q0 = f2w(P, o); q5 = f2w(P + 5 * vol, o); }
            if (zs) { q1 = f2w(P + vol, o); q2 = f2w(P + 2 * vol, o); }
            if (xs) { q3 = f2w(P + 3 * vol, o); q4 = f2w(P + 4 * vol, o); }
            const float bz = __ldg(p.lz.b_n + k), az = __ldg(p.lz.a_n + k);
            pml2(dHz_dy, ys, by, ay, q0, P, o);
            pml2(dHy_dz, zs, bz, az, q1, P + vol, o);
            pml2(dHx_dz, zs, bz, az, q2, P + 2 * vol, o);
            pml2x(dHz_dx, xs, bx, ax, q3, P + 3 * vol, o);
            pml2x(dHy_dx, xs, bx, ax, q4, P + 4 * vol, o);
            pml2(dHx_dy, ys, by, ay, q5, P + 5 * vol, o);
        }
        float2 ex = curl2(e0, c0, dHz_dy, dHy_dz);
        float2 ey = curl2(e1, c1, dHx_dz, dHz_dx);
        float2 ez = curl2(e2, c2, dHy_dx, dHx_dy);
        if (taps) {
            const int2 *cm = p.colmap + (long long)s * p.colmap_stride + j * pitch + i;
            const int *tk = p.tapk + (long long)s * p.itap_stride;
            const float *inc = p.inc + ((long long)jstep * (int)S + s) * p.inc_ntl;
            const int2 cc0 = __ldg(cm), cc1 = __ldg(cm + 1);
            if (cc0.y) { const float3 a = ho_taps(tk, inc, k, cc0); ex.x += a.x; ey.x += a.y; ez.x += a.z; }
            if (cc1.y) { const float3 a = ho_taps(tk, inc, k, cc1); ex.y += a.x; ey.y += a.y; ez.y += a.z; }
        }
        f2s(En, o, ex);
        f2s(En + vol, o, ey);
        f2s(En + 2 * vol, o, ez);
        xa = xb; xb = xc; xc = xd;
        ya = yb; yb = yc; yc = yd;
    }
}

template <int KZ, int MB>
void go_ho4k(const StepParams<float> &p, const HoTab<float> &w, int S, int jstep, cudaStream_t st, bool h) {
    const int gx = (p.nx / 2 + 31) / 32, gy = (p.ny + 3) / 4, nzb = (p.nz + KZ - 1) / KZ;
    const int nbig = big_blocks(p.sms, nzb, KZ, gx * gy * S, MB);
    const dim3 grid(gx, gy, (nbig + std::max(p.nz - nbig * KZ, 0)) * S);
    const unsigned mS = div_magic((unsigned)S);
    if (h) launch_pdl(k_h_ho4<KZ, MB>, grid, dim3(32, 4), st, p, w, jstep, (unsigned)S, mS, nbig);
    else if (far_fields(p.vol, S)) launch_pdl(k_e_ho4<KZ, MB, true>, grid, dim3(32, 4), st, p, w, jstep, (unsigned)S, mS, nbig);
    else launch_pdl(k_e_ho4<KZ, MB, false>, grid, dim3(32, 4), st, p, w, jstep, (unsigned)S, mS, nbig);
}
template <int MB>
void go_ho4(const StepParams<float> &p, const HoTab<float> &w, int S, int jstep, cudaStream_t st, bool h, int kz) {
    if (kz == 2) go_ho4k<2, MB>(p, w, S, jstep, st, h);
    else if (kz == 4) go_ho4k<4, MB>(p, w, S, jstep, st, h);
    else go_ho4k<8, MB>(p, w, S, jstep, st, h);
}

}  // namespace

bool ho4_supported(int kz, int mb) { return (kz == 2 || kz == 4 || kz == 8) && (mb == 4 || mb == 6 || mb == 8); }

cudaError_t launch_ho4(const StepParams<float> &p, const HoTab<float> &w, int S, int jstep, cudaStream_t st, bool h,
                       int kz, int mb) {
    if (p.nx % 2 != 0 || !p.cEm || !p.lx.b_h || !ho4_supported(kz, mb)) return cudaErrorInvalidValue;
    if (mb == 4) go_ho4<4>(p, w, S, jstep, st, h, kz);
    else if (mb == 6) go_ho4<6>(p, w, S, jstep, st, h, kz);
    else go_ho4<8>(p, w, S, jstep, st, h, kz);
    g_launches++;
    return cudaGetLastError();
}

template <typename R>
cudaError_t launch_ho(const StepParams<R> &p, const HoTab<R> &w, int S, int jstep, cudaStream_t st, int which) {
    bool lean_h = false, lean_e = false;       // FP32: the lean kernels for the halves that select them
    if constexpr (sizeof(R) == 4) {
        lean_h = p.LEAN_h != 0;
        lean_e = p.LEAN_e != 0;
    }
    const dim3 blk(kHoX, kHoY);
    const dim3 grid((p.NX + kHoX - 1) / kHoX, (p.NY + kHoY - 1) / kHoY, S * ((p.NZ + kHoZ - 1) / kHoZ));
    cudaError_t e = cudaSuccess;
    if (which & 1) {                           // the H half first, then the E half
        if (lean_h) {
            if constexpr (sizeof(R) == 4) e = launch_ho4(p, w, S, jstep, st, true, p.KZ_h, p.MB_h);
        } else {
            launch_pdl(k_h_ho<R>, grid, blk, st, p, w, jstep);
            g_launches++;
        }
    }
    if (e == cudaSuccess && (which & 4)) {
        if (lean_e) {
            if constexpr (sizeof(R) == 4) e = launch_ho4(p, w, S, jstep, st, false, p.KZ_e, p.MB_e);
        } else {
            launch_pdl(k_e_ho<R>, grid, blk, st, p, w, jstep);
            g_launches++;
        }
    }
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

template cudaError_t launch_ho<float>(const StepParams<float> &, const HoTab<float> &, int, int, cudaStream_t, int);
template cudaError_t launch_ho<double>(const StepParams<double> &, const HoTab<double> &, int, int, cudaStream_t,
                                       int);

}  // namespace csem
