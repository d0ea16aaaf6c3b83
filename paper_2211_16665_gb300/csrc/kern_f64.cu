// FP64 H and E step kernels (second order; Sec. 2, Eq. 4 with the unsplit CPML).
//
// What bounds them is the FP64 pipe, which takes a warp's instruction for sixteen cycles whether all of
// its lanes work or not, so they spend as few FP64 instructions as the scheme allows:
//  * H adds each scaled difference with one FMA (table dt/(mu0 h)), and its CPML memory is kept scaled by
//    dt/mu0, so a component takes four operations off the slabs; E, whose dt/eps varies from edge to edge,
//    takes five.  The general kernels' six came from scaling, combining and adding one by one;
//  * a recursion step takes three more (table a/h: psi <- b psi + (a/h) difference);
//  * the threads of a plane take the cells of the x slabs first and the others after them, so a warp either
//    needs the x recursion in every lane or not at all (68 cells with 20 of them in the slabs put slab lanes
//    into every warp of a row-by-row order).  Rows and planes decide on the y and z slabs.
// The rest is latency: a plane's loads, its CPML memory among them, are issued together (after the stores of the
// plane's other slabs they came one L2 latency later each), and blocks have 128 threads, so that 4, 6 or 8 of them
// per SM leave the registers for that.
// 68^3, npml 10, 1500 steps with volumes: 89.0 ms with the general kernels (H 28.7 and E 26.6 us per launch, 64 % and
// 58 % of the FP64 pipe's issue slots), 58.3 ms with the fewer operations, 56.7 with the loads together, 53.2 with
// blocks of 128 too (55.3 with these alone).
#include "csem_internal.cuh"

namespace csem {

namespace {

constexpr int kB64 = 128;

// The cell (i, j) of thread t of a plane: the x slabs' cells (2 npml per row), padded to whole warps, then the others.
struct Cell { int i, j; };
__host__ __device__ inline int slab_threads(int ny, int npml) { return (2 * npml * ny + 31) / 32 * 32; }
__device__ __forceinline__ Cell cell_of(int t, int nx, int ny, int npml) {
    const int n1 = slab_threads(ny, npml);
    if (t < n1) {
        const int np2 = 2 * npml, j = t / np2, c = t - j * np2;
        return Cell{c < npml ? c : nx - np2 + c, j};
    }
    const int u = t - n1, ni = nx - 2 * npml, j = u / ni;
    return Cell{npml + u - j * ni, j};
}

}  // namespace

template <int KZ, int MINB>
__global__ void __launch_bounds__(kB64, MINB) k_h64(const StepParams<double> p, const int jstep) {
    const int nx = p.nx, ny = p.ny, nz = p.nz, npml = p.npml, np2 = 2 * npml;
    const Cell c = cell_of(blockIdx.x * kB64 + threadIdx.x, nx, ny, npml);
    const int i = c.i, j = c.j, s = blockIdx.z, k0 = blockIdx.y * KZ;
    if (j >= ny) return;
    const int vol = (int)p.vol, plane = (int)p.plane, pitch = p.pitch;
    const int sx = slab_half(i, nx, npml), sy = slab_half(j, ny, npml);
    const double cx = __ldg(p.ax.c_h + i), cy = __ldg(p.ay.c_h + j);
    double bx = 0, gx = 0, by = 0, gy = 0;
    if (sx >= 0) { bx = __ldg(p.ax.b_h + i); gx = __ldg(p.ax.g_h + i); }
    if (sy >= 0) { by = __ldg(p.ay.b_h + j); gy = __ldg(p.ay.g_h + j); }
    pdl_wait();
    const int n = *p.step + jstep;
    const double *__restrict__ Ex = p.ering + (long long)s * p.ering_stride + (long long)(n % p.nslot) * 3 * p.vol;
    const double *__restrict__ Ey = Ex + vol, *__restrict__ Ez = Ex + 2 * vol;
    double *H = p.H + (long long)s * 3 * vol;
    double *P = p.psi + (long long)s * p.psi_stride;
    double *psx = P, *psy = P + 6 * p.sx, *psz = P + 6 * p.sx + 6 * p.sy;
    int idx = k0 * plane + j * pitch + i;
    double exc = __ldg(Ex + idx), eyc = __ldg(Ey + idx);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk, idx += plane) {
        const int k = k0 + kk;
        if (k >= nz) break;
        const double ezc = __ldg(Ez + idx), exk = __ldg(Ex + idx + plane), eyk = __ldg(Ey + idx + plane);
        const double zy = __ldg(Ez + idx + pitch) - ezc, yz = eyk - eyc, xz = exk - exc;
        const double zx = __ldg(Ez + idx + 1) - ezc, yx = __ldg(Ey + idx + 1) - eyc, xy = __ldg(Ex + idx + pitch) - exc;
        const int sz = slab_half(k, nz, npml);
        const double cz = __ldg(p.az.c_h + k);
        double *qy = psy + (k * np2 + sy) * pitch + i, *qz = psz + (sz * p.NY + j) * pitch + i, *qx = psx + (k * p.NY + j) * np2 + sx;
        double y0 = 0, y1 = 0, z0 = 0, z1 = 0, x0 = 0, x1 = 0, bz = 0, gz = 0;
        if (sy >= 0) { y0 = qy[0]; y1 = qy[p.sy]; }
        if (sz >= 0) { z0 = qz[0]; z1 = qz[p.sz]; bz = __ldg(p.az.b_h + k); gz = __ldg(p.az.g_h + k); }
        if (sx >= 0) { x0 = qx[0]; x1 = qx[p.sx]; }
        double hx = fma(cz, yz, fma(-cy, zy, H[idx]));
        double hy = fma(cx, zx, fma(-cz, xz, H[vol + idx]));
        double hz = fma(cy, xy, fma(-cx, yx, H[2 * vol + idx]));
        if (sy >= 0) {
            const double a = fma(gy, zy, by * y0), b = fma(gy, xy, by * y1);
            qy[0] = a; qy[p.sy] = b;
            hx -= a; hz += b;
        }
        if (sz >= 0) {
            const double a = fma(gz, yz, bz * z0), b = fma(gz, xz, bz * z1);
            qz[0] = a; qz[p.sz] = b;
            hx += a; hy -= b;
        }
        if (sx >= 0) {
            const double a = fma(gx, zx, bx * x0), b = fma(gx, yx, bx * x1);
            qx[0] = a; qx[p.sx] = b;
            hy += a; hz -= b;
        }
        H[idx] = hx; H[vol + idx] = hy; H[2 * vol + idx] = hz;
        exc = exk;
        eyc = eyk;
    }
}

template <int KZ, int MINB>
__global__ void __launch_bounds__(kB64, MINB) k_e64(const StepParams<double> p, const int jstep) {
    const int nx = p.nx, ny = p.ny, nz = p.nz, npml = p.npml, np2 = 2 * npml;
    const Cell c = cell_of(blockIdx.x * kB64 + threadIdx.x, nx, ny, npml);
    const int i = c.i, j = c.j, s = blockIdx.z, k0 = blockIdx.y * KZ;
    if (j >= ny) return;
    const int vol = (int)p.vol, plane = (int)p.plane, pitch = p.pitch;
    const int sx = slab_node(i, nx, npml), sy = slab_node(j, ny, npml);
    const double ix = __ldg(p.ax.ih_n + i), iy = __ldg(p.ay.ih_n + j);
    double bx = 0, gx = 0, by = 0, gy = 0;
    if (sx >= 0) { bx = __ldg(p.ax.b_n + i); gx = __ldg(p.ax.g_n + i); }
    if (sy >= 0) { by = __ldg(p.ay.b_n + j); gy = __ldg(p.ay.g_n + j); }
    const bool xin = i >= 1, yin = j >= 1;
    const int im = xin ? 1 : 0, jm = yin ? pitch : 0;     // lower neighbours, clamped on the outer faces
    pdl_wait();
    const int n = *p.step + jstep;
    const double *__restrict__ Eo = p.ering + (long long)s * p.ering_stride + (long long)(n % p.nslot) * 3 * p.vol;
    double *En = p.ering + (long long)s * p.ering_stride + (long long)((n + 1) % p.nslot) * 3 * p.vol;
    const double *Hx = p.H + (long long)s * 3 * vol, *Hy = Hx + vol, *Hz = Hx + 2 * vol;   // plain loads: see pdl_wait
    double *P = p.psi + (long long)s * p.psi_stride;
    double *psx = P + 2 * p.sx, *psy = P + 6 * p.sx + 2 * p.sy, *psz = P + 6 * p.sx + 6 * p.sy + 2 * p.sz;
    int idx = k0 * plane + j * pitch + i;
    double hxm = (k0 > 0) ? Hx[idx - plane] : 0.0, hym = (k0 > 0) ? Hy[idx - plane] : 0.0;
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk, idx += plane) {
        const int k = k0 + kk;
        if (k >= nz) break;
        const double hxc = Hx[idx], hyc = Hy[idx], hzc = Hz[idx];
        const double zy = hzc - Hz[idx - jm], yz = hyc - hym, xz = hxc - hxm;
        const double zx = hzc - Hz[idx - im], yx = hyc - Hy[idx - im], xy = hxc - Hx[idx - jm];
        const int sz = slab_node(k, nz, npml);
        const double iz = __ldg(p.az.ih_n + k);
        double *qy = psy + (k * np2 + sy) * pitch + i, *qz = psz + (sz * p.NY + j) * pitch + i, *qx = psx + (k * p.NY + j) * np2 + sx;
        double y0 = 0, y1 = 0, z0 = 0, z1 = 0, x0 = 0, x1 = 0, bz = 0, gz = 0;
        if (sy >= 0) { y0 = qy[0]; y1 = qy[p.sy]; }
        if (sz >= 0) { z0 = qz[0]; z1 = qz[p.sz]; bz = __ldg(p.az.b_n + k); gz = __ldg(p.az.g_n + k); }
        if (sx >= 0) { x0 = qx[0]; x1 = qx[p.sx]; }
        const double e0 = __ldg(Eo + idx), e1 = __ldg(Eo + vol + idx), e2 = __ldg(Eo + 2 * vol + idx);
        const double c0 = __ldg(p.cE + idx), c1 = __ldg(p.cE + vol + idx), c2 = __ldg(p.cE + 2 * vol + idx);
        double tx = fma(-iz, yz, iy * zy), ty = fma(-ix, zx, iz * xz), tz = fma(-iy, xy, ix * yx);
        const bool zin = k >= 1;
        if (sy >= 0) {
            if (zin) { const double a = fma(gy, zy, by * y0); qy[0] = a; tx += a; }
            if (xin) { const double b = fma(gy, xy, by * y1); qy[p.sy] = b; tz -= b; }
        }
        if (sz >= 0) {
            if (yin) { const double a = fma(gz, yz, bz * z0); qz[0] = a; tx -= a; }
            if (xin) { const double b = fma(gz, xz, bz * z1); qz[p.sz] = b; ty += b; }
        }
        if (sx >= 0) {
            if (zin) { const double a = fma(gx, zx, bx * x0); qx[0] = a; ty -= a; }
            if (yin) { const double b = fma(gx, yx, bx * x1); qx[p.sx] = b; tz += b; }
        }
        // tangential E on the outer faces keeps its zero
        if (yin && zin) En[idx] = fma(c0, tx, e0);
        if (xin && zin) En[vol + idx] = fma(c1, ty, e1);
        if (xin && yin) En[2 * vol + idx] = fma(c2, tz, e2);
        hxm = hxc;
        hym = hyc;
    }
    // source term E^{n+1} -= dt/eps J'^{n+1/2}: this thread owns its column's taps
    if (p.colmap) {
        const int2 cm = p.colmap[s * p.colmap_stride + j * pitch + i];
        for (int u = cm.x; u < cm.x + cm.y; ++u) {
            const Tap tp = p.itaps[(long long)s * p.itap_stride + u];
            const int k = (int)(tp.idx / plane);
            if (k < k0 || k >= k0 + KZ) continue;
            const double *cf = p.coef + ((long long)s * p.n_emit + tp.emit) * p.J;
            const double *T = p.T + (long long)n * p.J;
            double amp = 0.0;
            for (int jj = 0; jj < p.J; ++jj) amp += cf[jj] * T[jj];
            const int o = tp.comp * vol + (int)tp.idx;
            const double add = -p.cE[o] * tp.w * amp;
            if (add != 0.0) En[o] += add;
        }
    }
}

namespace {
template <int KZ, int MB> void go64(const StepParams<double> &p, int S, int jstep, cudaStream_t st, bool h) {
    const int threads = slab_threads(p.ny, p.npml) + (p.nx - 2 * p.npml) * p.ny;
    const dim3 grid((unsigned)((threads + kB64 - 1) / kB64), (unsigned)((p.nz + KZ - 1) / KZ), (unsigned)S);
    if (h) launch_pdl(k_h64<KZ, MB>, grid, dim3(kB64), st, p, jstep);
    else launch_pdl(k_e64<KZ, MB>, grid, dim3(kB64), st, p, jstep);
}
template <int MB> bool kz64(const StepParams<double> &p, int S, int jstep, cudaStream_t st, bool h, int kz) {
    switch (kz) {
        case 1: go64<1, MB>(p, S, jstep, st, h); return true;
        case 2: go64<2, MB>(p, S, jstep, st, h); return true;
        case 4: go64<4, MB>(p, S, jstep, st, h); return true;
        case 8: go64<8, MB>(p, S, jstep, st, h); return true;
        default: return false;
    }
}
}  // namespace

cudaError_t launch_field64(const StepParams<double> &p, int S, int jstep, cudaStream_t st, bool h, int kz, int mb) {
    bool ok = false;
    if (mb == 4) ok = kz64<4>(p, S, jstep, st, h, kz);
    else if (mb == 6) ok = kz64<6>(p, S, jstep, st, h, kz);
    else if (mb == 8) ok = kz64<8>(p, S, jstep, st, h, kz);
    if (!ok) return cudaErrorInvalidValue;
    g_launches++;
    return cudaGetLastError();
}

}  // namespace csem
