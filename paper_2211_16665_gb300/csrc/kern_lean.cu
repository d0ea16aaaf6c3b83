// Lean FP32 H and E step kernels (Sec. 2, Eq. 4 with the unsplit CPML): W
// consecutive cells (W = 1 or 2; i a multiple of W) of one (j, k) row per
// thread, the cell range [0,nx) x [0,ny) x [0,nz), KZ planes along z per thread.
// With nx odd the last thread's second cell is the row's entry nx: its dt/eps and
// spacings are zero, so its values stay zero.  They compute what the scalar kernels compute,
// entry by entry, with every load of a plane independent of the others, so that
// a plane's loads are in flight together:
//  * the CPML memory lives in arrays of its own (12 per source: 0-5 for H, 6-11
//    for E).  The y- and z-slab arrays have the field layout.  The x-slab arrays
//    (3, 4, 9, 10) are compact: row (k, j) holds the cells i < lo and i >= hi (lo =
//    npml rounded up, hi = nx - npml rounded down to even), so the slab entries of
//    consecutive rows are contiguous;
//  * the coefficient tables are padded to whole 16-byte groups, and the CPML
//    coefficients are zero off the slabs and on the outer nodes.  A cell in the
//    rounded-out slab but not in the CPML keeps psi = 0;
//  * the x-slab recursion runs on every lane (lanes off the slab start from zero and
//    have zero coefficients) and only slab lanes load and store;
//  * a block whose plane is off the z slabs and whose rows are off the y slabs
//    takes a code path without the y/z recursion, with fewer live values;
//  * E is advanced with dt/eps set to zero on the PEC edges (tangential E on the
//    outer faces), so all three components are written unconditionally, the PEC
//    edges keep their zero, and the curl's lower neighbours are clamped to the
//    cell itself on the outer faces (what they give there is multiplied by 0);
//  * the source taps of the thread's columns are added to the new values in
//    registers before the store; the column map is read only where a per-row,
//    per-32-column flag marks a tap (a byte shared by a warp), inside that rare
//    branch, so it holds no registers elsewhere.
// W stays small so that a plane's loaded values fit the register budget.
// The block is 32 x 4 threads (32 W cells of 4 rows; 128 threads, so 4, 6 or 8
// resident blocks per SM give 128, 85 or 64 registers per thread); blockIdx.z
// runs over (z block, source) with the source fastest; the planes of the last, partial
// wave of blocks go to blocks of one plane (big_blocks).
// What bounds them: DRAM where the fields exceed L2 (two sources of 256 x 256 x 128 move
// their bytes at the rate of a copy, so only bytes count: see kFarBytes), L2 latency and
// the partial wave where they fit (128 x 128 x 96: 27 us a step, 24 with big_blocks and
// E^n past L1), and the launches themselves below about 10^5 cells.
#include "csem_internal.cuh"

// 0: everything but the instances for other rows than multiples of four; 1, 2: the H and the E instances for those
#ifndef CSEM_LEAN_UNIT
#define CSEM_LEAN_UNIT 0
#endif

namespace csem {

namespace {

constexpr int kLeanX = 32, kLeanRows = 4;
// rows of a multiple of four cells, and others with the roundings of the scalar or of the four-cell kernels (Rounding)
constexpr int kRowsFour = 0, kRowsScalar = 1, kRowsVec = 2;

template <int W> struct Vec { float v[W]; };
template <int W> __device__ __forceinline__ Vec<W> ldc(const float *p) {
    Vec<W> r;
    if constexpr (W == 1) r.v[0] = __ldg(p);
    else { const float2 t = __ldg(reinterpret_cast<const float2 *>(p)); r.v[0] = t.x; r.v[1] = t.y; }
    return r;
}
template <int W> __device__ __forceinline__ Vec<W> ldw(const float *p) {
    Vec<W> r;
    if constexpr (W == 1) r.v[0] = *p;
    else { const float2 t = *reinterpret_cast<const float2 *>(p); r.v[0] = t.x; r.v[1] = t.y; }
    return r;
}
template <int W> __device__ __forceinline__ void stv(float *p, const Vec<W> &a) {
    if constexpr (W == 1) *p = a.v[0];
    else *reinterpret_cast<float2 *>(p) = make_float2(a.v[0], a.v[1]);
}
// The same at a byte offset (32 bits, unsigned) from a base that is the same for the whole block: the base stays
// in uniform registers and an access costs one add for its offset, where a 64-bit index per access took three to
// four.  An offset reaches 4 GB, a component of 2^30 entries.
template <int W> __device__ __forceinline__ Vec<W> ldc(const float *b, unsigned o) {
    return ldc<W>(reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o));
}
template <int W> __device__ __forceinline__ Vec<W> ldw(const float *b, unsigned o) {
    return ldw<W>(reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o));
}
template <int W> __device__ __forceinline__ void stv(float *b, unsigned o, const Vec<W> &a) {
    stv<W>(reinterpret_cast<float *>(reinterpret_cast<char *>(b) + o), a);
}
// E^n in the E update, read once and by one thread: it passes L1 by, which leaves L1 to the rows of H that the
// neighbouring threads read again (128 x 128 x 96, 1024 steps with volumes: 27.2 -> 25.6 ms).
template <int W> __device__ __forceinline__ Vec<W> lde(const float *b, unsigned o) {
    const float *p = reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o);
    Vec<W> r;
    if constexpr (W == 1) asm("ld.global.nc.L1::no_allocate.f32 %0, [%1];" : "=f"(r.v[0]) : "l"(p));
    else asm("ld.global.nc.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(r.v[0]), "=f"(r.v[1]) : "l"(p));
    return r;
}
// A store that L2 keeps longest.
template <int W> __device__ __forceinline__ void stl(float *b, unsigned o, const Vec<W> &a) {
    float *p = reinterpret_cast<float *>(reinterpret_cast<char *>(b) + o);
    uint64_t keep;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
    if constexpr (W == 1) asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(p), "f"(a.v[0]), "l"(keep) : "memory");
    else asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;" ::"l"(p), "f"(a.v[0]), "f"(a.v[1]), "l"(keep) : "memory");
}
__device__ __forceinline__ float ldc1(const float *b, unsigned o) {
    return __ldg(reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o));
}
template <int W> __device__ __forceinline__ Vec<W> zv() {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = 0.f;
    return r;
}
// The roundings are spelled out.  Left to itself the compiler fuses one product or the other of a sum of two, by
// instance; a gradient multiplies such a difference by up to 10^4 (the adjoint basis is ill-conditioned), so it then
// changes with every new instance of a kernel.  Here every instance gives the same bits, whatever its cells and planes
// per thread, blocks per SM, order and size of its z blocks.  Which products are fused follows the kernels that were
// compiled from the plain expressions, so results are what they were: h_plane and e_plane say where, and Rounding
// (csem_internal.cuh) which of those kernels.
// a - b
template <int W> __device__ __forceinline__ Vec<W> dif(const Vec<W> &a, const Vec<W> &b) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = __fsub_rn(a.v[e], b.v[e]);
    return r;
}
// a s (shared or per-cell s)
template <int W> __device__ __forceinline__ Vec<W> mul(const Vec<W> &a, float s) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = __fmul_rn(a.v[e], s);
    return r;
}
template <int W> __device__ __forceinline__ Vec<W> mul(const Vec<W> &a, const Vec<W> &s) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = __fmul_rn(a.v[e], s.v[e]);
    return r;
}
// a s + c with one rounding
template <int W> __device__ __forceinline__ Vec<W> mad(const Vec<W> &a, float s, const Vec<W> &c) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = fmaf(a.v[e], s, c.v[e]);
    return r;
}
template <int W> __device__ __forceinline__ Vec<W> mad(const Vec<W> &a, const Vec<W> &s, const Vec<W> &c) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = fmaf(a.v[e], s.v[e], c.v[e]);
    return r;
}
template <int W> __device__ __forceinline__ Vec<W> neg(const Vec<W> &a) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e < W; ++e) r.v[e] = -a.v[e];
    return r;
}
// CPML recursion psi <- b psi + a d, then d += psi (shared or per-cell b, a).  bf: b psi is fused to the rounded a d,
// else a d to the rounded b psi.
__device__ __forceinline__ void cpml1(bool bf, float &ps, float &d, float b, float a) {
    ps = bf ? fmaf(b, ps, __fmul_rn(a, d)) : fmaf(a, d, __fmul_rn(b, ps));
    d = __fadd_rn(d, ps);
}
template <int W> __device__ __forceinline__ void cpml(bool bf, Vec<W> &ps, Vec<W> &d, float b, float a) {
#pragma unroll
    for (int e = 0; e < W; ++e) cpml1(bf, ps.v[e], d.v[e], b, a);
}
template <int W> __device__ __forceinline__ void cpml(bool bf, Vec<W> &ps, Vec<W> &d, const Vec<W> &b, const Vec<W> &a) {
#pragma unroll
    for (int e = 0; e < W; ++e) cpml1(bf, ps.v[e], d.v[e], b.v[e], a.v[e]);
}
// u s - v and v - u s, the product rounded first or (fuse) fused to v.  RT: fuse is known at run time only; u times one
// and then s fused, or u times s and then one fused, costs one multiplication where a select costs three instructions.
template <int W, bool RT> __device__ __forceinline__ Vec<W> mulsub(bool fuse, const Vec<W> &u, float s, const Vec<W> &v) {
    if constexpr (RT) return mad<W>(mul<W>(u, fuse ? 1.f : s), fuse ? s : 1.f, neg<W>(v));
    return fuse ? mad<W>(u, s, neg<W>(v)) : dif<W>(mul<W>(u, s), v);
}
template <int W, bool RT> __device__ __forceinline__ Vec<W> submul(bool fuse, const Vec<W> &v, const Vec<W> &u, float s) {
    if constexpr (RT) return mad<W>(mul<W>(u, fuse ? 1.f : s), fuse ? -s : -1.f, v);
    return fuse ? mad<W>(u, -s, v) : dif<W>(v, mul<W>(u, s));
}
// the W cells shifted by one: (prev, a0, .., a_{W-2}) and (a1, .., a_{W-1}, next)
template <int W> __device__ __forceinline__ Vec<W> down(float prev, const Vec<W> &a) {
    Vec<W> r;
    r.v[0] = prev;
#pragma unroll
    for (int e = 1; e < W; ++e) r.v[e] = a.v[e - 1];
    return r;
}
template <int W> __device__ __forceinline__ Vec<W> up(const Vec<W> &a, float next) {
    Vec<W> r;
#pragma unroll
    for (int e = 0; e + 1 < W; ++e) r.v[e] = a.v[e + 1];
    r.v[W - 1] = next;
    return r;
}

// Per-thread constants shared by the planes of a lean kernel.
template <int W> struct LeanRow {
    int i, j, nxs, ixs;                  // nxs: slab entries per row, ixs: the cells' place among them
    bool xs, ys;
    Vec<W> ihx, bx, ax;
    float ihy, by, ay;
    __device__ __forceinline__ unsigned xoff(const StepParams<float> &p, int k) const {   // bytes, plane k
        return 4u * (unsigned)((k * p.ny + j) * nxs + ixs);
    }
};
template <int W>
__device__ __forceinline__ void lean_row(const StepParams<float> &p, const AxisTab<float> &tx, const AxisTab<float> &ty,
                                         bool half, int i, int j, LeanRow<W> &r) {
    const int npml = p.npml;
    r.i = i; r.j = j;
    const int lo = (npml + 1) & ~1, hi = (p.nx - npml) & ~1;
    r.nxs = lo + ((p.nx + 1) & ~1) - hi;
    r.xs = npml > 0 && (i < lo || i >= hi);
    r.ixs = (i < lo) ? i : i - hi + lo;
    r.ihx = ldc<W>((half ? tx.ih_h : tx.ih_n) + i);
    r.bx = ldc<W>((half ? tx.b_h : tx.b_n) + i);
    r.ax = ldc<W>((half ? tx.a_h : tx.a_n) + i);
    r.ihy = __ldg((half ? ty.ih_h : ty.ih_n) + j);
    r.ys = half ? ((j < npml) || (j >= p.ny - npml)) : ((j < npml) || (j > p.ny - npml));
    r.by = r.ys ? __ldg((half ? ty.b_h : ty.b_n) + j) : 0.f;
    r.ay = r.ys ? __ldg((half ? ty.a_h : ty.a_n) + j) : 0.f;
}

// Source term E^{n+1} -= dt/eps J'^{n+1/2} for the taps in plane k of one
// column (first tap, count in cm): the increments were computed for the chunk's
// steps by k_tap_inc, so each tap costs two independent loads.
__device__ __forceinline__ void lean_taps(const int *__restrict__ tk, const float *__restrict__ inc, int k, int2 cm,
                                          float &x, float &y, float &z) {
    for (int u = cm.x; u < cm.x + cm.y; ++u) {
        const int code = __ldg(tk + u);
        const float v = __ldg(inc + u);
        if ((code >> 2) != k) continue;
        if ((code & 3) == 0) x += v;
        else if ((code & 3) == 1) y += v;
        else z += v;
    }
}

}  // namespace

// One plane k of the H update for the thread's W cells; YZ: the y/z recursion
// may apply (a block on a y or z slab); FAR: see kFarBytes.  ROWS: on rows of four the
// products of a difference off the slabs are fused, but for those of Hy and Hz in the last of every group of planes
// (last; GEN: known at run time only), and b psi is fused in the recursions.  On other rows no product is fused off the
// slabs, and in the recursions a d, but along x b psi with the four-cell kernels' rounding.  o: byte offset of the cells in a component, xo: of their
// x-slab entries.  exc, eyc: Ex, Ey of plane k (in), of plane k+1 (out).
template <int W, bool YZ, bool FAR, bool GEN, int ROWS>
__device__ __forceinline__ void h_plane(const StepParams<float> &p, const float *__restrict__ E, float *__restrict__ H,
                                        float *__restrict__ ps, const LeanRow<W> &r, int k, bool last, unsigned o, unsigned xo,
                                        Vec<W> &exc, Vec<W> &eyc) {
    const long long vol = p.vol;
    const unsigned plane = 4u * (unsigned)p.plane, pitch = 4u * (unsigned)p.pitch;
    const int npml = p.npml;
    constexpr bool four = ROWS == kRowsFour, bf = ROWS != kRowsScalar;
    const float *Ey = E + vol, *Ez = E + 2 * vol;
    float *Hy = H + vol, *Hz = H + 2 * vol;
    const Vec<W> ezc = ldc<W>(Ez, o);
    const Vec<W> exk = ldc<W>(E, o + plane), eyk = ldc<W>(Ey, o + plane);
    const Vec<W> exj = ldc<W>(E, o + pitch), ezj = ldc<W>(Ez, o + pitch);
    const float eyn = ldc1(Ey, o + 4u * W), ezn = ldc1(Ez, o + 4u * W);
    const float ihz = __ldg(p.lz.ih_h + k);
    Vec<W> hx = ldw<W>(H, o), hy = ldw<W>(Hy, o), hz = ldw<W>(Hz, o);
    float *px3 = ps + 3 * vol, *px4 = ps + 4 * vol;
    Vec<W> q3 = zv<W>(), q4 = zv<W>();
    if (r.xs) { q3 = ldw<W>(px3, xo); q4 = ldw<W>(px4, xo); }
    bool zs = false, ys = false;
    float bz = 0.f, az = 0.f;
    Vec<W> q0 = zv<W>(), q1 = zv<W>(), q2 = zv<W>(), q5 = zv<W>();
    if constexpr (YZ) {
        zs = (k < npml) || (k >= p.nz - npml);
        ys = r.ys;
        if (zs) { bz = __ldg(p.lz.b_h + k); az = __ldg(p.lz.a_h + k); }
        if (ys) { q0 = ldw<W>(ps, o); q5 = ldw<W>(ps + 5 * vol, o); }
        if (zs) { q1 = ldw<W>(ps + vol, o); q2 = ldw<W>(ps + 2 * vol, o); }
    }
    const Vec<W> ezx = up<W>(ezc, ezn), eyx = up<W>(eyc, eyn);   // Ez, Ey at i+1 .. i+W

    // Hx at (i, j+1/2, k+1/2)
    Vec<W> zy = dif<W>(ezj, ezc), yz = dif<W>(eyk, eyc), c;
    if constexpr (YZ) {
        zy = mul<W>(zy, r.ihy); yz = mul<W>(yz, ihz);
        if (ys) { cpml<W>(four, q0, zy, r.by, r.ay); stv<W>(ps, o, q0); }
        if (zs) { cpml<W>(four, q1, yz, bz, az); stv<W>(ps + vol, o, q1); }
        c = dif<W>(zy, yz);
    } else c = mulsub<W, false>(four, zy, r.ihy, mul<W>(yz, ihz));
    hx = mad<W>(c, -p.cH, hx);
    // Hy at (i+1/2, j, k+1/2)
    Vec<W> xz = dif<W>(exk, exc), zx = mul<W>(dif<W>(ezx, ezc), r.ihx);
    if constexpr (YZ) {
        xz = mul<W>(xz, ihz);
        if (zs) { cpml<W>(four, q2, xz, bz, az); stv<W>(ps + 2 * vol, o, q2); }
    }
    cpml<W>(bf, q3, zx, r.bx, r.ax);
    if (r.xs) stv<W>(px3, xo, q3);
    if constexpr (YZ) c = dif<W>(xz, zx);
    else c = mulsub<W, GEN && four>(four && !last, xz, ihz, zx);
    hy = mad<W>(c, -p.cH, hy);
    // Hz at (i+1/2, j+1/2, k)
    Vec<W> yx = mul<W>(dif<W>(eyx, eyc), r.ihx), xy = dif<W>(exj, exc);
    cpml<W>(bf, q4, yx, r.bx, r.ax);
    if (r.xs) stv<W>(px4, xo, q4);
    if constexpr (YZ) {
        xy = mul<W>(xy, r.ihy);
        if (ys) { cpml<W>(four, q5, xy, r.by, r.ay); stv<W>(ps + 5 * vol, o, q5); }
        c = dif<W>(yx, xy);
    } else c = submul<W, GEN && four>(four && !last, yx, xy, r.ihy);
    hz = mad<W>(c, -p.cH, hz);

    if constexpr (FAR) { stl<W>(H, o, hx); stl<W>(Hy, o, hy); stl<W>(Hz, o, hz); }
    else { stv<W>(H, o, hx); stv<W>(Hy, o, hy); stv<W>(Hz, o, hz); }
    exc = exk;
    eyc = eyk;
}

// H over the KZ planes from z block kb of the tile (xb, yb) of source s (the tile: 32 W
// cells of 4 rows, one W-cell column per thread): k_h_lean's block with its coordinates
// as arguments, for the wave-ordered step (k_h_lean keeps its own copy, compiled as tuned).
template <int W, int KZ>
__device__ __forceinline__ void h_tile(const StepParams<float> &p, const int jstep, int xb, int yb, int kb, int s) {
    const int i = (xb * kLeanX + (int)threadIdx.x) * W;
    const int j = yb * kLeanRows + (int)threadIdx.y;
    const int k0 = kb * KZ;
    if (i >= p.nx || j >= p.ny) return;
    const int k1 = min(k0 + KZ, p.nz);
    const int sl = slot_of(p, *p.step + jstep);
    const int plane = (int)p.plane, npml = p.npml;
    const long long vol = p.vol;
    const float *__restrict__ E = p.ering + (long long)s * p.ering_stride + (long long)sl * 3 * p.vol;
    float *__restrict__ H = p.H + (long long)s * 3 * vol;
    float *__restrict__ ps = p.psiL + (long long)s * 12 * vol;
    LeanRow<W> r;
    lean_row<W>(p, p.lx, p.ly, true, i, j, r);
    const int j0 = yb * kLeanRows;
    const bool yblk = (j0 < npml) || (j0 + kLeanRows > p.ny - npml);

    unsigned o = 4u * (unsigned)(k0 * plane + j * p.pitch + i), xo = r.xoff(p, k0);
    const unsigned dx = 4u * (unsigned)(p.ny * r.nxs);
    Vec<W> exc = ldc<W>(E, o), eyc = ldc<W>(E + p.vol, o);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk, o += 4u * (unsigned)plane, xo += dx) {
        const int k = k0 + kk;
        if (k >= k1) break;
        const bool last = (k & p.rnd.h_mask) == p.rnd.h_mask;
        if (yblk || k < npml || k >= p.nz - npml) h_plane<W, true, false, true, kRowsFour>(p, E, H, ps, r, k, last, o, xo, exc, eyc);
        else h_plane<W, false, false, true, kRowsFour>(p, E, H, ps, r, k, last, o, xo, exc, eyc);
    }
}

// GEN: the last z blocks have one plane (big_blocks), or groups of planes that round alike are not the z blocks.
template <int W, int KZ, int MINB, bool FAR, bool GEN, int ROWS>
__global__ void __launch_bounds__(kLeanX *kLeanRows, MINB) k_h_lean(const StepParams<float> p, const int jstep, const unsigned S,
                                                                       const unsigned mS, const int nbig) {
    const int i = (blockIdx.x * kLeanX + threadIdx.x) * W;
    const int j = blockIdx.y * kLeanRows + threadIdx.y;
    const int zb = (int)div_by(blockIdx.z, mS);   // the source runs fastest: the sources of one
    const int s = (int)(blockIdx.z - zb * S);     // z block follow one another
    const bool one = GEN && zb >= nbig;           // big_blocks
    const int k0 = one ? nbig * KZ + (zb - nbig) : zb * KZ, k1 = min(k0 + (one ? 1 : KZ), p.nz);
    if (i >= p.nx || j >= p.ny) return;
    const int plane = (int)p.plane, npml = p.npml;
    const long long vol = p.vol;
    LeanRow<W> r;
    lean_row<W>(p, p.lx, p.ly, true, i, j, r);
    pdl_wait();
    const int sl = slot_of(p, *p.step + jstep);
    const float *__restrict__ E = p.ering + (long long)s * p.ering_stride + (long long)sl * 3 * p.vol;
    float *__restrict__ H = p.H + (long long)s * 3 * vol;
    float *__restrict__ ps = p.psiL + (long long)s * 12 * vol;
    const int j0 = blockIdx.y * kLeanRows;
    const bool yblk = (j0 < npml) || (j0 + kLeanRows > p.ny - npml);

    unsigned o = 4u * (unsigned)(k0 * plane + j * p.pitch + i), xo = r.xoff(p, k0);
    const unsigned dx = 4u * (unsigned)(p.ny * r.nxs);
    Vec<W> exc = ldc<W>(E, o), eyc = ldc<W>(E + p.vol, o);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk, o += 4u * (unsigned)plane, xo += dx) {
        const int k = k0 + kk;
        if (k >= k1) break;
        const bool last = GEN ? (k & p.rnd.h_mask) == p.rnd.h_mask : kk == KZ - 1;
        if (yblk || k < npml || k >= p.nz - npml) h_plane<W, true, FAR, GEN, ROWS>(p, E, H, ps, r, k, last, o, xo, exc, eyc);
        else h_plane<W, false, FAR, GEN, ROWS>(p, E, H, ps, r, k, last, o, xo, exc, eyc);
    }
}

// H loads of the E update: plain (the H kernel may still run when an E block starts, see pdl_wait), or (CG)
// from L2 only, for H that other blocks of the same launch wrote (L1 is not coherent with them).
template <int W, bool CG> __device__ __forceinline__ Vec<W> ldh(const float *b, unsigned o) {
    if constexpr (!CG) return ldw<W>(b, o);
    const float *p = reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o);
    Vec<W> r;
    if constexpr (W == 1) r.v[0] = __ldcg(p);
    else { const float2 t = __ldcg(reinterpret_cast<const float2 *>(p)); r.v[0] = t.x; r.v[1] = t.y; }
    return r;
}
template <bool CG> __device__ __forceinline__ float ldh1(const float *b, unsigned o) {
    const float *p = reinterpret_cast<const float *>(reinterpret_cast<const char *>(b) + o);
    return CG ? __ldcg(p) : *p;
}

// One plane k of the E update; o, xo as in h_plane; oj, oi: from o to the lower neighbours along y and x (0 on
// the outer faces).  ROWS, GEN: as in h_plane, but on rows of four Ey's products are never fused, and on
// other rows all recursions fuse b psi with the four-cell kernels' rounding; there the taps are added one by one, as the
// general kernels add them.  hxm, hym: Hx, Hy of plane k-1 (in), of plane k (out).
template <int W, bool YZ, bool CG, bool GEN, int ROWS>
__device__ __forceinline__ void e_plane(const StepParams<float> &p, const float *__restrict__ Eo, float *__restrict__ En,
                                        const float *H, float *__restrict__ ps, const LeanRow<W> &r, int s,
                                        int S, int jstep, int k, bool last, unsigned o, unsigned xo, unsigned oj,
                                        unsigned oi, bool taps, Vec<W> &hxm, Vec<W> &hym) {
    const long long vol = p.vol;
    const int npml = p.npml;
    constexpr bool four = ROWS == kRowsFour, bf = ROWS != kRowsScalar;
    const float *__restrict__ cE = p.cEm;
    const float *Hy = H + vol, *Hz = H + 2 * vol;
    const Vec<W> hxc = ldh<W, CG>(H, o), hyc = ldh<W, CG>(Hy, o), hzc = ldh<W, CG>(Hz, o);
    const Vec<W> hxj = ldh<W, CG>(H, o - oj), hzj = ldh<W, CG>(Hz, o - oj);
    const float hyp = ldh1<CG>(Hy, o - oi), hzp = ldh1<CG>(Hz, o - oi);
    const Vec<W> eo0 = lde<W>(Eo, o), eo1 = lde<W>(Eo + vol, o), eo2 = lde<W>(Eo + 2 * vol, o);
    const Vec<W> c0 = ldc<W>(cE, o), c1 = ldc<W>(cE + vol, o), c2 = ldc<W>(cE + 2 * vol, o);
    const float ihz = __ldg(p.lz.ih_n + k);
    float *px3 = ps + 3 * vol, *px4 = ps + 4 * vol;
    Vec<W> q3 = zv<W>(), q4 = zv<W>();
    if (r.xs) { q3 = ldw<W>(px3, xo); q4 = ldw<W>(px4, xo); }
    bool zs = false, ys = false;
    float bz = 0.f, az = 0.f;
    Vec<W> q0 = zv<W>(), q1 = zv<W>(), q2 = zv<W>(), q5 = zv<W>();
    if constexpr (YZ) {
        zs = (k < npml) || (k > p.nz - npml);
        ys = r.ys;
        if (zs) { bz = __ldg(p.lz.b_n + k); az = __ldg(p.lz.a_n + k); }
        if (ys) { q0 = ldw<W>(ps, o); q5 = ldw<W>(ps + 5 * vol, o); }
        if (zs) { q1 = ldw<W>(ps + vol, o); q2 = ldw<W>(ps + 2 * vol, o); }
    }
    const Vec<W> hzx = down<W>(hzp, hzc), hyx = down<W>(hyp, hyc);   // Hz, Hy at i-1 .. i+W-2

    // Ex at (i+1/2, j, k)
    Vec<W> zy = dif<W>(hzc, hzj), yz = dif<W>(hyc, hym), c;
    if constexpr (YZ) {
        zy = mul<W>(zy, r.ihy); yz = mul<W>(yz, ihz);
        if (ys) { cpml<W>(bf, q0, zy, r.by, r.ay); stv<W>(ps, o, q0); }
        if (zs) { cpml<W>(bf, q1, yz, bz, az); stv<W>(ps + vol, o, q1); }
        c = dif<W>(zy, yz);
    } else c = mulsub<W, false>(four, zy, r.ihy, mul<W>(yz, ihz));
    Vec<W> e0 = mad<W>(c, c0, eo0);
    // Ey at (i, j+1/2, k)
    Vec<W> xz = dif<W>(hxc, hxm), zx = mul<W>(dif<W>(hzc, hzx), r.ihx);
    if constexpr (YZ) {
        xz = mul<W>(xz, ihz);
        if (zs) { cpml<W>(bf, q2, xz, bz, az); stv<W>(ps + 2 * vol, o, q2); }
    }
    cpml<W>(bf, q3, zx, r.bx, r.ax);
    if (r.xs) stv<W>(px3, xo, q3);
    if constexpr (YZ) c = dif<W>(xz, zx);
    else c = mulsub<W, false>(false, xz, ihz, zx);
    Vec<W> e1 = mad<W>(c, c1, eo1);
    // Ez at (i, j, k+1/2)
    Vec<W> yx = mul<W>(dif<W>(hyc, hyx), r.ihx), xy = dif<W>(hxc, hxj);
    cpml<W>(bf, q4, yx, r.bx, r.ax);
    if (r.xs) stv<W>(px4, xo, q4);
    if constexpr (YZ) {
        xy = mul<W>(xy, r.ihy);
        if (ys) { cpml<W>(bf, q5, xy, r.by, r.ay); stv<W>(ps + 5 * vol, o, q5); }
        c = dif<W>(yx, xy);
    } else c = submul<W, GEN && four>(four && !last, yx, xy, r.ihy);
    Vec<W> e2 = mad<W>(c, c2, eo2);

    if (taps) {
        const int2 *cm = p.colmap + (long long)s * p.colmap_stride + r.j * p.pitch + r.i;
        const int *tk = p.tapk + (long long)s * p.itap_stride;
        const float *inc = p.inc + ((long long)jstep * S + s) * p.inc_ntl;
        for (int e = 0; e < W; ++e) {
            const int2 c = __ldg(cm + e);
            if (c.y == 0) continue;
            if constexpr (four) {
                float3 a = make_float3(0.f, 0.f, 0.f);
                lean_taps(tk, inc, k, c, a.x, a.y, a.z);
                e0.v[e] += a.x; e1.v[e] += a.y; e2.v[e] += a.z;
            } else lean_taps(tk, inc, k, c, e0.v[e], e1.v[e], e2.v[e]);
        }
    }
    stv<W>(En, o, e0);
    stv<W>(En + vol, o, e1);
    stv<W>(En + 2 * vol, o, e2);
    hxm = hxc;
    hym = hyc;
}

// E over the KZ planes from z block kb of the tile (xb, yb) of source s (S sources per
// launch): k_e_lean's block with its coordinates as arguments, H read through ldh<CG>.
template <int W, int KZ, bool CG>
__device__ __forceinline__ void e_tile(const StepParams<float> &p, const int jstep, int xb, int yb, int kb, int s,
                                       int S) {
    const int i = (xb * kLeanX + (int)threadIdx.x) * W;
    const int j = yb * kLeanRows + (int)threadIdx.y;
    const int k0 = kb * KZ;
    if (i >= p.nx || j >= p.ny) return;
    const int k1 = min(k0 + KZ, p.nz);
    const int sl = slot_of(p, *p.step + jstep);
    const int plane = (int)p.plane, pitch = p.pitch, npml = p.npml;
    const long long vol = p.vol;
    const float *__restrict__ ring = p.ering + (long long)s * p.ering_stride;
    const float *__restrict__ Eo = ring + (long long)sl * 3 * p.vol;
    float *__restrict__ En = const_cast<float *>(ring) + (long long)slot_after(p, sl) * 3 * p.vol;
    const float *H = p.H + (long long)s * 3 * vol;
    float *__restrict__ ps = p.psiL + (long long)s * 12 * vol + 6 * vol;
    LeanRow<W> r;
    lean_row<W>(p, p.lx, p.ly, false, i, j, r);
    const int j0 = yb * kLeanRows;
    const bool yblk = (j0 < npml) || (j0 + kLeanRows - 1 > p.ny - npml);
    const bool taps = p.colmap && p.inc && p.tflag[s * p.tflag_stride + j * p.nseg + (i >> 5)];

    unsigned o = 4u * (unsigned)(k0 * plane + j * pitch + i), xo = r.xoff(p, k0);
    const unsigned dx = 4u * (unsigned)(p.ny * r.nxs), oj = j > 0 ? 4u * (unsigned)pitch : 0u, oi = i > 0 ? 4u : 0u;
    const unsigned om = (k0 > 0) ? o - 4u * (unsigned)plane : o;      // clamped on the bottom face
    Vec<W> hxm = ldh<W, CG>(H, om), hym = ldh<W, CG>(H + p.vol, om);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk, o += 4u * (unsigned)plane, xo += dx) {
        const int k = k0 + kk;
        if (k >= k1) break;
        const bool last = (k & p.rnd.e_mask) == p.rnd.e_mask;
        if (yblk || k < npml || k > p.nz - npml)
            e_plane<W, true, CG, true, kRowsFour>(p, Eo, En, H, ps, r, s, S, jstep, k, last, o, xo, oj, oi, taps, hxm, hym);
        else e_plane<W, false, CG, true, kRowsFour>(p, Eo, En, H, ps, r, s, S, jstep, k, last, o, xo, oj, oi, taps, hxm, hym);
    }
}

template <int W, int KZ, int MINB, bool FAR, bool GEN, int ROWS>
__global__ void __launch_bounds__(kLeanX *kLeanRows, MINB) k_e_lean(const StepParams<float> p, const int jstep, const unsigned S,
                                                                       const unsigned mS, const int nbig) {
    const int i = (blockIdx.x * kLeanX + threadIdx.x) * W;
    const int j = blockIdx.y * kLeanRows + threadIdx.y;
    const int zq = (int)div_by(blockIdx.z, mS);   // the source runs fastest: the sources of one z
    const int s = (int)(blockIdx.z - zq * S);     // block share the dt/eps reads in L2
    int k0 = (FAR ? (p.nz + KZ - 1) / KZ - 1 - zq : zq) * KZ, k1 = min(k0 + KZ, p.nz);   // downwards where FAR (kFarBytes)
    if constexpr (GEN) {                          // big_blocks
        const int at = zq < nbig ? zq * KZ : nbig * KZ + (zq - nbig), len = zq < nbig ? KZ : 1;
        k0 = FAR ? max(p.nz - at - len, 0) : at;
        k1 = FAR ? p.nz - at : min(at + len, p.nz);
    }
    if (i >= p.nx || j >= p.ny) return;
    LeanRow<W> r;
    lean_row<W>(p, p.lx, p.ly, false, i, j, r);
    pdl_wait();
    const int sl = slot_of(p, *p.step + jstep);
    const int plane = (int)p.plane, pitch = p.pitch, npml = p.npml;
    const long long vol = p.vol;
    const float *__restrict__ ring = p.ering + (long long)s * p.ering_stride;
    const float *__restrict__ Eo = ring + (long long)sl * 3 * p.vol;
    float *__restrict__ En = const_cast<float *>(ring) + (long long)slot_after(p, sl) * 3 * p.vol;
    const float *H = p.H + (long long)s * 3 * vol;        // plain loads: see pdl_wait
    float *__restrict__ ps = p.psiL + (long long)s * 12 * vol + 6 * vol;
    const int j0 = blockIdx.y * kLeanRows;
    const bool yblk = (j0 < npml) || (j0 + kLeanRows - 1 > p.ny - npml);
    const bool taps = p.colmap && p.inc && p.tflag[s * p.tflag_stride + j * p.nseg + (i >> 5)];

    unsigned o = 4u * (unsigned)(k0 * plane + j * pitch + i), xo = r.xoff(p, k0);
    const unsigned dx = 4u * (unsigned)(p.ny * r.nxs), oj = j > 0 ? 4u * (unsigned)pitch : 0u, oi = i > 0 ? 4u : 0u;
    const unsigned om = (k0 > 0) ? o - 4u * (unsigned)plane : o;      // clamped on the bottom face
    Vec<W> hxm = ldh<W, false>(H, om), hym = ldh<W, false>(H + p.vol, om);
#pragma unroll
    for (int kk = 0; kk < KZ; ++kk, o += 4u * (unsigned)plane, xo += dx) {
        const int k = k0 + kk;
        if (k >= k1) break;
        const bool last = GEN ? (k & p.rnd.e_mask) == p.rnd.e_mask : kk == KZ - 1;
        if (yblk || k < npml || k > p.nz - npml) e_plane<W, true, false, GEN, ROWS>(p, Eo, En, H, ps, r, s, (int)S, jstep, k, last, o, xo, oj, oi, taps, hxm, hym);
        else e_plane<W, false, false, GEN, ROWS>(p, Eo, En, H, ps, r, s, (int)S, jstep, k, last, o, xo, oj, oi, taps, hxm, hym);
    }
}

// Launches of one half (H or E) on rows of one kind; the kinds and halves are compiled in three units (see the end).
namespace {
template <int W, int KZ, int MB, int ROWS, bool H, bool GEN, bool FAR>
void lean_launch(const StepParams<float> &p, dim3 grid, int nbig, int S, int jstep, cudaStream_t st) {
    const dim3 block(kLeanX, kLeanRows);
    const unsigned mS = div_magic((unsigned)S);
    if constexpr (H) launch_pdl(k_h_lean<W, KZ, MB, FAR, GEN, ROWS>, grid, block, st, p, jstep, (unsigned)S, mS, nbig);
    else launch_pdl(k_e_lean<W, KZ, MB, FAR, GEN, ROWS>, grid, block, st, p, jstep, (unsigned)S, mS, nbig);
}
template <int ROWS, bool H, int W, int KZ, int MB>
void lean_go(const StepParams<float> &p, int S, int jstep, cudaStream_t st) {
    const int nv = (p.nx + W - 1) / W, nzb = (p.nz + KZ - 1) / KZ;
    const int gx = (nv + kLeanX - 1) / kLeanX, gy = (p.ny + kLeanRows - 1) / kLeanRows;
    const int nbig = big_blocks(p.sms, nzb, KZ, gx * gy * S, MB);
    const dim3 grid(gx, gy, (nbig < nzb ? nbig + p.nz - nbig * KZ : nzb) * S);
    const bool gen = nbig < nzb || (ROWS == kRowsFour && (H ? p.rnd.h_mask : p.rnd.e_mask) != KZ - 1);
    const bool far = far_fields(p.vol, S);
    if constexpr (KZ > 1 || ROWS == kRowsFour) {
        if (gen && far) return lean_launch<W, KZ, MB, ROWS, H, true, true>(p, grid, nbig, S, jstep, st);
        if (gen) return lean_launch<W, KZ, MB, ROWS, H, true, false>(p, grid, nbig, S, jstep, st);
    }
    if (far) lean_launch<W, KZ, MB, ROWS, H, false, true>(p, grid, nbig, S, jstep, st);
    else lean_launch<W, KZ, MB, ROWS, H, false, false>(p, grid, nbig, S, jstep, st);
}
template <int ROWS, bool H, int W, int MB>
bool lean_kz(const StepParams<float> &p, int S, int jstep, cudaStream_t st, int kz) {
    switch (kz) {
        case 1: lean_go<ROWS, H, W, 1, MB>(p, S, jstep, st); return true;
        case 2: lean_go<ROWS, H, W, 2, MB>(p, S, jstep, st); return true;
        case 4: lean_go<ROWS, H, W, 4, MB>(p, S, jstep, st); return true;
        default: return false;
    }
}
template <int ROWS, bool H>
bool lean_half(const StepParams<float> &p, int S, int jstep, cudaStream_t st, int w, int kz, int mb) {
    if (w == 1 && mb == 6) return lean_kz<ROWS, H, 1, 6>(p, S, jstep, st, kz);
    if (w == 1 && mb == 8) return lean_kz<ROWS, H, 1, 8>(p, S, jstep, st, kz);
    if (w == 2 && mb == 4) return lean_kz<ROWS, H, 2, 4>(p, S, jstep, st, kz);
    if (w == 2 && mb == 6) return lean_kz<ROWS, H, 2, 6>(p, S, jstep, st, kz);
    if (w == 2 && mb == 8) return lean_kz<ROWS, H, 2, 8>(p, S, jstep, st, kz);
    return false;
}
}  // namespace

// The instances for other rows than multiples of four: kern_lean_h.cu and kern_lean_e.cu.
bool lean_other_h(const StepParams<float> &p, int S, int jstep, cudaStream_t st, int w, int kz, int mb);
bool lean_other_e(const StepParams<float> &p, int S, int jstep, cudaStream_t st, int w, int kz, int mb);
#if CSEM_LEAN_UNIT == 1
bool lean_other_h(const StepParams<float> &p, int S, int jstep, cudaStream_t st, int w, int kz, int mb) {
    return p.rnd.h_bf ? lean_half<kRowsVec, true>(p, S, jstep, st, w, kz, mb)
                      : lean_half<kRowsScalar, true>(p, S, jstep, st, w, kz, mb);
}
#elif CSEM_LEAN_UNIT == 2
bool lean_other_e(const StepParams<float> &p, int S, int jstep, cudaStream_t st, int w, int kz, int mb) {
    return p.rnd.e_bf ? lean_half<kRowsVec, false>(p, S, jstep, st, w, kz, mb)
                      : lean_half<kRowsScalar, false>(p, S, jstep, st, w, kz, mb);
}
#else

// One whole step (H then E) in one launch, ordered by tickets: every block takes the next
// ticket from a counter, and the tickets run through the z blocks ("chunks") as
//   H(0) .. H(lag-1), then H(c + lag), E(c) for c = 0, 1, .., then the remaining E(c),
// each chunk being all tiles of its z block (the sources of a tile next to one another).
// The E tiles of chunk c read H of chunks c and c-1, which the H tiles of those chunks
// write in the same launch: the H tiles count themselves done per chunk (after a fence),
// and an E tile's thread 0 waits (bounded, about a second) until both chunks are complete.
// No H tile waits, and an E tile waits only for tiles that took earlier tickets, so every
// wait ends.  The lag keeps the E tiles far enough behind that the H tiles they need have
// usually finished, and near enough that the E^n and H^{n+1/2} they read were touched a few
// chunks before and are still in L2: that is the point of the ordering -- E reads them
// from L2 instead of DRAM.  H is read from L2 only (__ldcg) by the E tiles.  The last
// block to finish resets the counters, so the next launch starts from zero.
// wave[0]: ticket counter, wave[1]: finished blocks, wave[2 + c]: H tiles done in chunk c.
// Chunks of the wave-ordered step: z blocks, and tiles per z block (every source).
template <int W, int KZ> __device__ __forceinline__ unsigned wave_nkb(const StepParams<float> &p) {
    return (unsigned)((p.nz + KZ - 1) / KZ);
}
template <int W, int KZ> __device__ __forceinline__ unsigned wave_tc(const StepParams<float> &p, int S) {
    return (unsigned)((p.nx / W + kLeanX - 1) / kLeanX) * (unsigned)((p.ny + kLeanRows - 1) / kLeanRows) * (unsigned)S;
}

template <int W, int KZ, int MINB>
__global__ void __launch_bounds__(kLeanX *kLeanRows, MINB) k_step_wave(const StepParams<float> p, const int jstep,
                                                                     const int S, const int lag) {
    __shared__ int tile[5];                        // H (1) or E (0), z block, source, x tile, y tile
    const int tid = threadIdx.y * kLeanX + threadIdx.x;
    if (tid == 0) {                                // thread 0 takes the ticket and decodes it
        const unsigned t = atomicAdd(p.wave, 1u);
        const unsigned nkb = wave_nkb<W, KZ>(p), tc = wave_tc<W, KZ>(p, S);
        const unsigned nxb = (unsigned)((p.nx / W + kLeanX - 1) / kLeanX);
        const unsigned L = (unsigned)min(max(lag, 1), (int)nkb);
        bool h;
        unsigned kb, r;
        if (t < L * tc) {
            h = true; kb = t / tc; r = t % tc;
        } else {
            const unsigned u = t - L * tc, mid = (nkb - L) * 2u * tc;
            if (u < mid) {
                const unsigned ph = u / (2u * tc), q = u % (2u * tc);
                h = q < tc;
                kb = h ? L + ph : ph;
                r = h ? q : q - tc;
            } else {
                h = false; kb = (nkb - L) + (u - mid) / tc; r = (u - mid) % tc;
            }
        }
        tile[0] = h ? 1 : 0;
        tile[1] = (int)kb;
        tile[2] = (int)(r % (unsigned)S);
        tile[3] = (int)((r / (unsigned)S) % nxb);
        tile[4] = (int)(r / ((unsigned)S * nxb));
        if (!h) {                                  // E: wait until H of z blocks kb and kb - 1 is complete
            // the test hook makes the wait unsatisfiable; once one wait gave up, the others skip it
            const unsigned need = tc + (p.fault_tx ? 1u : 0u);
            const unsigned *done = p.wave + 2;
            const unsigned long long t0 = gtimer_ns();
            for (unsigned it = 0;; ++it) {
                const unsigned a = *(volatile const unsigned *)&done[kb];
                const unsigned b = kb ? *(volatile const unsigned *)&done[kb - 1] : need;
                if (a >= need && b >= need) break;
                if ((*(volatile int *)p.err) & kErrWaveWait) break;
                if (it >= (1u << 24) || ((it & 63) == 63 && gtimer_ns() - t0 > kWaitNs)) {
                    atomicOr(p.err, kErrWaveWait);
                    break;
                }
                __nanosleep(128);
            }
            __threadfence();
        }
    }
    __syncthreads();
    if (tile[0]) {
        h_tile<W, KZ>(p, jstep, tile[3], tile[4], tile[1], tile[2]);
        __syncthreads();
        if (tid == 0) {
            __threadfence();                       // the block's H stores before the count
            atomicAdd(p.wave + 2 + tile[1], 1u);
        }
    } else {
        e_tile<W, KZ, true>(p, jstep, tile[3], tile[4], tile[1], tile[2], S);
    }
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        const unsigned nkb = wave_nkb<W, KZ>(p);
        if (atomicAdd(p.wave + 1, 1u) == 2u * nkb * wave_tc<W, KZ>(p, S) - 1u) {   // all others finished
            p.wave[0] = 0u;
            p.wave[1] = 0u;
            for (unsigned c = 0; c < nkb; ++c) p.wave[2 + c] = 0u;
            __threadfence();
        }
    }
}

// Increment -dt/eps J'^{n+1/2} of every injection tap (Sec. 2, Eq. 4 source
// term; the amplitude sum_j coef_j T_j(n) in FP64, one rounding to FP32, the same
// value the other step kernels add) for the steps jstep in [0, nsteps) after the
// device step counter: inc[(jstep*S + s)*inc_ntl + u].
__global__ void k_tap_inc(const StepParams<float> p, const int S, const int nsteps, const int nt) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int ntl = p.inc_ntl;
    if (t >= (long long)nsteps * S * ntl) return;
    const int u = (int)(t % ntl);
    const int s = (int)((t / ntl) % S);
    const int jstep = (int)(t / ((long long)ntl * S));
    pdl_wait();
    const int n = *p.step + jstep;
    float v = 0.f;
    if (n < nt) {
        const Tap tp = p.itaps[(long long)s * p.itap_stride + u];
        const double *cf = p.coef + ((long long)s * p.n_emit + tp.emit) * p.J;
        const double *T = p.T + (long long)n * p.J;
        double amp = 0.0;
        for (int jj = 0; jj < p.J; ++jj) amp += cf[jj] * T[jj];
        const long long o = (long long)tp.comp * p.vol + tp.idx;   // up to 3 * 2^30
        v = (float)(-(double)p.cE[o] * tp.w * amp);
    }
    p.inc[t] = v;
}

// dt/eps with the PEC edges zeroed: Ex needs 1 <= j < ny, 1 <= k < nz, i < nx;
// Ey 1 <= i < nx, 1 <= k < nz, j < ny; Ez 1 <= i < nx, 1 <= j < ny, k < nz.
__global__ void k_mask_coef(const StepParams<float> p, const float *__restrict__ cE, float *__restrict__ cEm) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * p.vol) return;
    const int c = (int)(t / p.vol);
    const int idx = (int)(t - (long long)c * p.vol);
    const int k = idx / (int)p.plane;
    const int r = idx - k * (int)p.plane;
    const int j = r / p.pitch;
    const int i = r - j * p.pitch;
    const bool xi = (i >= 1 && i < p.nx), yi = (j >= 1 && j < p.ny), zi = (k >= 1 && k < p.nz);
    bool ok;
    if (c == 0) ok = (i < p.nx) && yi && zi;
    else if (c == 1) ok = xi && (j < p.ny) && zi;
    else ok = xi && yi && (k < p.nz);
    cEm[t] = ok ? cE[t] : 0.f;
}

cudaError_t launch_field_lean(const StepParams<float> &p, int S, int jstep, cudaStream_t st, bool h, int w, int kz,
                              int mb) {
    if (!p.psiL || !p.cEm || !p.lx.ih_n) return cudaErrorInvalidValue;
    bool ok;
    if (p.nx % 4 != 0) ok = h ? lean_other_h(p, S, jstep, st, w, kz, mb) : lean_other_e(p, S, jstep, st, w, kz, mb);
    else ok = h ? lean_half<kRowsFour, true>(p, S, jstep, st, w, kz, mb) : lean_half<kRowsFour, false>(p, S, jstep, st, w, kz, mb);
    if (!ok) return cudaErrorInvalidValue;
    g_launches++;
    return cudaGetLastError();
}

bool wave_supported(const StepParams<float> &p, int kz, int mb) {
    return p.wave && p.nx % 4 == 0 && p.psiL && p.cEm && p.lx.ih_n && (kz == 2 || kz == 4) &&
           (mb == 6 || mb == 8) && p.nz <= kMaxWaveChunks * kz;
}

cudaError_t launch_step_wave(const StepParams<float> &p, int S, int jstep, cudaStream_t st) {
    const int kz = p.WAVE_kz, mb = p.WAVE_mb, lag = p.WAVE_lag;
    if (!wave_supported(p, kz, mb) || lag < 1) return cudaErrorInvalidValue;
    const long long nxb = (p.nx / 2 + kLeanX - 1) / kLeanX, nyb = (p.ny + kLeanRows - 1) / kLeanRows;
    const long long nblk = 2LL * ((p.nz + kz - 1) / kz) * nxb * nyb * S;
    const dim3 block(kLeanX, kLeanRows);
    if (kz == 2 && mb == 6) k_step_wave<2, 2, 6><<<(unsigned)nblk, block, 0, st>>>(p, jstep, S, lag);
    else if (kz == 2) k_step_wave<2, 2, 8><<<(unsigned)nblk, block, 0, st>>>(p, jstep, S, lag);
    else if (mb == 6) k_step_wave<2, 4, 6><<<(unsigned)nblk, block, 0, st>>>(p, jstep, S, lag);
    else k_step_wave<2, 4, 8><<<(unsigned)nblk, block, 0, st>>>(p, jstep, S, lag);
    g_launches++;
    return cudaGetLastError();
}

cudaError_t launch_tap_inc(const StepParams<float> &p, int S, int nsteps, int nt, cudaStream_t st) {
    const long long n = (long long)nsteps * S * p.inc_ntl;
    if (n <= 0 || !p.inc || !p.itaps) return cudaSuccess;
    g_launches++;
    return launch_pdl(k_tap_inc, dim3((unsigned)((n + 255) / 256)), dim3(256), st, p, S, nsteps, nt);
}

cudaError_t launch_mask_coef(const StepParams<float> &p, const float *cE, float *cEm, cudaStream_t st) {
    const long long n = 3 * p.vol;
    k_mask_coef<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(p, cE, cEm);
    g_launches++;
    return cudaGetLastError();
}

#endif  // CSEM_LEAN_UNIT

}  // namespace csem
