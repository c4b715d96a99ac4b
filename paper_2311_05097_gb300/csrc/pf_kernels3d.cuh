// 3D fused time step: D3Q7 order-parameter lattice and D3Q19 flow lattice
// (the 3D extension of Sec. 3; see the readings of the 3D lattices in the
// oracle), pull streaming, Hermite-moment MRT collision.
//
// A CTA owns a TX x TY column of cells and marches through a chunk of planes in z.
// Shared-memory rings hold the planes the stencils need:
//   phi, phi0       planes z-2 .. z+2 on the tile + 2 frame (ring of 5),
//   mu_phi          planes z-1 .. z+1 on the tile + 1 frame (ring of 4),
//   T = S u - u S   (antisymmetric: xy, xz, yz) of the previous step, planes
//                   z-1 .. z+1 on the tile + 1 frame (ring of 4).
// Each plane costs two barriers.  Halo re-reads hit L2; each cell's own
// populations are read once from DRAM.
#pragma once

#include "pf_common.cuh"

namespace pf {

// D3Q19 velocities: rest, 6 faces, 12 edges; D3Q7 uses the first 7.
__device__ constexpr int C19X[19] = {0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0};
__device__ constexpr int C19Y[19] = {0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1};
__device__ constexpr int C19Z[19] = {0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1};
// opposite direction (pairs 1-2, 3-4, ..., 17-18)
__device__ __forceinline__ int opp19(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }

template <class R>
__device__ __forceinline__ void from_hermite19(const R h[19], R f[19], R cs2);

// Hermite-moment MRT collision of one D3Q19 cell.  Raw moments m = M0 f with
// rows 1, c_a, c_a^2, c_x c_y, c_x c_z, c_y c_z, c_x c_y^2, c_x c_z^2,
// c_y c_x^2, c_y c_z^2, c_z c_x^2, c_z c_y^2, c_x^2 c_y^2, c_x^2 c_z^2,
// c_y^2 c_z^2; Hermite moments h = N_H m; relaxation in h; back by N_H^-1
// and M0^-1.
template <class R>
__device__ __forceinline__ void collide19(R f[19], const R heq[19], const R hF[19], const R S[19],
                                          R cs2)
{
    const R cs4 = cs2 * cs2;
    R m[19];
    m[0] = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8] + f[9] + f[10] + f[11] + f[12] +
           f[13] + f[14] + f[15] + f[16] + f[17] + f[18];
    m[1] = f[1] - f[2] + f[7] - f[8] + f[9] - f[10] + f[11] - f[12] + f[13] - f[14];
    m[2] = f[3] - f[4] + f[7] - f[8] - f[9] + f[10] + f[15] - f[16] + f[17] - f[18];
    m[3] = f[5] - f[6] + f[11] - f[12] - f[13] + f[14] + f[15] - f[16] - f[17] + f[18];
    const R exy = f[7] + f[8] + f[9] + f[10], exz = f[11] + f[12] + f[13] + f[14],
            eyz = f[15] + f[16] + f[17] + f[18];
    m[4] = f[1] + f[2] + exy + exz;
    m[5] = f[3] + f[4] + exy + eyz;
    m[6] = f[5] + f[6] + exz + eyz;
    m[7] = f[7] + f[8] - f[9] - f[10];
    m[8] = f[11] + f[12] - f[13] - f[14];
    m[9] = f[15] + f[16] - f[17] - f[18];
    m[10] = f[7] - f[8] + f[9] - f[10];    // c_x c_y^2
    m[11] = f[11] - f[12] + f[13] - f[14]; // c_x c_z^2
    m[12] = f[7] - f[8] - f[9] + f[10];    // c_y c_x^2
    m[13] = f[15] - f[16] + f[17] - f[18]; // c_y c_z^2
    m[14] = f[11] - f[12] - f[13] + f[14]; // c_z c_x^2
    m[15] = f[15] - f[16] - f[17] + f[18]; // c_z c_y^2
    m[16] = exy;
    m[17] = exz;
    m[18] = eyz;
    R h[19];
    h[0] = m[0];
    h[1] = m[1];
    h[2] = m[2];
    h[3] = m[3];
    h[4] = m[4] - cs2 * m[0];
    h[5] = m[5] - cs2 * m[0];
    h[6] = m[6] - cs2 * m[0];
    h[7] = m[7];
    h[8] = m[8];
    h[9] = m[9];
    h[10] = m[10] - cs2 * m[1];
    h[11] = m[11] - cs2 * m[1];
    h[12] = m[12] - cs2 * m[2];
    h[13] = m[13] - cs2 * m[2];
    h[14] = m[14] - cs2 * m[3];
    h[15] = m[15] - cs2 * m[3];
    h[16] = m[16] - cs2 * (m[4] + m[5]) + cs4 * m[0];
    h[17] = m[17] - cs2 * (m[4] + m[6]) + cs4 * m[0];
    h[18] = m[18] - cs2 * (m[5] + m[6]) + cs4 * m[0];
#pragma unroll
    for (int k = 0; k < 19; ++k)
        h[k] = h[k] - S[k] * (h[k] - heq[k]) + (R(1) - R(0.5) * S[k]) * hF[k];
    from_hermite19<R>(h, f, cs2);
}

// D3Q19 populations from Hermite moments: raw moments m = N_H^-1 h, then
// f = M0^-1 m.
template <class R>
__device__ __forceinline__ void from_hermite19(const R h[19], R f[19], R cs2)
{
    const R cs4 = cs2 * cs2;
    R m[19];
    m[0] = h[0];
    m[1] = h[1];
    m[2] = h[2];
    m[3] = h[3];
    m[4] = h[4] + cs2 * h[0];
    m[5] = h[5] + cs2 * h[0];
    m[6] = h[6] + cs2 * h[0];
    m[7] = h[7];
    m[8] = h[8];
    m[9] = h[9];
    m[10] = h[10] + cs2 * h[1];
    m[11] = h[11] + cs2 * h[1];
    m[12] = h[12] + cs2 * h[2];
    m[13] = h[13] + cs2 * h[2];
    m[14] = h[14] + cs2 * h[3];
    m[15] = h[15] + cs2 * h[3];
    m[16] = h[16] + cs2 * (h[4] + h[5]) + cs4 * h[0];
    m[17] = h[17] + cs2 * (h[4] + h[6]) + cs4 * h[0];
    m[18] = h[18] + cs2 * (h[5] + h[6]) + cs4 * h[0];
    const R hh = R(0.5), q = R(0.25);
    f[0] = m[0] - m[4] - m[5] - m[6] + m[16] + m[17] + m[18];
    f[1] = hh * (m[1] + m[4] - m[10] - m[11] - m[16] - m[17]);
    f[2] = hh * (-m[1] + m[4] + m[10] + m[11] - m[16] - m[17]);
    f[3] = hh * (m[2] + m[5] - m[12] - m[13] - m[16] - m[18]);
    f[4] = hh * (-m[2] + m[5] + m[12] + m[13] - m[16] - m[18]);
    f[5] = hh * (m[3] + m[6] - m[14] - m[15] - m[17] - m[18]);
    f[6] = hh * (-m[3] + m[6] + m[14] + m[15] - m[17] - m[18]);
    f[7] = q * (m[7] + m[10] + m[12] + m[16]);
    f[8] = q * (m[7] - m[10] - m[12] + m[16]);
    f[9] = q * (-m[7] + m[10] - m[12] + m[16]);
    f[10] = q * (-m[7] - m[10] + m[12] + m[16]);
    f[11] = q * (m[8] + m[11] + m[14] + m[17]);
    f[12] = q * (m[8] - m[11] - m[14] + m[17]);
    f[13] = q * (-m[8] + m[11] - m[14] + m[17]);
    f[14] = q * (-m[8] - m[11] + m[14] + m[17]);
    f[15] = q * (m[9] + m[13] + m[15] + m[18]);
    f[16] = q * (m[9] - m[13] - m[15] + m[18]);
    f[17] = q * (-m[9] + m[13] - m[15] + m[18]);
    f[18] = q * (-m[9] - m[13] + m[15] + m[18]);
}

// D3Q7 Hermite collision (rows 1, c_a, c_a^2 - cs^2).
template <class R>
__device__ __forceinline__ void collide7(R f[7], const R heq[7], const R hF[7], const R S[7], R cs2)
{
    R h[7];
    h[0] = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6];
    h[1] = f[1] - f[2];
    h[2] = f[3] - f[4];
    h[3] = f[5] - f[6];
    h[4] = f[1] + f[2] - cs2 * h[0];
    h[5] = f[3] + f[4] - cs2 * h[0];
    h[6] = f[5] + f[6] - cs2 * h[0];
#pragma unroll
    for (int k = 0; k < 7; ++k)
        h[k] = h[k] - S[k] * (h[k] - heq[k]) + (R(1) - R(0.5) * S[k]) * hF[k];
    const R hh = R(0.5), c0 = hh * cs2 * h[0];
    f[0] = (R(1) - R(3) * cs2) * h[0] - h[4] - h[5] - h[6];
    f[1] = c0 + hh * (h[1] + h[4]);
    f[2] = c0 + hh * (-h[1] + h[4]);
    f[3] = c0 + hh * (h[2] + h[5]);
    f[4] = c0 + hh * (-h[2] + h[5]);
    f[5] = c0 + hh * (h[3] + h[6]);
    f[6] = c0 + hh * (-h[3] + h[6]);
}

// The unit-rate collisions (every rate of a non-conserved moment but the
// flow's second-order ones is 1: h* = h - (h - heq) + hF/2 = heq + hF/2,
// Eq. 37).  D3Q7: the result follows from heq and hF alone (moment 0 is phi
// itself); f is only written.
template <class R>
__device__ __forceinline__ void collide7_unit(R f[7], const R heq[7], const R hF[7], R cs2)
{
    R h[7];
    h[0] = heq[0];
#pragma unroll
    for (int k = 1; k < 7; ++k) h[k] = heq[k] + R(0.5) * hF[k];
    const R hh = R(0.5), c0 = hh * cs2 * h[0];
    f[0] = (R(1) - R(3) * cs2) * h[0] - h[4] - h[5] - h[6];
    f[1] = c0 + hh * (h[1] + h[4]);
    f[2] = c0 + hh * (-h[1] + h[4]);
    f[3] = c0 + hh * (h[2] + h[5]);
    f[4] = c0 + hh * (-h[2] + h[5]);
    f[5] = c0 + hh * (h[3] + h[6]);
    f[6] = c0 + hh * (-h[3] + h[6]);
}

// D3Q19 at unit rates s1, s3, s4: moment 0 relaxes at s0 and the second-order
// moments 4-9 at s_2a (diagonal) and s_2b (off-diagonal) of Eq. 35, all from
// f; moments 1-3 and 16-18 at heq + hF/2; 10-15 are zero.
template <class R>
__device__ __forceinline__ void collide19_unit(R f[19], const R heq[19], const R hF[19], R s0, R s2a, R s2b,
                                               R cs2)
{
    R h[19];
    const R m0 = f[0] + f[1] + f[2] + f[3] + f[4] + f[5] + f[6] + f[7] + f[8] + f[9] + f[10] + f[11] + f[12] +
                 f[13] + f[14] + f[15] + f[16] + f[17] + f[18];
    const R exy = f[7] + f[8] + f[9] + f[10], exz = f[11] + f[12] + f[13] + f[14],
            eyz = f[15] + f[16] + f[17] + f[18];
    h[0] = m0 - s0 * m0 + (R(1) - R(0.5) * s0) * hF[0];  // (heq[0] = 0)
    const R d[3] = {f[1] + f[2] + exy + exz - cs2 * m0, f[3] + f[4] + exy + eyz - cs2 * m0,
                    f[5] + f[6] + exz + eyz - cs2 * m0};
    const R o[3] = {f[7] + f[8] - f[9] - f[10], f[11] + f[12] - f[13] - f[14], f[15] + f[16] - f[17] - f[18]};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        h[1 + k] = heq[1 + k] + R(0.5) * hF[1 + k];
        h[4 + k] = d[k] - s2a * (d[k] - heq[4 + k]) + (R(1) - R(0.5) * s2a) * hF[4 + k];
        h[7 + k] = o[k] - s2b * (o[k] - heq[7 + k]) + (R(1) - R(0.5) * s2b) * hF[7 + k];
        h[16 + k] = heq[16 + k] + R(0.5) * hF[16 + k];
    }
#pragma unroll
    for (int k = 10; k < 16; ++k) h[k] = R(0);
    from_hermite19<R>(h, f, cs2);
}

// 1/x: the hardware's approximate reciprocal in FP32 (within 1 ulp; the
// arguments are a density, a bounded 1 - phi0 and rates >= 1/2), the exact
// quotient in FP64 (whose path matches the oracle to 1e-12)
template <class R>
__device__ __forceinline__ R recip(R x)
{
    if constexpr (sizeof(R) == 4) {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
        return r;
    } else {
        return R(1) / x;
    }
}

// a store marked streaming (evict first): the new state is read again only in
// the next step, after the rest of the state has passed through the L2
template <class T>
__device__ __forceinline__ void st_stream(T *p, T v)
{
    if constexpr (sizeof(T) == 2)
        __stcs(reinterpret_cast<unsigned short *>(p), *reinterpret_cast<const unsigned short *>(&v));
    else
        __stcs(p, v);
}

// D3Q19 isotropic stencils (weights 1/18 faces, 1/36 edges, cs^2 = 1/3) on
// three shared-memory planes (below, centre, above) of width W.
template <class R, int W>
__device__ __forceinline__ void grad19(const R *lo, const R *mid, const R *hi, int x, int y, R &gx,
                                       R &gy, R &gz)
{
    auto at = [&](const R *pl, int dx, int dy) { return pl[(y + dy) * W + (x + dx)]; };
    const R f6 = R(1) / R(6), f12 = R(1) / R(12);
    gx = f6 * (at(mid, 1, 0) - at(mid, -1, 0)) +
         f12 * (at(mid, 1, 1) + at(mid, 1, -1) - at(mid, -1, 1) - at(mid, -1, -1) + at(hi, 1, 0) +
                at(lo, 1, 0) - at(hi, -1, 0) - at(lo, -1, 0));
    gy = f6 * (at(mid, 0, 1) - at(mid, 0, -1)) +
         f12 * (at(mid, 1, 1) + at(mid, -1, 1) - at(mid, 1, -1) - at(mid, -1, -1) + at(hi, 0, 1) +
                at(lo, 0, 1) - at(hi, 0, -1) - at(lo, 0, -1));
    gz = f6 * (at(hi, 0, 0) - at(lo, 0, 0)) +
         f12 * (at(hi, 1, 0) + at(hi, -1, 0) + at(hi, 0, 1) + at(hi, 0, -1) - at(lo, 1, 0) -
                at(lo, -1, 0) - at(lo, 0, 1) - at(lo, 0, -1));
}

template <class R, int W>
__device__ __forceinline__ R lap19(const R *lo, const R *mid, const R *hi, int x, int y)
{
    auto at = [&](const R *pl, int dx, int dy) { return pl[(y + dy) * W + (x + dx)]; };
    const R c = at(mid, 0, 0);
    const R faces = at(mid, 1, 0) + at(mid, -1, 0) + at(mid, 0, 1) + at(mid, 0, -1) + at(hi, 0, 0) +
                    at(lo, 0, 0);
    const R edges = at(mid, 1, 1) + at(mid, -1, -1) + at(mid, 1, -1) + at(mid, -1, 1) + at(hi, 1, 0) +
                    at(lo, -1, 0) + at(lo, 1, 0) + at(hi, -1, 0) + at(hi, 0, 1) + at(lo, 0, -1) +
                    at(lo, 0, 1) + at(hi, 0, -1);
    // 6 * (1/18 sum_faces (v - c) + 1/36 sum_edges (v - c))
    return R(1) / R(3) * (faces - R(6) * c) + R(1) / R(6) * (edges - R(12) * c);
}

// Domain and tile coordinates of tile t.  SINGLE: a launch over one domain,
// whose descriptor D1 is a kernel parameter: its sizes, pointers and constants
// are then operands from the constant bank and everything derived from the
// block index is uniform, which frees about forty registers of a thread.
// (build_tiles orders the tiles x, y, z chunk.)
template <bool SINGLE>
__device__ __forceinline__ const DomainDev &tile_of(const StepArgs &A, const DomainDev &D1, int t, int &tx, int &ty, int &tz)
{
    if constexpr (SINGLE) {
        const int r = t / D1.tiles_x;
        tx = t - r * D1.tiles_x;
        tz = r / D1.tiles_y;
        ty = r - tz * D1.tiles_y;
        return D1;
    } else {
        const DomainDev &Dm = A.doms[A.tile_dom[t]];
        const int2 txy = A.tile_xy[t];
        tx = txy.x;
        tz = txy.y / Dm.tiles_y;
        ty = txy.y - tz * Dm.tiles_y;
        return Dm;
    }
}

// the plane of phi of the step under way (k_phi3d)
__device__ __forceinline__ float *phi_of_step(const DomainDev &Dm) { return reinterpret_cast<float *>(Dm.phi0) + Dm.plane; }

// One particle near a tile: its centre as the nearest whole cell i and the rest
// f = fh + fl, |f| <= 1/2, in two parts of the arithmetic type (FP64: fh alone; FP32:
// fh in steps of 2^-16 and fl), f2 = |f|^2.  fast: the whole cells are those of the
// image nearest to the tile, in the tile's coordinates, and serve every cell of its
// frames.  Otherwise (the box is too small for one image, or the frames hold mirror
// rows) they are the domain's, and each cell takes its minimum image from its own
// wrapped coordinates: a table coordinate may lie several lengths of a box narrower
// than the tile from the image.
template <class R>
struct Near3 {
    int i[3], k, own, fast;
    R fh[3], fl[3], f2, Rp, lim2, ct;
    R u[3], w[3];
};

// Indicator of a cell d whole cells from the particle's (offset d - f).  FP32: the
// squared distance is |d|^2 - 2 d.f + f2, where |d|^2 and d.fh are exact (for
// |d| < 128; beyond, far within the result's rounding), their difference carries its
// error and the other terms are small, so it is rounded once, as that of FP64
// arithmetic is, whose pipe (two lanes per SM and clock) stays free.  Three
// placements of three spheres in 96 x 80 x 112: 189, 210 and 226 us per step; with
// plain FP32 sums, an ulp of R off in the distance, 189, 211 and 227.
template <class R>
__device__ __forceinline__ R near_phi0_3d(const Near3<R> &q, const int (&d)[3], R D)
{
    const R x = R(d[0]), y = R(d[1]), z = R(d[2]);
    R r2;
    if constexpr (sizeof(R) == 8) {
        const R rx = x - q.fh[0], ry = y - q.fh[1], rz = z - q.fh[2];
        r2 = rx * rx + ry * ry + rz * rz;
    } else {
        const R whole = __fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)));
        const R dh = __fmaf_rn(z, q.fh[2], __fmaf_rn(y, q.fh[1], __fmul_rn(x, q.fh[0])));
        const R dl = __fmaf_rn(z, q.fl[2], __fmaf_rn(y, q.fl[1], __fmul_rn(x, q.fl[0])));
        // (|d|^2 >= |2 d.fh|: d are whole numbers and |fh| <= 1/2, so err is exact)
        const R s = __fmaf_rn(R(-2), dh, whole);
        const R err = __fmaf_rn(R(-2), dh, whole - s);
        r2 = s + (err + __fmaf_rn(R(-2), dl, q.f2));
    }
    if (r2 >= q.lim2) return R(0);
    return R(0.5) * (R(1) + tanh(R(2) * (q.Rp - sqrt(r2)) / D));
}

// Sums of six values over a warp by halving exchanges: each step a lane keeps
// half of its components and adds its partner's (9 FP64 additions; six shuffle
// trees take 30, and two FP64 lanes per SM and clock made them the force's
// cost).  Lane 4 c holds the sum of component c.
__device__ __forceinline__ double warp_sum6(const double v[6], int lane)
{
    double a[4], b[2];
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double up = i < 2 ? v[4 + i] : 0.0;
        a[i] = (h16 ? up : v[i]) + __shfl_xor_sync(0xffffffffu, h16 ? v[i] : up, 16);
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) b[i] = (h8 ? a[2 + i] : a[i]) + __shfl_xor_sync(0xffffffffu, h8 ? a[i] : a[2 + i], 8);
    double c = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
    c += __shfl_xor_sync(0xffffffffu, c, 2);
    return c + __shfl_xor_sync(0xffffffffu, c, 1);
}

// dynamic shared memory of the particle step: the near particles, each warp's
// force and torque sums, and with own contact angles the W and V plane rings
template <class R, int TX, int TY>
constexpr size_t step3d_moving_smem(int np, bool wv)
{
    return (size_t)np * (sizeof(Near3<R>) + (TX * TY / 32) * 6 * sizeof(double)) +
           (wv ? 2 * 5 * (size_t)(TX + 4) * (TY + 4) * sizeof(R) : 0);
}

// The step of FP64 and of free particles, and every policy's macroscopic pass
// (the FP32-arithmetic step without particles is k_step3d_pair).
// EXT: the instantiation also handles domains with walls at the ends of y
// UNIT: every domain of the launch has unit rates for its non-conserved
// moments: the collisions above.
// MOVING: a tile lists the particles whose indicator reaches its chunk (with
// the image nearest to it), each plane visits those that reach the plane, a
// warp's force terms are summed in FP64 and kept per warp until the chunk ends
// (one barrier per chunk; before, every cell of every frame evaluated every
// particle in FP64 and a barrier followed each particle and plane: 4055 thread
// instructions per cell, one block of 202 registers per SM).  Three spheres in
// 96 x 80 x 112 (FP32): 1240 us per step, 925 with the shorter chunks, 190 to 230 by
// their places now; with the FP64 minimum image per cell kept for boxes below 2 reach
// + tile, 501.  In FP32
// arithmetic phi comes from k_phi3d's plane, as in k_step3d_pair, and the
// domain's descriptor is a kernel parameter.
template <class P, int TX, int TY, bool MOVING, int MODE, bool EXT, bool UNIT = false>
__global__ void __launch_bounds__(TX *TY, (sizeof(typename P::real) == 4 && !MOVING) ? 3 : (MOVING && sizeof(typename P::real) == 4 ? 2 : 1))
    k_step3d(const __grid_constant__ StepArgs A, const __grid_constant__ DomainDev D1)
{
    constexpr bool SINGLE = MOVING && MODE == MODE_STEP;             // (particles: single simulations only)
    constexpr bool PHIT = SINGLE && sizeof(typename P::real) == 4;  // phi from k_phi3d
    using R = typename P::real;
    using ST = typename P::store;
    using AX = typename P::aux;
    constexpr int NT = TX * TY;
    constexpr int FX = TX + 4, FY = TY + 4, FP = FX * FY;  // tile + 2 frame (one plane)
    constexpr int WX = TX + 2, WY = TY + 2, WP = WX * WY;  // tile + 1 frame
    __shared__ R s_phi[5][FP];
    __shared__ R s_p0[5][FP];
    __shared__ R s_mu[4][WP];
    __shared__ R s_T[4][3][WP];
    __shared__ int s_gx[TX + 6];
    __shared__ int s_gy[TY + 6];   // wrapped row offsets y * pitch
    __shared__ int s_gyi[TY + 6];  // wrapped rows
    __shared__ int s_out[EXT ? TY + 6 : 1];  // walls: the row lies beyond a wall (mirror image)
    __shared__ int s_nn;                     // near particles of the tile
    // MOVING: the near particles, each warp's sums of force and torque, then with
    // A.wv W and V of every staged phi0 plane (the same ring of 5)
    extern __shared__ __align__(16) unsigned char s_dyn3d[];
    constexpr int NW = NT / 32;
    double *const s_facc = reinterpret_cast<double *>(s_dyn3d);  // [near particle][warp][6]
    Near3<R> *const s_near = reinterpret_cast<Near3<R> *>(s_facc + (MOVING ? A.np * NW * 6 : 0));
    R *const s_W = reinterpret_cast<R *>(s_near + (MOVING ? A.np : 0));
    R *const s_V = s_W + 5 * FP;

    const int tid = threadIdx.x;
    const int lx = tid % TX, ly = tid / TX;
    // a step that timed out (bit 2) leaves no fields to read: nothing is written
    [[maybe_unused]] int lost = 0;
    if constexpr (MODE == MODE_MACROS) lost = *A.flags & 4;

    for (int t = blockIdx.x; t < A.ntiles; t += gridDim.x) {
        int tx, ty, tz;
        const DomainDev &Dm = tile_of<SINGLE>(A, D1, t, tx, ty, tz);
        const int nx = Dm.nx, ny = Dm.ny, nz = Dm.nz;
        const int plane = (int)Dm.plane;  // 26 * plane < 2^31 (checked at create)
        const int zstride = Dm.pitch * ny;
        const int x0 = tx * TX;
        const int y0 = ty * TY;
        const int zc = Dm.zc;
        const int z0 = tz * zc;
        const DevParams &p = Dm.p;
        const KParams<R> &kp = kparams<R>(Dm);

        __syncthreads();
        const int wall = EXT ? Dm.wall_y : 0;
        for (int k = tid; k < TX + 6; k += NT) s_gx[k] = wrap_idx(x0 - 3 + k, nx);
        for (int k = tid; k < TY + 6; k += NT) {
            if constexpr (EXT) {
                const int y = y0 - 3 + k;
                int yy, out = 0;
                if (wall) {
                    // rows beyond a wall read their mirror image (clamped: the
                    // rows that far out only feed cells beyond the domain)
                    yy = y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
                    out = y < 0 || y >= ny;
                    yy = min(max(yy, 0), ny - 1);
                } else {
                    yy = wrap_idx(y, ny);
                }
                s_gyi[k] = yy;
                s_gy[k] = yy * Dm.pitch;
                s_out[k] = out;
            } else {
                const int yy = wrap_idx(y0 - 3 + k, ny);
                s_gyi[k] = yy;
                s_gy[k] = yy * Dm.pitch;
            }
        }
        __syncthreads();
        if constexpr (MOVING) {
            // the particles whose reach meets the box of the tile's frames and
            // planes (minimum image, conservative by a cell), in their order
            if (tid < 32) {
                int n = 0;
                for (int k0 = 0; k0 < A.np; k0 += 32) {
                    const int k = k0 + tid;
                    bool hit = false;
                    Near3<R> q;
                    if (k < A.np) {
                        const ParticleDev &pp = A.parts[k];
                        const double mid[3] = {x0 + 0.5 * (TX - 1), y0 + 0.5 * (TY - 1), z0 + 0.5 * (zc - 1)};
                        const double ext[3] = {0.5 * TX + 2.0, 0.5 * TY + 2.0, 0.5 * zc + 2.0};
                        const int n3[3] = {nx, ny, nz}, len[3] = {TX, TY, zc};
                        const double reach = pp.R + indicator_cut<R>(p);
                        double e2 = 0.0, f2 = 0.0, cell[3];
                        bool fast = true;
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            double dd = mid[a] - pp.x[a];
                            const bool bounded = a == 1 && wall;
                            // the image nearest to the tile is `shift` box lengths away
                            const double shift = bounded ? 0.0 : n3[a] * rint(dd / n3[a]);
                            dd -= shift;
                            const double ex = fmax(fabs(dd) - ext[a], 0.0);
                            e2 += ex * ex;
                            const double whole = rint(pp.x[a]), f = pp.x[a] - whole;
                            cell[a] = whole + shift;
                            f2 += f * f;
                            q.fh[a] = sizeof(R) == 8 ? (R)f : (R)(rint(f * 65536.0) / 65536.0);
                            q.fl[a] = (R)(f - (double)q.fh[a]);
                            // with walls rows beyond them are mirror rows: their cells are not
                            // where the table says
                            fast = fast && (bounded ? !(y0 - 3 < 0 || y0 + TY + 3 > ny) : n3[a] >= 2.0 * reach + 6.0 + len[a]);
                        }
                        hit = e2 < (reach + 1.0) * (reach + 1.0);
                        const int at[3] = {x0, y0, z0};
#pragma unroll
                        for (int a = 0; a < 3; ++a)
                            q.i[a] = fast ? (int)cell[a] - at[a]
                                          : (a == 1 && wall ? (int)cell[a] : wrap_idx((int)cell[a], n3[a]));
                        q.f2 = (R)f2;
                        q.k = k;
                        q.own = pp.own;
                        q.fast = fast;
                        q.Rp = (R)pp.R;
                        q.lim2 = (R)(reach * reach);
                        q.ct = pp.own ? (R)pp.ct : R(0);
#pragma unroll
                        for (int a = 0; a < 3; ++a) {
                            q.u[a] = (R)pp.u[a];
                            q.w[a] = (R)pp.w[a];
                        }
                    }
                    const unsigned m = __ballot_sync(0xffffffffu, hit);
                    if (hit) s_near[n + __popc(m & ((1u << tid) - 1u))] = q;
                    n += __popc(m);
                }
                if (tid == 0) s_nn = n;
            }
            for (int q = tid; q < A.np * NW * 6; q += NT) s_facc[q] = 0.0;
            __syncthreads();
        }
        [[maybe_unused]] const int nn = MOVING ? s_nn : 0;
        // whole cells d of an offset d - f within the domain (component a of particle q):
        // those of its minimum image (min_image's rule; |d| < n, so one shift reaches it)
        [[maybe_unused]] auto wrapped = [](const Near3<R> &q, int a, int d, int n) -> int {
            const R fh2 = R(2) * q.fh[a], fl2 = R(2) * q.fl[a];  // (exact, as the differences are)
            if (R(2 * d - n) - fh2 > fl2) return d - n;
            if (R(2 * d + n) - fh2 < fl2) return d + n;
            return d;
        };
        // whole cells of the offset of plane z (of the chunk's run z0 - 2 ..) to particle q
        [[maybe_unused]] auto near_z = [&](const Near3<R> &q, int z) -> int {
            return q.fast ? z - z0 - q.i[2] : wrapped(q, 2, wrap_near(z, nz) - q.i[2], nz);
        };
        // offset of cell (table cx, cy of the tile + 3 frame, plane z) to near particle q,
        // rounded once, and its indicator there
        [[maybe_unused]] auto near_at = [&](const Near3<R> &q, int cx, int cy, int z, R &rx, R &ry, R &rz) -> R {
            int d[3];
            d[2] = near_z(q, z);
            if (q.fast) {
                d[0] = cx - 3 - q.i[0];
                d[1] = cy - 3 - q.i[1];
            } else {
                d[0] = wrapped(q, 0, s_gx[cx] - q.i[0], nx);
                d[1] = s_gyi[cy] - q.i[1];  // (no image across a wall)
                if (!(EXT && wall)) d[1] = wrapped(q, 1, d[1], ny);
            }
            rx = (R(d[0]) - q.fh[0]) - q.fl[0];
            ry = (R(d[1]) - q.fh[1]) - q.fl[1];
            rz = (R(d[2]) - q.fh[2]) - q.fl[2];
            return near_phi0_3d<R>(q, d, (R)p.D);
        };
        // whether near particle q may reach plane z (uniform)
        [[maybe_unused]] auto meets = [&](const Near3<R> &q, int z) -> bool {
            const R dz = (R(near_z(q, z)) - q.fh[2]) - q.fl[2];
            return dz * dz < q.lim2;
        };
        // a tile whose frames reach beyond a wall
        const bool wall_tile = EXT && wall && (y0 - 3 < 0 || y0 + TY + 3 > ny);
        // sign of the y-odd products T_xy, T_yz at table row r under a wall mirror
        auto wsign = [&](int r) -> R {
            if constexpr (EXT) return s_out[r] ? R(-1) : R(1);
            return R(1);
        };

        const ST *fs = reinterpret_cast<const ST *>(Dm.f[A.par]);
        ST *fd = reinterpret_cast<ST *>(Dm.f[A.par ^ 1]);
        const AX *as = reinterpret_cast<const AX *>(Dm.aux[A.par]);
        AX *ad = reinterpret_cast<AX *>(Dm.aux[A.par ^ 1]);
        const AX *ph0 = reinterpret_cast<const AX *>(Dm.phi0);
        const long long *rs = reinterpret_cast<const long long *>(Dm.rest[A.par]);
        long long *rd = reinterpret_cast<long long *>(Dm.rest[A.par ^ 1]);
        const R isc1 = kp.inv_scale[0], isc2 = kp.inv_scale[1];
        const R c_dw = kp.c_dw, c_lap = kp.c_lap, c_pen = kp.c_pen, c_wet = kp.c_wet,
                c_wlap = kp.c_wlap;

        // the planes touched lie in [z0 - 3, min(z0 + zc, nz) + 2], inside
        // [-nz, 2 nz) since nz >= 4
        auto zoff = [&](int z) { return wrap_near(z, nz) * zstride; };
        auto cidx = [&](int tx_, int ty_, int zo) {  // tile+3 table coordinates
            return zo + s_gy[ty_] + s_gx[tx_];
        };
        // offset of the population that table cell (cx, cy) of plane z pulls as
        // direction i of the lattice starting at plane `base`: from cell - c_i,
        // or, where that lies beyond a wall, its own opposite population
        // (halfway bounce-back)
        auto pull = [&](int base, int i, int cx, int cy, int z) -> int {
            if constexpr (EXT) {
                if (wall_tile && s_out[cy - C19Y[i]] && !s_out[cy])
                    return (base + opp19(i)) * plane + cidx(cx, cy, zoff(z));
            }
            return base * plane + i * plane + cidx(cx - C19X[i], cy - C19Y[i], zoff(z - C19Z[i]));
        };
        // phi at (frame x, frame y) of plane z: pull and sum the D3Q7 populations
        auto phi_at = [&](int hx, int hy, int z, R *keep, ST *keepq) -> R {
            const int cx = hx + 1, cy = hy + 1;
            R acc;
            if constexpr (PHIT) {
                acc = phi_of_step(Dm)[cidx(cx, cy, zoff(z))];
                if constexpr (!UNIT) {
                    if (keep) {
                        // (the rest population does not enter the collision's moments
                        // beyond phi: keep[0] is set by the caller)
#pragma unroll
                        for (int i = P::MIX ? 1 : 0; i < 7; ++i) {
                            const ST qv = ldg(fs + pull(0, i, cx, cy, z));
                            keep[i] = Conv<P>::ld(qv, isc1);
                            if (keepq) keepq[i] = qv;
                        }
                    }
                }
            } else if constexpr (P::MIX) {
                acc = float_of_fixed(rs[cidx(cx, cy, zoff(z))]);
                if (keep) keep[0] = acc;
#pragma unroll
                for (int i = 1; i < 7; ++i) {
                    const ST qv = ldg(fs + pull(0, i, cx, cy, z));
                    const R v = Conv<P>::ld(qv, isc1);
                    if (keep) keep[i] = v;
                    if (keepq) keepq[i] = qv;
                    acc += v;
                }
            } else {
                acc = R(0);
#pragma unroll
                for (int i = 0; i < 7; ++i) {
                    const R v = Conv<P>::ld(ldg(fs + pull(0, i, cx, cy, z)), isc1);
                    if (keep) keep[i] = v;
                    acc += v;
                }
            }
            return acc;
        };
        // total indicator at (frame x, frame y) of plane z; with own particle
        // angles (Wo set) also W = sum_s cos(theta_s) phi0_s and V = sum_s
        // cos(theta_s) phi0_s^3, every solid without an own angle counted as one
        auto phi0_at = [&](int hx, int hy, int z, R *Wo, R *Vo) -> R {
            const int cx = hx + 1, cy = hy + 1;
            R v = (R)ldg(ph0 + cidx(cx, cy, zoff(z)));
            if constexpr (MOVING) {
                R dflt = v, w = R(0), vv = R(0);
                for (int j = 0; j < nn; ++j) {
                    const Near3<R> &q = s_near[j];
                    if (!meets(q, z)) continue;
                    R rx, ry, rz;
                    const R pk = near_at(q, cx, cy, z, rx, ry, rz);
                    v += pk;
                    if (Wo) {
                        if (q.own) {
                            w += q.ct * pk;
                            vv += q.ct * pk * pk * pk;
                        } else {
                            dflt += pk;
                        }
                    }
                }
                if (Wo) {
                    const R ct = (R)p.cos_t;
                    *Wo = ct * dflt + w;
                    *Vo = ct * dflt * dflt * dflt + vv;
                }
            }
            return v;
        };
        auto load_phi_plane = [&](int z) {
            const int slot = wrap_idx(z, 5);
            for (int r = tid; r < FP; r += NT) {
                const int hx = r % FX, hy = r / FX;
                s_phi[slot][r] = phi_at(hx, hy, z, nullptr, nullptr);
                if (MOVING && A.wv)
                    s_p0[slot][r] = phi0_at(hx, hy, z, s_W + slot * FP + r, s_V + slot * FP + r);
                else
                    s_p0[slot][r] = phi0_at(hx, hy, z, nullptr, nullptr);
            }
        };
        auto load_T_plane = [&](int z) {
            const int slot = wrap_idx(z, 4);
            const int zo = zoff(z);
            for (int r = tid; r < WP; r += NT) {
                const int wx = r % WX, wy = r / WX;
                const int id = cidx(wx + 2, wy + 2, zo);
                const R ux = (R)ldg(as + 0 * plane + id), uy = (R)ldg(as + 1 * plane + id),
                        uz = (R)ldg(as + 2 * plane + id);
                const R Sx = (R)ldg(as + 3 * plane + id), Sy = (R)ldg(as + 4 * plane + id),
                        Sz = (R)ldg(as + 5 * plane + id);
                const R sg = wsign(wy + 2);  // T_xy and T_yz are odd under the wall mirror
                s_T[slot][0][r] = sg * (Sx * uy - ux * Sy);
                s_T[slot][1][r] = Sx * uz - ux * Sz;
                s_T[slot][2][r] = sg * (Sy * uz - uy * Sz);
            }
        };
        auto mu_plane = [&](int z) {
            const int slot = wrap_idx(z, 4);
            const R *lo = s_phi[wrap_idx(z - 1, 5)], *mid = s_phi[wrap_idx(z, 5)], *hi = s_phi[wrap_idx(z + 1, 5)];
            const R *lo0 = s_p0[wrap_idx(z - 1, 5)], *mid0 = s_p0[wrap_idx(z, 5)], *hi0 = s_p0[wrap_idx(z + 1, 5)];
            for (int r = tid; r < WP; r += NT) {
                const int hx = r % WX + 1, hy = r / WX + 1;
                const R ph = mid[hy * FX + hx], p0 = mid0[hy * FX + hx];
                const R lp = lap19<R, FX>(lo, mid, hi, hx, hy);
                if (MOVING && A.wv) {
                    // wetting summed per solid (own particle angles), through W and V
                    const R *Wl = s_W + wrap_idx(z - 1, 5) * FP, *Wm = s_W + wrap_idx(z, 5) * FP,
                            *Wh = s_W + wrap_idx(z + 1, 5) * FP;
                    const R Wv = Wm[hy * FX + hx], Vv = s_V[wrap_idx(z, 5) * FP + hy * FX + hx];
                    s_mu[slot][r] = c_dw * ph * (ph - R(1)) * (ph + R(1)) - c_lap * lp + c_pen * p0 * p0 * ph +
                                    c_dw * (R(3) * ph * ph * Wv + Vv - Wv) - c_lap * lap19<R, FX>(Wl, Wm, Wh, hx, hy);
                    continue;
                }
                const R lp0 = lap19<R, FX>(lo0, mid0, hi0, hx, hy);
                s_mu[slot][r] = c_dw * ph * (ph - R(1)) * (ph + R(1)) - c_lap * lp + c_pen * p0 * p0 * ph +
                                c_wet * p0 * (R(3) * ph * ph + p0 * p0 - R(1)) - c_wlap * lp0;
            }
        };

        // walls: phi beyond a wall is the mirror image of phi inside (no flux);
        // refills the rows of plane z's slot beyond the wall (after a barrier)
        auto mirror_phi_plane = [&](int z) {
            if constexpr (EXT) {
                const int slot = wrap_idx(z, 5);
                for (int r = tid; r < FP; r += NT) {
                    const int hx = r % FX, hy = r / FX;
                    if (!s_out[hy + 1]) continue;
                    const int y = y0 - 2 + hy;
                    const int hym = (y < 0 ? -1 - y : 2 * ny - 1 - y) - (y0 - 2);
                    if (hym >= 0 && hym < FY && !s_out[hym + 1]) s_phi[slot][r] = s_phi[slot][hym * FX + hx];
                }
            }
        };

        // prologue: phi planes z0-2 .. z0+1, T planes z0-1, z0, mu planes z0-1, z0
        for (int z = z0 - 2; z <= z0 + 1; ++z) load_phi_plane(z);
        if constexpr (MODE == MODE_STEP) {
            load_T_plane(z0 - 1);
            load_T_plane(z0);
        }
        __syncthreads();
        if (!PHIT && wall_tile) {  // (k_phi3d's plane is read at the mirror rows themselves)
            for (int z = z0 - 2; z <= z0 + 1; ++z) mirror_phi_plane(z);
            __syncthreads();
        }
        mu_plane(z0 - 1);
        mu_plane(z0);
        __syncthreads();

        const int zend = min(z0 + zc, nz);
        for (int z = z0; z < zend; ++z) {
            // phase 1: phi plane z+2 and T plane z+1
            load_phi_plane(z + 2);
            if constexpr (MODE == MODE_STEP) load_T_plane(z + 1);
            __syncthreads();
            if (!PHIT && wall_tile) {
                mirror_phi_plane(z + 2);
                __syncthreads();
            }
            // phase 2: mu plane z+1
            mu_plane(z + 1);
            __syncthreads();

            // phase 3: own cell of plane z
            const int gx = x0 + lx, gy = y0 + ly;
            const bool valid = gx < nx && gy < ny;
            const int zo = zoff(z);
            const int id = cidx(lx + 3, ly + 3, zo);
            const int hx = lx + 2, hy = ly + 2, wxy = (ly + 1) * WX + (lx + 1);
            const R *plo = s_phi[wrap_idx(z - 1, 5)], *pmid = s_phi[wrap_idx(z, 5)], *phi_hi = s_phi[wrap_idx(z + 1, 5)];
            const R *mlo = s_mu[wrap_idx(z - 1, 4)], *mmid = s_mu[wrap_idx(z, 4)], *mhi = s_mu[wrap_idx(z + 1, 4)];

            R f1[7];
            ST q1[7];
            const R phi = phi_at(hx, hy, z, f1, q1);
            // PHIT, 16-bit: k_phi3d left the exact phi where the rest population was
            [[maybe_unused]] int sold = 0;
            if constexpr (P::MIX && !(PHIT && UNIT)) {
#pragma unroll
                for (int i = 1; i < 7; ++i) sold += fix24_stored<ST>(q1[i]);
                if constexpr (PHIT) f1[0] = float_of_fixed(rs[id] - fix24_to_rest(sold, p.klog2[0]));
            }
            const R phi0 = s_p0[wrap_idx(z, 5)][hy * FX + hx];
            R gpx, gpy, gpz, gmx, gmy, gmz;
            grad19<R, FX>(plo, pmid, phi_hi, hx, hy, gpx, gpy, gpz);
            grad19<R, WX>(mlo, mmid, mhi, lx + 1, ly + 1, gmx, gmy, gmz);
            const R mu = mmid[wxy];
            const R drho = kp.drho;
            const R rho = drho * phi + kp.rhom;
            const R muv = kp.dmu * phi + kp.mum;
            // conservative Allen-Cahn option: theta n = (2/D)(1 - phi^2) grad phi/|grad phi|
            // and the mass flux M (rho1 - rho2)/2 (grad phi - theta n)
            const bool cac = Dm.p.phase_model == 1;
            R tnx = R(0), tny = R(0), tnz = R(0);
            if (cac) {
                const R g2 = gpx * gpx + gpy * gpy + gpz * gpz;
                const R th = kp.two_over_D * (R(1) - phi * phi);
                const R inv = g2 > R(1e-24) ? R(1) / sqrt(g2) : R(0);
                tnx = th * gpx * inv;
                tny = th * gpy * inv;
                tnz = th * gpz * inv;
            }
            const R Sx = cac ? kp.Mdrho * (gpx - tnx) : kp.Mdrho * gmx;
            const R Sy = cac ? kp.Mdrho * (gpy - tny) : kp.Mdrho * gmy;
            const R Sz = cac ? kp.Mdrho * (gpz - tnz) : kp.Mdrho * gmz;
            const R grx = drho * gpx, gry = drho * gpy, grz = drho * gpz;
            R Fx = mu * gpx + kp.Fb[0], Fy = mu * gpy + kp.Fb[1], Fz = mu * gpz + kp.Fb[2];
            if constexpr (MODE == MODE_STEP) {
                // F_c,b = 1/2 sum_a d_a T_ab with T antisymmetric (previous step)
                const int s0_ = wrap_idx(z - 1, 4), s1_ = wrap_idx(z, 4), s2_ = wrap_idx(z + 1, 4);
                R axy, ayx, azx, axz, ayz, azy, dummy;
                // d/dx, d/dy, d/dz of T_xy
                grad19<R, WX>(s_T[s0_][0], s_T[s1_][0], s_T[s2_][0], lx + 1, ly + 1, axy, ayx, azx);
                R bx, by, bz;
                grad19<R, WX>(s_T[s0_][1], s_T[s1_][1], s_T[s2_][1], lx + 1, ly + 1, bx, by, bz);
                R cx_, cy_, cz_;
                grad19<R, WX>(s_T[s0_][2], s_T[s1_][2], s_T[s2_][2], lx + 1, ly + 1, cx_, cy_, cz_);
                (void)azx;
                (void)by;
                (void)cx_;
                (void)dummy;
                (void)axz;
                (void)ayz;
                (void)azy;
                Fx += R(0.5) * (-ayx - bz);   // -d_y T_xy - d_z T_xz
                Fy += R(0.5) * (axy - cz_);   //  d_x T_xy - d_z T_yz
                Fz += R(0.5) * (bx + cy_);    //  d_x T_xz + d_y T_yz
            } else {
                // macroscopic pass: F_c from the lagged fields read directly
                R T[3][3][3][3];
#pragma unroll
                for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
                    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
                        for (int dx = -1; dx <= 1; ++dx) {
                            const int nid = cidx(lx + 3 + dx, ly + 3 + dy, zoff(z + dz));
                            const R ux = (R)ldg(as + 0 * plane + nid), uy = (R)ldg(as + 1 * plane + nid),
                                    uz = (R)ldg(as + 2 * plane + nid);
                            const R sx = (R)ldg(as + 3 * plane + nid), sy = (R)ldg(as + 4 * plane + nid),
                                    sz = (R)ldg(as + 5 * plane + nid);
                            const R sg = wsign(ly + 3 + dy);
                            T[0][dz + 1][dy + 1][dx + 1] = sg * (sx * uy - ux * sy);
                            T[1][dz + 1][dy + 1][dx + 1] = sx * uz - ux * sz;
                            T[2][dz + 1][dy + 1][dx + 1] = sg * (sy * uz - uy * sz);
                        }
                R g[3][3];
#pragma unroll
                for (int c = 0; c < 3; ++c)
                    grad19<R, 3>(&T[c][0][0][0], &T[c][1][0][0], &T[c][2][0][0], 1, 1, g[c][0], g[c][1], g[c][2]);
                Fx += R(0.5) * (-g[0][1] - g[1][2]);
                Fy += R(0.5) * (g[0][0] - g[2][2]);
                Fz += R(0.5) * (g[1][0] + g[2][1]);
            }
            if constexpr (MOVING) {
                const R lphi = lap19<R, FX>(plo, pmid, phi_hi, hx, hy);
                R g0x, g0y, g0z;
                grad19<R, FX>(s_p0[wrap_idx(z - 1, 5)], s_p0[wrap_idx(z, 5)], s_p0[wrap_idx(z + 1, 5)], hx, hy,
                              g0x, g0y, g0z);
                if (A.wv) {
                    // sum over solids of mu_phi0,s grad phi0_s with their own angles
                    const int s0w = wrap_idx(z - 1, 5) * FP, s1w = wrap_idx(z, 5) * FP, s2w = wrap_idx(z + 1, 5) * FP;
                    R gWx, gWy, gWz, gVx, gVy, gVz;
                    grad19<R, FX>(s_W + s0w, s_W + s1w, s_W + s2w, hx, hy, gWx, gWy, gWz);
                    grad19<R, FX>(s_V + s0w, s_V + s1w, s_V + s2w, hx, hy, gVx, gVy, gVz);
                    const R pen = c_pen * phi0 * phi * phi;
                    const R aW = c_dw * phi * (phi * phi - R(1)) - c_lap * lphi, aV = c_dw * phi;
                    Fx += pen * g0x + aW * gWx + aV * gVx;
                    Fy += pen * g0y + aW * gWy + aV * gVy;
                    Fz += pen * g0z + aW * gWz + aV * gVz;
                } else {
                    const R mu0 = c_pen * phi0 * phi * phi +
                                  c_wet * phi * (R(3) * phi0 * phi0 + phi * phi - R(1)) - c_wlap * lphi;
                    Fx += mu0 * g0x;
                    Fy += mu0 * g0y;
                    Fz += mu0 * g0z;
                }
            }

            R f2[19];
#pragma unroll
            for (int i = 0; i < 19; ++i)
                f2[i] = Conv<P>::ld(ldg(fs + pull(7, i, lx + 3, ly + 3, z)), isc2);
            R jx = R(0), jy = R(0), jz = R(0), sum_f = R(0);
#pragma unroll
            for (int i = 1; i < 19; ++i) {
                jx += (R)C19X[i] * f2[i];
                jy += (R)C19Y[i] * f2[i];
                jz += (R)C19Z[i] * f2[i];
                sum_f += f2[i];
            }
            const R irho = recip(rho);
            const R usx = (jx + R(0.5) * Fx) * irho, usy = (jy + R(0.5) * Fy) * irho,
                    usz = (jz + R(0.5) * Fz) * irho;
            R fpx = -phi0 * usx, fpy = -phi0 * usy, fpz = -phi0 * usz;
            if constexpr (MOVING) {
                // the solids' velocity in the penalty force, and the hydrodynamic
                // force and torque on each particle (Eq. 27): F = -sum rho phi0_k
                // (u_s - u*), T = -sum r x (...), summed per warp in FP64
                for (int j = 0; j < nn; ++j) {
                    const Near3<R> &q = s_near[j];
                    if (!meets(q, z)) continue;
                    R rx, ry, rz;
                    const R pk = near_at(q, lx + 3, ly + 3, z, rx, ry, rz);
                    R vx = R(0), vy = R(0), vz = R(0);
                    if (pk != R(0)) {
                        vx = q.u[0] + q.w[1] * rz - q.w[2] * ry;
                        vy = q.u[1] + q.w[2] * rx - q.w[0] * rz;
                        vz = q.u[2] + q.w[0] * ry - q.w[1] * rx;
                        fpx += pk * vx;
                        fpy += pk * vy;
                        fpz += pk * vz;
                    }
                    if constexpr (MODE == MODE_STEP) {
                        const bool hit = valid && pk != R(0);
                        if (!__any_sync(0xffffffffu, hit)) continue;
                        double c6[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
                        if (hit) {
                            const double fx = (double)(rho * pk * (vx - usx)), fy = (double)(rho * pk * (vy - usy)),
                                         fz = (double)(rho * pk * (vz - usz));
                            c6[0] = -fx;
                            c6[1] = -fy;
                            c6[2] = -fz;
                            c6[3] = -((double)ry * fz - (double)rz * fy);
                            c6[4] = -((double)rz * fx - (double)rx * fz);
                            c6[5] = -((double)rx * fy - (double)ry * fx);
                        }
                        const double sum = warp_sum6(c6, tid & 31);
                        const int comp = (tid & 31) >> 2;
                        if ((tid & 3) == 0 && comp < 6) s_facc[(j * NW + (tid >> 5)) * 6 + comp] += sum;
                    }
                }
            }
            const R ux = usx + R(0.5) * fpx, uy = usy + R(0.5) * fpy, uz = usz + R(0.5) * fpz;
            const R Ftx = Fx + rho * fpx, Fty = Fy + rho * fpy, Ftz = Fz + rho * fpz;
            const R upx = (R)ldg(as + 0 * plane + id),
                    upy = (R)ldg(as + 1 * plane + id),
                    upz = (R)ldg(as + 2 * plane + id);
            const R Spx = (R)ldg(as + 3 * plane + id),
                    Spy = (R)ldg(as + 4 * plane + id),
                    Spz = (R)ldg(as + 5 * plane + id);
            const R php = (R)ldg(as + 6 * plane + id);

            R solid = R(1) - phi0;
            const R seps = kp.solid_eps;
            solid = solid < seps ? seps : solid;
            R nu;
            if constexpr (sizeof(R) == 4)
                nu = muv * irho * recip(solid);
            else
                nu = muv / (rho * solid);
            const R inv_s2a = R(0.5) + kp.two_over_1md0 * nu;
            const R inv_s2b = R(0.5) + kp.inv_cs2 * nu;
            const R Kf = kp.K;
            const R H = Kf * (kp.Hc0 - kp.Hc1 * inv_s2a);
            const R ugr = ux * grx + uy * gry + uz * grz;
            const R rus_u = (rho * ux - Sx) * ux + (rho * uy - Sy) * uy + (rho * uz - Sz) * uz;
            const R Su = Sx * ux + Sy * uy + Sz * uz, Sup = Spx * upx + Spy * upy + Spz * upz;
            const R dt_term = R(2) * (ux * Ftx + uy * Fty + uz * Ftz) - (Su - Sup);
            const R Pr = kp.Pfac * (sum_f + (R(0.5) + H) * ugr - kp.w0f * rus_u * kp.inv_1mcs2 +
                                      Kf * R(0.5) * dt_term);

            if constexpr (MODE == MODE_MACROS) {
                if (valid && !lost) {
                    const long long N = (long long)nx * ny * nz;
                    const long long o = ((long long)z * ny + gy) * nx + gx;
                    double phv = (double)phi;
                    if constexpr (P::MIX) phv = double_of_fixed(rs[id] + fix24_to_rest(sold, p.klog2[0]));
                    const MacroOut mo = A.mouts ? A.mouts[A.tile_dom[t]] : A.mout;
                    if (mo.phi) mo.phi[o] = phv;
                    if (mo.rho) mo.rho[o] = (double)rho;
                    if (mo.u) mo.u[o] = (double)ux;
                    if (mo.u) mo.u[N + o] = (double)uy;
                    if (mo.u) mo.u[2 * N + o] = (double)uz;
                    if (mo.P) mo.P[o] = (double)Pr;
                    if (mo.mu) mo.mu[o] = (double)mu;
                    if (mo.phi0) mo.phi0[o] = (double)phi0;
                    if (MOVING && A.wv) {
                        if (mo.W) mo.W[o] = (double)s_W[wrap_idx(z, 5) * FP + hy * FX + hx];
                        if (mo.V) mo.V[o] = (double)s_V[wrap_idx(z, 5) * FP + hy * FX + hx];
                    }
                }
                continue;
            } else {
                const R cs2 = kp.cs2, cs4 = kp.cs4;
                // order-parameter lattice (D3Q7)
                const R em = cac ? phi : kp.eta * mu;  // Allen-Cahn: eta mu -> phi
                {
                    R heq[7], hF[7], S[7];
                    heq[0] = phi;
                    heq[1] = phi * ux;
                    heq[2] = phi * uy;
                    heq[3] = phi * uz;
                    heq[4] = heq[5] = heq[6] = cs2 * (em - phi);
                    hF[0] = R(0);
                    hF[1] = phi * ux - php * upx;
                    hF[2] = phi * uy - php * upy;
                    hF[3] = phi * uz - php * upz;
                    if (cac) {
                        hF[1] += cs2 * tnx;
                        hF[2] += cs2 * tny;
                        hF[3] += cs2 * tnz;
                    }
                    hF[4] = hF[5] = hF[6] = R(0);
                    if constexpr (UNIT) {
                        collide7_unit<R>(f1, heq, hF, cs2);
                    } else {
                        S[0] = kp.s0;
                        S[1] = S[2] = S[3] = kp.s1phi;
                        S[4] = S[5] = S[6] = kp.s2;
                        collide7<R>(f1, heq, hF, S, cs2);
                    }
                }
                // flow lattice (D3Q19)
                {
                    R heq[19], hF[19], S[19];
                    const R Xx = rho * ux * ux - Sx * ux, Xy = rho * uy * uy - Sy * uy, Xz = rho * uz * uz - Sz * uz;
                    const R c4r = cs4 * kp.inv_1mcs2;
                    heq[0] = R(0);
                    heq[1] = rho * ux;
                    heq[2] = rho * uy;
                    heq[3] = rho * uz;
                    heq[4] = Pr + Xx;
                    heq[5] = Pr + Xy;
                    heq[6] = Pr + Xz;
                    heq[7] = rho * ux * uy - R(0.5) * (Sx * uy + ux * Sy);
                    heq[8] = rho * ux * uz - R(0.5) * (Sx * uz + ux * Sz);
                    heq[9] = rho * uy * uz - R(0.5) * (Sy * uz + uy * Sz);
#pragma unroll
                    for (int k = 10; k < 16; ++k) heq[k] = R(0);
                    heq[16] = -cs2 * Pr - c4r * Xz;
                    heq[17] = -cs2 * Pr - c4r * Xy;
                    heq[18] = -cs2 * Pr - c4r * Xx;
                    const R c3 = R(1) - R(3) * cs2;
                    const R Mxx = R(2) * ux * Ftx - (Sx * ux - Spx * upx) + R(2) * cs2 * ux * grx + c3 * ugr;
                    const R Myy = R(2) * uy * Fty - (Sy * uy - Spy * upy) + R(2) * cs2 * uy * gry + c3 * ugr;
                    const R Mzz = R(2) * uz * Ftz - (Sz * uz - Spz * upz) + R(2) * cs2 * uz * grz + c3 * ugr;
                    const R Mxy = ux * Fty + Ftx * uy - R(0.5) * ((Sx * uy + ux * Sy) - (Spx * upy + upx * Spy)) +
                                  cs2 * (ux * gry + grx * uy);
                    const R Mxz = ux * Ftz + Ftx * uz - R(0.5) * ((Sx * uz + ux * Sz) - (Spx * upz + upx * Spz)) +
                                  cs2 * (ux * grz + grx * uz);
                    const R Myz = uy * Ftz + Fty * uz - R(0.5) * ((Sy * uz + uy * Sz) - (Spy * upz + upy * Spz)) +
                                  cs2 * (uy * grz + gry * uz);
                    hF[0] = ugr;
                    hF[1] = Ftx;
                    hF[2] = Fty;
                    hF[3] = Ftz;
                    hF[4] = Mxx;
                    hF[5] = Myy;
                    hF[6] = Mzz;
                    hF[7] = Mxy;
                    hF[8] = Mxz;
                    hF[9] = Myz;
#pragma unroll
                    for (int k = 10; k < 16; ++k) hF[k] = R(0);
                    hF[16] = -c4r * Mzz;
                    hF[17] = -c4r * Myy;
                    hF[18] = -c4r * Mxx;
                    const R s2a = recip(inv_s2a), s2b = recip(inv_s2b);
                    if constexpr (UNIT) {
                        collide19_unit<R>(f2, heq, hF, kp.s0, s2a, s2b, cs2);
                    } else {
                        S[0] = kp.s0;
                        S[1] = S[2] = S[3] = kp.s1;
                        S[4] = S[5] = S[6] = s2a;
                        S[7] = S[8] = S[9] = s2b;
#pragma unroll
                        for (int k = 10; k < 16; ++k) S[k] = kp.s3;
                        S[16] = S[17] = S[18] = kp.s4;
                        collide19<R>(f2, heq, hF, S, cs2);
                    }
                }
                if (valid) {
                    if constexpr (P::MIX) {
                        const R sc1 = kp.scale[0];
                        const int k1 = p.klog2[0];
                        int bad = 0, snew = 0;
#pragma unroll
                        for (int i = 1; i < 7; ++i) {
                            ST qv = Conv<P>::st(f1[i], sc1);
                            if constexpr (P::id == 3) qv = bf16_flush(qv);
                            snew += fix24_sat<ST>(qv, &bad);
                            st_stream(fd + i * plane + id, qv);
                        }
                        // exact: sum of the cell's order-parameter populations is unchanged
                        st_stream(rd + id, rs[id] + fix24_to_rest(PHIT ? -snew : sold - snew, k1));
                        if (bad) atomicOr(A.flags, 2);
                    } else {
#pragma unroll
                        for (int i = 0; i < 7; ++i) st_stream(fd + i * plane + id, Conv<P>::st(f1[i], R(1)));
                    }
                    const R sc2 = P::MIX ? kp.scale[1] : R(1);
#pragma unroll
                    for (int i = 0; i < 19; ++i) st_stream(fd + (7 + i) * plane + id, Conv<P>::st(f2[i], sc2));
                    st_stream(ad + 0 * plane + id, (AX)ux);
                    st_stream(ad + 1 * plane + id, (AX)uy);
                    st_stream(ad + 2 * plane + id, (AX)uz);
                    st_stream(ad + 3 * plane + id, (AX)Sx);
                    st_stream(ad + 4 * plane + id, (AX)Sy);
                    st_stream(ad + 5 * plane + id, (AX)Sz);
                    st_stream(ad + 6 * plane + id, (AX)phi);
                    if (!isfinite(phi) || !isfinite(ux) || !isfinite(uy) || !isfinite(uz)) atomicOr(A.flags, 1);
                }
            }
        }
        if constexpr (MOVING && MODE == MODE_STEP) {
            // the warps' sums in order; particles out of the chunk's reach: zero partials
            __syncthreads();
            for (int q = tid; q < 6 * A.np; q += NT) A.partials[(long long)q * A.ntiles + t] = 0.0;
            __syncthreads();
            for (int q = tid; q < 6 * nn; q += NT) {
                const int j = q / 6, c = q - 6 * j;
                double acc = 0.0;
                for (int w = 0; w < NW; ++w) acc += s_facc[(j * NW + w) * 6 + c];
                A.partials[((long long)s_near[j].k * 6 + c) * A.ntiles + t] = acc;
            }
        }
    }
}

}  // namespace pf
