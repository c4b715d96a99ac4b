// 3D time step of the FP32-arithmetic policies, two cells per thread.
//
// The update of k_step3d (Sec. 3.3, steps 2-6; D3Q7 + D3Q19) in two launches:
//   k_phi3d       phi of every cell (Eq. 31: the pulled order-parameter
//                 populations summed once) into a plane of its own; the 16-bit
//                 policies also replace the rest population by the cell's exact
//                 fixed-point phi, which is all the update needs of that lattice
//                 at unit rates;
//   k_step3d_pair everything else, marching tiles of TX x TY columns in z.
//
// k_step3d, which ran these policies before, spent 1860 thread instructions per cell at 160^3
// (16-bit storage) and waited on global loads at 24 warps per SM: every cell of
// the tile + 2 frame pulled and summed seven populations.  Here the frames are
// loads of one float, and a thread owns two cells that advance together as the
// lanes of packed FP32 (f32x2) arithmetic: the same column in two chunks of
// z, zc planes apart.  The rings hold float2 (chunk A, chunk B), so every
// stencil value of both cells is one 8-byte shared-memory load and one packed
// operation, with no lane shuffles and no misaligned pairs in x; what a split
// in x or y would share between the two cells (frame columns) is small against
// that.  The frames of phi and phi0 are copied two planes ahead (cp.async); the
// cell's own populations and lagged fields are loaded at the top of a plane
// and used after its two barriers.
// Measured per step, before and after: 256^3 with 16-bit storage 1399 -> 1042 us
// (1127 instructions per cell, 129 of them k_phi3d's), 131 x 100 x 90 in FP32 between
// walls 280 -> 125 us.  What bounds it now is issue: 1996 instructions per thread and
// plane at 0.44 per clock and scheduler with 16 warps per SM, which registers cap.
// Constants pre-paired as float2 kernel parameters were slower (1115 us).
#pragma once

#include "pf_kernels2d_pair.cuh"
#include "pf_kernels3d.cuh"

namespace pf {

// phi of every cell of the tiles' columns: TX x TY threads, gridDim.y pieces of
// the planes of a tile's chunks.  A streaming pass: 20 bytes in and 12 out per cell
// (16-bit storage), 28 in and 4 out (FP32).
template <class P, int TX, int TY, bool EXT, bool SINGLE>
__global__ void __launch_bounds__(TX *TY) k_phi3d(const __grid_constant__ StepArgs A, const __grid_constant__ DomainDev D1,
                                                   int chunks)
{
    using ST = typename P::store;
    for (int t = blockIdx.x; t < A.ntiles; t += gridDim.x) {
        int tx, ty, tz;
        const DomainDev &Dm = tile_of<SINGLE>(A, D1, t, tx, ty, tz);
        const int nx = Dm.nx, ny = Dm.ny, nz = Dm.nz;
        const int x = tx * TX + threadIdx.x % TX, y = ty * TY + threadIdx.x / TX;
        if (x >= nx || y >= ny) continue;
        const int z0 = tz * chunks * Dm.zc, zn = min(chunks * Dm.zc, nz - z0);
        const int per = (zn + gridDim.y - 1) / gridDim.y;
        const int za = z0 + blockIdx.y * per, zb = min(za + per, z0 + zn);
        const int plane = (int)Dm.plane, zstride = Dm.pitch * ny;
        const ST *fs = reinterpret_cast<const ST *>(Dm.f[A.par]);
        [[maybe_unused]] long long *rs = reinterpret_cast<long long *>(Dm.rest[A.par]);
        [[maybe_unused]] const int k1 = Dm.p.klog2[0];
        const bool wall = EXT && Dm.wall_y;
        const int own = y * Dm.pitch + x;
        // pulled from x -+ 1, y -+ 1 (beyond a wall: the cell's own opposite population)
        const int xw = y * Dm.pitch + (x == 0 ? nx - 1 : x - 1), xe = y * Dm.pitch + (x == nx - 1 ? 0 : x + 1);
        const bool bs = wall && y == 0, bn = wall && y == ny - 1;
        const int ys = (bs ? 4 * plane + own : 3 * plane + (y == 0 ? ny - 1 : y - 1) * Dm.pitch + x);
        const int yn = (bn ? 3 * plane + own : 4 * plane + (y == ny - 1 ? 0 : y + 1) * Dm.pitch + x);
        float *out = phi_of_step(Dm);
        // BATCH planes' loads in flight before the first sum
        constexpr int BATCH = 4;
        for (int z = za; z < zb; z += BATCH) {
            ST q[BATCH][P::MIX ? 6 : 7];
            [[maybe_unused]] long long r[BATCH];
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                const int zz = min(z + j, zb - 1);
                const int zo = zz * zstride, zm = (zz == 0 ? nz - 1 : zz - 1) * zstride,
                          zp = (zz == nz - 1 ? 0 : zz + 1) * zstride;
                if constexpr (P::MIX) r[j] = rs[zo + own];
                else q[j][6] = ldg(fs + zo + own);
                q[j][0] = ldg(fs + plane + zo + xw);
                q[j][1] = ldg(fs + 2 * plane + zo + xe);
                q[j][2] = ldg(fs + zo + ys);
                q[j][3] = ldg(fs + zo + yn);
                q[j][4] = ldg(fs + 5 * plane + zm + own);
                q[j][5] = ldg(fs + 6 * plane + zp + own);
            }
#pragma unroll
            for (int j = 0; j < BATCH; ++j) {
                if (z + j >= zb) break;
                const int id = (z + j) * zstride + own;
                if constexpr (P::MIX) {
                    int images = 0;
#pragma unroll
                    for (int i = 0; i < 6; ++i) images += fix24_stored<ST>(q[j][i]);
                    const long long e = r[j] + fix24_to_rest(images, k1);
                    rs[id] = e;
                    out[id] = float_of_fixed(e);
                } else {
                    float acc = q[j][6];
#pragma unroll
                    for (int i = 0; i < 6; ++i) acc += q[j][i];
                    out[id] = acc;
                }
            }
        }
    }
}

__device__ __forceinline__ void cp_async4(float *dst, const float *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// D3Q19 isotropic gradient (weights 1/18 faces, 1/36 edges, cs^2 = 1/3) of two
// cells at index c of three float2 planes (below, centre, above) of width W;
// opposite edges are differenced once and shared by two components
template <int W>
__device__ __forceinline__ void grad19_pair(const float2 *lo, const float2 *mid, const float2 *hi, int c, F2 &gx,
                                            F2 &gy, F2 &gz)
{
    auto at = [&](const float2 *p, int d) -> F2 { return {p[c + d]}; };
    const F2 a = at(mid, W + 1) - at(mid, -W - 1), b = at(mid, 1 - W) - at(mid, W - 1);
    const F2 d = at(hi, 1) - at(lo, -1), e = at(lo, 1) - at(hi, -1);
    const F2 f = at(hi, W) - at(lo, -W), g = at(lo, W) - at(hi, -W);
    const F2 f6 = mk2(1.0f / 6.0f), f12 = mk2(1.0f / 12.0f);
    gx = fma2(f6, at(mid, 1) - at(mid, -1), f12 * ((a + b) + (d + e)));
    gy = fma2(f6, at(mid, W) - at(mid, -W), f12 * ((a - b) + (f + g)));
    gz = fma2(f6, at(hi, 0) - at(lo, 0), f12 * ((d - e) + (f - g)));
}

template <int W>
__device__ __forceinline__ F2 lap19_pair(const float2 *lo, const float2 *mid, const float2 *hi, int c)
{
    auto at = [&](const float2 *p, int d) -> F2 { return {p[c + d]}; };
    const F2 v = at(mid, 0);
    const F2 faces = ((at(mid, 1) + at(mid, -1)) + (at(mid, W) + at(mid, -W))) + (at(hi, 0) + at(lo, 0));
    const F2 edges = (((at(mid, W + 1) + at(mid, -W - 1)) + (at(mid, 1 - W) + at(mid, W - 1))) +
                      ((at(hi, 1) + at(lo, -1)) + (at(lo, 1) + at(hi, -1)))) +
                     ((at(hi, W) + at(lo, -W)) + (at(lo, W) + at(hi, -W)));
    return fma2(mk2(1.0f / 3.0f), fma2(mk2(-6.0f), v, faces), mk2(1.0f / 6.0f) * fma2(mk2(-12.0f), v, edges));
}

// D3Q19 populations of two cells from Hermite moments (m = N_H^-1 h, f = M0^-1 m);
// third = the moments 10-15 (null: zero)
__device__ __forceinline__ void from_hermite19_pair(const F2 h[10], const F2 *third, const F2 h16[3], F2 f[19], F2 cs2,
                                                    F2 cs4)
{
    const F2 m4 = fma2(cs2, h[0], h[4]), m5 = fma2(cs2, h[0], h[5]), m6 = fma2(cs2, h[0], h[6]);
    const F2 c4 = cs4 * h[0];
    const F2 m16 = fma2(cs2, h[4] + h[5], h16[0] + c4), m17 = fma2(cs2, h[4] + h[6], h16[1] + c4),
             m18 = fma2(cs2, h[5] + h[6], h16[2] + c4);
    F2 t[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) t[k] = third ? fma2(cs2, h[1 + k / 2], third[k]) : cs2 * h[1 + k / 2];
    const F2 hh = mk2(0.5f), q = mk2(0.25f);
    f[0] = (h[0] - (m4 + m5)) + ((m16 - m6) + (m17 + m18));
    auto face = [&](F2 m1, F2 m2, F2 ta, F2 tb, F2 ea, F2 eb, F2 &fp, F2 &fm) {
        const F2 even = m2 - (ea + eb), odd = m1 - (ta + tb);
        fp = hh * (even + odd);
        fm = hh * (even - odd);
    };
    face(h[1], m4, t[0], t[1], m16, m17, f[1], f[2]);
    face(h[2], m5, t[2], t[3], m16, m18, f[3], f[4]);
    face(h[3], m6, t[4], t[5], m17, m18, f[5], f[6]);
    // edges: (+, +), (-, -), (+, -), (-, +) of a pair of axes
    auto edge = [&](F2 off, F2 ta, F2 tb, F2 e, F2 *o) {
        const F2 s = e + off, d = e - off, p = ta + tb, m = ta - tb;
        o[0] = q * (s + p);
        o[1] = q * (s - p);
        o[2] = q * (d + m);
        o[3] = q * (d - m);
    };
    edge(h[7], t[0], t[2], m16, f + 7);
    edge(h[8], t[1], t[4], m17, f + 11);
    edge(h[9], t[3], t[5], m18, f + 15);
}

// the second-order and zeroth raw moments the flow collision needs
struct Mom19 {
    F2 m0, sum, d[3], o[3], exy, exz, eyz;  // sum: without the rest population
};
__device__ __forceinline__ Mom19 moments19_pair(const F2 f[19])
{
    Mom19 m;
    m.exy = (f[7] + f[8]) + (f[9] + f[10]);
    m.exz = (f[11] + f[12]) + (f[13] + f[14]);
    m.eyz = (f[15] + f[16]) + (f[17] + f[18]);
    const F2 fx = f[1] + f[2], fy = f[3] + f[4], fz = f[5] + f[6];
    m.d[0] = fx + (m.exy + m.exz);
    m.d[1] = fy + (m.exy + m.eyz);
    m.d[2] = fz + (m.exz + m.eyz);
    m.sum = ((fx + fy) + fz) + ((m.exy + m.exz) + m.eyz);
    m.m0 = f[0] + m.sum;
    m.o[0] = (f[7] + f[8]) - (f[9] + f[10]);
    m.o[1] = (f[11] + f[12]) - (f[13] + f[14]);
    m.o[2] = (f[15] + f[16]) - (f[17] + f[18]);
    return m;
}

// ring sizes in planes (see the hazards at the top of the plane loop)
constexpr int P3_PHI = 6, P3_P0 = 5, P3_MU = 3, P3_T = 4, P3_RAW = 6;
template <int TX, int TY>
constexpr int step3d_pair_smem()
{
    return (int)sizeof(float2) * ((P3_PHI + P3_P0) * (TX + 4) * (TY + 4) + (P3_MU + 3 * P3_T + P3_RAW) * (TX + 2) * (TY + 2));
}

// EXT: the instantiation also handles domains with walls at the ends of y;
// UNIT: every domain of the launch has unit rates for its non-conserved
// moments (and the Cahn-Hilliard lattice).  Two CTAs of 256 threads per SM:
// 128 registers each (80 registers for three CTAs would spill the pairs' 19
// populations), 95 KB of shared memory.
template <class P, int TX, int TY, bool EXT, bool UNIT, bool SINGLE>
__global__ void __launch_bounds__(TX *TY, 2) k_step3d_pair(const __grid_constant__ StepArgs A,
                                                           const __grid_constant__ DomainDev D1)
{
    using ST = typename P::store;
    constexpr int NT = TX * TY;
    constexpr int FX = TX + 4, FY = TY + 4, FP = FX * FY;  // tile + 2 frame (one plane)
    constexpr int WX = TX + 2, WY = TY + 2, WP = WX * WY;  // tile + 1 frame
    static_assert(FP <= 2 * NT && WP <= 2 * NT, "at most two frame cells per thread");
    extern __shared__ __align__(16) float2 s_pair3d[];
    float2 *const s_phi = s_pair3d, *const s_p0 = s_phi + P3_PHI * FP, *const s_mu = s_p0 + P3_P0 * FP,
                  *const s_T = s_mu + P3_MU * WP,  // [slot][component][WP]
                  *const s_raw = s_T + 3 * P3_T * WP;  // u, S of one plane of the tile + 1 frame
    const int tid = threadIdx.x, lx = tid % TX, ly = tid / TX;

    for (int t = blockIdx.x; t < A.ntiles; t += gridDim.x) {
        int tx, ty, tz;
        const DomainDev &Dm = tile_of<SINGLE>(A, D1, t, tx, ty, tz);
        const int nx = Dm.nx, ny = Dm.ny, nz = Dm.nz, pitch = Dm.pitch;
        const int plane = (int)Dm.plane;  // 26 * plane < 2^31 (checked at create)
        const int zstride = pitch * ny, zspan = zstride * nz;
        const int x0 = tx * TX, y0 = ty * TY;
        const int zc = Dm.zc, za = tz * 2 * zc;
        const int nk = min(zc, nz - za), nkb = nz - (za + zc);  // planes of the chunks (nkb may be <= 0)
        const KParams<float> &kp = Dm.kf;
        const int wall = EXT ? Dm.wall_y : 0;

        // wrapped column / row of a table coordinate; with walls a row beyond
        // one is its mirror image (clamped: rows that far out only feed cells
        // beyond the domain)
        auto col = [&](int x) { return wrap_idx(x, nx); };
        auto row = [&](int y) -> int {
            if (EXT && wall) {
                const int m = y < 0 ? -1 - y : (y >= ny ? 2 * ny - 1 - y : y);
                return min(max(m, 0), ny - 1);
            }
            return wrap_idx(y, ny);
        };
        // frame cells of this thread: the tile + 2 frame r and r + NT; the tile + 1
        // frame from the other end, so that the second cells fall to other warps
        const int fo0 = row(y0 - 2 + tid / FX) * pitch + col(x0 - 2 + tid % FX);
        const int r1 = tid + NT;
        const bool f1on = r1 < FP;
        const int fo1 = f1on ? row(y0 - 2 + r1 / FX) * pitch + col(x0 - 2 + r1 % FX) : fo0;
        const int w0 = tid, w1 = WP - 1 - (NT - 1 - tid);
        const bool w1on = w1 >= NT;
        const int wo0 = row(y0 - 1 + w0 / WX) * pitch + col(x0 - 1 + w0 % WX);
        const int wo1 = w1on ? row(y0 - 1 + w1 / WX) * pitch + col(x0 - 1 + w1 % WX) : wo0;
        const int wf0 = (w0 / WX + 1) * FX + w0 % WX + 1, wf1 = w1on ? (w1 / WX + 1) * FX + w1 % WX + 1 : wf0;
        float sg0 = 1.0f, sg1 = 1.0f;  // T_xy and T_yz are odd under the wall mirror
        if (EXT && wall) {
            const int ya = y0 - 1 + w0 / WX, yb = y0 - 1 + w1 / WX;
            if (ya < 0 || ya >= ny) sg0 = -1.0f;
            if (yb < 0 || yb >= ny) sg1 = -1.0f;
        }
        // own cell: offsets in its plane of the cells it pulls from
        const int gx = x0 + lx, gy = y0 + ly;
        const bool valid = gx < nx && gy < ny;
        const int xc = col(gx), xw = col(gx - 1), xe = col(gx + 1);
        const int yc = row(gy) * pitch, ys = row(gy - 1) * pitch, yn = row(gy + 1) * pitch;
        const bool bs = EXT && wall && gy == 0, bn = EXT && wall && gy == ny - 1;

        const ST *fs = reinterpret_cast<const ST *>(Dm.f[A.par]);
        ST *fd = reinterpret_cast<ST *>(Dm.f[A.par ^ 1]);
        const float *as = reinterpret_cast<const float *>(Dm.aux[A.par]);
        float *ad = reinterpret_cast<float *>(Dm.aux[A.par ^ 1]);
        const float *ph0 = reinterpret_cast<const float *>(Dm.phi0), *pht = phi_of_step(Dm);
        const long long *rs = reinterpret_cast<const long long *>(Dm.rest[A.par]);
        long long *rd = reinterpret_cast<long long *>(Dm.rest[A.par ^ 1]);

        // plane offsets of both chunks, kept wrapped as they advance
        auto zwrap = [&](int z) { return wrap_idx(z, nz) * zstride; };
        auto znext = [&](int zo) { return zo + zstride == zspan ? 0 : zo + zstride; };
        int am = zwrap(za - 1), a0 = zwrap(za), ap = zwrap(za + 1);
        int bm = zwrap(za + zc - 1), b0 = zwrap(za + zc), bp = zwrap(za + zc + 1);

        // copies of phi and phi0 of the planes at zoa, zob into ring slots
        auto copy_plane = [&](int zoa, int zob, int sp, int s0) {
            float2 *dp = s_phi + sp * FP, *d0 = s_p0 + s0 * FP;
            cp_async4(&dp[tid].x, pht + zoa + fo0);
            cp_async4(&dp[tid].y, pht + zob + fo0);
            cp_async4(&d0[tid].x, ph0 + zoa + fo0);
            cp_async4(&d0[tid].y, ph0 + zob + fo0);
            if (f1on) {
                cp_async4(&dp[r1].x, pht + zoa + fo1);
                cp_async4(&dp[r1].y, pht + zob + fo1);
                cp_async4(&d0[r1].x, ph0 + zoa + fo1);
                cp_async4(&d0[r1].y, ph0 + zob + fo1);
            }
        };
        // u, S of a plane of the tile + 1 frame: each thread copies the cells it
        // turns into T itself (no barrier between the two)
        auto copy_raw = [&](int zoa, int zob) {
#pragma unroll
            for (int j = 0; j < 6; ++j) {
                cp_async4(&s_raw[j * WP + w0].x, as + j * plane + zoa + wo0);
                cp_async4(&s_raw[j * WP + w0].y, as + j * plane + zob + wo0);
            }
            if (w1on) {
#pragma unroll
                for (int j = 0; j < 6; ++j) {
                    cp_async4(&s_raw[j * WP + w1].x, as + j * plane + zoa + wo1);
                    cp_async4(&s_raw[j * WP + w1].y, as + j * plane + zob + wo1);
                }
            }
        };
        auto T_cell = [&](float sg, int w, float2 *dst) {
            F2 v[6];
#pragma unroll
            for (int j = 0; j < 6; ++j) v[j] = {s_raw[j * WP + w]};
            const F2 s = mk2(sg);
            dst[w] = (s * (v[3] * v[1] - v[0] * v[4])).v;
            dst[WP + w] = (v[3] * v[2] - v[0] * v[5]).v;
            dst[2 * WP + w] = (s * (v[4] * v[2] - v[1] * v[5])).v;
        };
        auto T_plane = [&](int slot) {
            float2 *dst = s_T + slot * 3 * WP;
            T_cell(sg0, w0, dst);
            if (w1on) T_cell(sg1, w1, dst);
        };
        const F2 c_dw = mk2(kp.c_dw), n_lap = mk2(-kp.c_lap), c_pen = mk2(kp.c_pen), c_wet = mk2(kp.c_wet),
                 n_wlap = mk2(-kp.c_wlap), one = mk2(1.0f), three = mk2(3.0f);
        auto mu_cell = [&](int c, const float2 *const p[3], const float2 *const q[3]) -> float2 {
            const F2 ph = {p[1][c]}, p0 = {q[1][c]};
            const F2 lp = lap19_pair<FX>(p[0], p[1], p[2], c), lp0 = lap19_pair<FX>(q[0], q[1], q[2], c);
            const F2 p02 = p0 * p0;
            F2 m = c_dw * ph * ((ph - one) * (ph + one));
            m = fma2(n_lap, lp, m);
            m = fma2(c_pen * p02, ph, m);
            m = fma2(c_wet * p0, fma2(three * ph, ph, p02) - one, m);
            return fma2(n_wlap, lp0, m).v;
        };
        // mu of the plane whose phi slot is sp, phi0 slot s0, into slot sm
        auto inc = [](int s, int n) { return s + 1 == n ? 0 : s + 1; };
        auto dec = [](int s, int n) { return s == 0 ? n - 1 : s - 1; };
        auto mu_plane = [&](int sp, int s0, int sm) {
            const float2 *const p[3] = {s_phi + dec(sp, P3_PHI) * FP, s_phi + sp * FP, s_phi + inc(sp, P3_PHI) * FP};
            const float2 *const q[3] = {s_p0 + dec(s0, P3_P0) * FP, s_p0 + s0 * FP, s_p0 + inc(s0, P3_P0) * FP};
            float2 *dst = s_mu + sm * WP;
            dst[w0] = mu_cell(wf0, p, q);
            if (w1on) dst[w1] = mu_cell(wf1, p, q);
        };

        __syncthreads();  // the previous tile's readers are done
        // prologue: phi, phi0 planes -2 .. 2 (slots 0 .. 4), T planes -1, 0 (slots 0,
        // 1), u, S of plane 1, mu planes -1, 0 (slots 0, 1)
        int fa = zwrap(za - 2), fb = zwrap(za + zc - 2);
        for (int k = 0; k < 5; ++k) {
            copy_plane(fa, fb, k, k);
            fa = znext(fa);
            fb = znext(fb);
        }
        copy_raw(am, bm);
        cp_async_commit();
        cp_async_wait<0>();
        T_plane(0);
        copy_raw(a0, b0);
        cp_async_commit();
        cp_async_wait<0>();
        T_plane(1);
        copy_raw(ap, bp);
        cp_async_commit();
        __syncthreads();
        mu_plane(1, 1, 0);
        mu_plane(2, 2, 1);
        __syncthreads();  // (plane 3's copy takes the phi0 slot of plane -2)
        int sp = 2, s0 = 2, sm = 1, sT = 1;  // slots of the plane being updated
        constexpr unsigned dirs7 = P::MIX ? 1u : 0u;

        // Ring hazards: at the top of a plane others may still update the plane
        // before it (reading phi z-2 .. z, phi0 z-1, T z-2 .. z): the copy of
        // plane z+3 takes a sixth phi and a fifth phi0 slot, T z+1 a fourth;
        // mu z+1 is written after the first barrier, when only mu z-1 and z
        // are still read.
        for (int k = 0; k < nk; ++k) {
            // phase 1: T of plane z+1 from the copies of a plane ago; phi, phi0 of plane
            // z+3 and u, S of plane z+2 on their way
            cp_async_wait<0>();
            T_plane(inc(sT, P3_T));
            {
                const int s3 = inc(inc(inc(sp, P3_PHI), P3_PHI), P3_PHI);
                const int q3 = inc(inc(inc(s0, P3_P0), P3_P0), P3_P0);
                copy_plane(fa, fb, s3, q3);
                copy_raw(znext(ap), znext(bp));
                cp_async_commit();
                fa = znext(fa);
                fb = znext(fb);
            }
            // the own cells' loads, used after the two barriers
            ST qa[19], qb[19];
            [[maybe_unused]] ST ea[7], eb[7];
            float la[7], lb[7];
            [[maybe_unused]] long long ra = 0, rb = 0;
            const int own = yc + xc;
            auto pull = [&](int base, int i, int zm, int z0_, int zp) -> int {
                const int cx = C19X[i], cy = C19Y[i], cz = C19Z[i];
                const int xo = cx > 0 ? xw : (cx < 0 ? xe : xc);
                if (EXT && cy != 0) {
                    if (cy > 0 ? bs : bn) return (base + opp19(i)) * plane + z0_ + own;
                }
                const int yo = cy > 0 ? ys : (cy < 0 ? yn : yc);
                return (base + i) * plane + (cz > 0 ? zm : (cz < 0 ? zp : z0_)) + yo + xo;
            };
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                qa[i] = ldg(fs + pull(7, i, am, a0, ap));
                qb[i] = ldg(fs + pull(7, i, bm, b0, bp));
            }
            if constexpr (!UNIT) {
#pragma unroll
                for (int i = dirs7; i < 7; ++i) {
                    ea[i] = ldg(fs + pull(0, i, am, a0, ap));
                    eb[i] = ldg(fs + pull(0, i, bm, b0, bp));
                }
            }
#pragma unroll
            for (int j = 0; j < 7; ++j) {
                la[j] = __ldg(as + j * plane + a0 + own);
                lb[j] = __ldg(as + j * plane + b0 + own);
            }
            if constexpr (P::MIX) {
                ra = __ldg(rs + a0 + own);
                rb = __ldg(rs + b0 + own);
            }
            __syncthreads();
            // phase 2: mu of plane z+1
            mu_plane(inc(sp, P3_PHI), inc(s0, P3_P0), inc(sm, P3_MU));
            __syncthreads();

            // phase 3: the own cells
            const float2 *plo = s_phi + dec(sp, P3_PHI) * FP, *pmid = s_phi + sp * FP, *phi_hi = s_phi + inc(sp, P3_PHI) * FP;
            const float2 *mlo = s_mu + dec(sm, P3_MU) * WP, *mmid = s_mu + sm * WP, *mhi = s_mu + inc(sm, P3_MU) * WP;
            const float2 *tlo = s_T + dec(sT, P3_T) * 3 * WP, *tmid = s_T + sT * 3 * WP, *thi = s_T + inc(sT, P3_T) * 3 * WP;
            const int cf = (ly + 2) * FX + lx + 2, cw = (ly + 1) * WX + lx + 1;
            const F2 phi = {pmid[cf]}, phi0 = {s_p0[s0 * FP + cf]}, mu = {mmid[cw]};
            F2 gpx, gpy, gpz, gmx, gmy, gmz;
            grad19_pair<FX>(plo, pmid, phi_hi, cf, gpx, gpy, gpz);
            grad19_pair<WX>(mlo, mmid, mhi, cw, gmx, gmy, gmz);
            const F2 half = mk2(0.5f), two = mk2(2.0f), drho = mk2(kp.drho), Mdrho = mk2(kp.Mdrho);
            const F2 rho = fma2(drho, phi, mk2(kp.rhom));
            // conservative Allen-Cahn option: theta n = (2/D)(1 - phi^2) grad phi/|grad phi|
            // and the mass flux M (rho1 - rho2)/2 (grad phi - theta n)
            const bool cac = !UNIT && Dm.p.phase_model == 1;
            F2 tnx = mk2(0.0f), tny = tnx, tnz = tnx;
            F2 Sx = Mdrho * gmx, Sy = Mdrho * gmy, Sz = Mdrho * gmz;
            if (cac) {
                const F2 g2 = fma2(gpx, gpx, fma2(gpy, gpy, gpz * gpz));
                const F2 th = mk2(kp.two_over_D) * (one - phi * phi);
                const F2 inv = mk2(g2.v.x > 1e-24f ? 1.0f / sqrtf(g2.v.x) : 0.0f,
                                   g2.v.y > 1e-24f ? 1.0f / sqrtf(g2.v.y) : 0.0f);
                tnx = th * gpx * inv;
                tny = th * gpy * inv;
                tnz = th * gpz * inv;
                Sx = Mdrho * (gpx - tnx);
                Sy = Mdrho * (gpy - tny);
                Sz = Mdrho * (gpz - tnz);
            }
            F2 Fx = fma2(mu, gpx, mk2(kp.Fb[0])), Fy = fma2(mu, gpy, mk2(kp.Fb[1])), Fz = fma2(mu, gpz, mk2(kp.Fb[2]));
            {
                // F_c,b = 1/2 sum_a d_a T_ab with T antisymmetric (previous step)
                F2 xx, xy, xz, yx, yy, yz, zx, zy, zz;
                grad19_pair<WX>(tlo, tmid, thi, cw, xx, xy, xz);                             // T_xy
                grad19_pair<WX>(tlo + WP, tmid + WP, thi + WP, cw, yx, yy, yz);              // T_xz
                grad19_pair<WX>(tlo + 2 * WP, tmid + 2 * WP, thi + 2 * WP, cw, zx, zy, zz);  // T_yz
                const F2 nh = mk2(-0.5f);
                Fx = fma2(nh, xy + yz, Fx);
                Fy = fma2(half, xx - zz, Fy);
                Fz = fma2(half, yx + zy, Fz);
            }
            F2 f2[19];
            const F2 isc2 = mk2(kp.inv_scale[1]);
#pragma unroll
            for (int i = 0; i < 19; ++i) {
                f2[i] = mk2(stored_to_float<ST>(qa[i]), stored_to_float<ST>(qb[i]));
                if constexpr (P::MIX) f2[i] = f2[i] * isc2;
            }
            const F2 jx = ((f2[1] - f2[2]) + (f2[7] - f2[8])) + ((f2[9] - f2[10]) + ((f2[11] - f2[12]) + (f2[13] - f2[14])));
            const F2 jy = ((f2[3] - f2[4]) + (f2[7] - f2[8])) + ((f2[10] - f2[9]) + ((f2[15] - f2[16]) + (f2[17] - f2[18])));
            const F2 jz = ((f2[5] - f2[6]) + (f2[11] - f2[12])) + ((f2[14] - f2[13]) + ((f2[15] - f2[16]) + (f2[18] - f2[17])));
            const Mom19 mom = moments19_pair(f2);
            const F2 irho = rcp2(rho);
            const F2 usx = fma2(half, Fx, jx) * irho, usy = fma2(half, Fy, jy) * irho, usz = fma2(half, Fz, jz) * irho;
            const F2 np0 = mk2(0.0f) - phi0;
            const F2 fpx = np0 * usx, fpy = np0 * usy, fpz = np0 * usz;
            const F2 ux = fma2(half, fpx, usx), uy = fma2(half, fpy, usy), uz = fma2(half, fpz, usz);
            const F2 Ftx = fma2(rho, fpx, Fx), Fty = fma2(rho, fpy, Fy), Ftz = fma2(rho, fpz, Fz);
            const F2 upx = mk2(la[0], lb[0]), upy = mk2(la[1], lb[1]), upz = mk2(la[2], lb[2]);
            const F2 Spx = mk2(la[3], lb[3]), Spy = mk2(la[4], lb[4]), Spz = mk2(la[5], lb[5]);
            const F2 php = mk2(la[6], lb[6]);

            // relaxation rates (Eq. 35) and pressure (Eq. 36b)
            F2 solid = one - phi0;
            solid = mk2(fmaxf(solid.v.x, kp.solid_eps), fmaxf(solid.v.y, kp.solid_eps));
            const F2 nu = fma2(mk2(kp.dmu), phi, mk2(kp.mum)) * irho * rcp2(solid);
            const F2 inv_s2a = fma2(mk2(kp.two_over_1md0), nu, half), inv_s2b = fma2(mk2(kp.inv_cs2), nu, half);
            const F2 Kf = mk2(kp.K);
            const F2 H = Kf * fma2(mk2(-kp.Hc1), inv_s2a, mk2(kp.Hc0));
            const F2 grx = drho * gpx, gry = drho * gpy, grz = drho * gpz;
            const F2 ugr = fma2(ux, grx, fma2(uy, gry, uz * grz));
            const F2 rux = rho * ux, ruy = rho * uy, ruz = rho * uz;
            const F2 Xx = (rux - Sx) * ux, Xy = (ruy - Sy) * uy, Xz = (ruz - Sz) * uz;
            const F2 dSx = Sx * ux - Spx * upx, dSy = Sy * uy - Spy * upy, dSz = Sz * uz - Spz * upz;
            const F2 uFx = ux * Ftx, uFy = uy * Fty, uFz = uz * Ftz;
            const F2 dt_term = two * ((uFx + uFy) + uFz) - ((dSx + dSy) + dSz);
            F2 Pr = fma2(half + H, ugr, mom.sum);
            Pr = fma2(mk2(-kp.w0f * kp.inv_1mcs2), (Xx + Xy) + Xz, Pr);
            Pr = mk2(kp.Pfac) * fma2(Kf * half, dt_term, Pr);

            const F2 cs2 = mk2(kp.cs2), cs4 = mk2(kp.cs4);
            const bool va = valid, vb = valid && k < nkb;
            const int ida = a0 + own, idb = b0 + own;
            // order-parameter lattice (D3Q7)
            {
                const F2 em = cac ? phi : mk2(kp.eta) * mu;  // Allen-Cahn: eta mu -> phi
                const F2 h0 = phi, h2 = cs2 * (em - phi);    // heq: phi, phi u, cs^2 (eta mu - phi)
                const F2 q1x = phi * ux, q1y = phi * uy, q1z = phi * uz;
                F2 gx1 = q1x - php * upx, gy1 = q1y - php * upy, gz1 = q1z - php * upz;  // hF 1-3
                if (cac) {
                    gx1 = fma2(cs2, tnx, gx1);
                    gy1 = fma2(cs2, tny, gy1);
                    gz1 = fma2(cs2, tnz, gz1);
                }
                F2 hx, hy, hz, hd[3], f1[7], hs = h0;
                [[maybe_unused]] int solda = 0, soldb = 0;
                if constexpr (UNIT) {
                    hx = fma2(half, gx1, q1x);
                    hy = fma2(half, gy1, q1y);
                    hz = fma2(half, gz1, q1z);
                    hd[0] = hd[1] = hd[2] = h2;
                } else {
                    const F2 isc1 = mk2(kp.inv_scale[0]);
#pragma unroll
                    for (int i = dirs7; i < 7; ++i) {
                        f1[i] = mk2(stored_to_float<ST>(ea[i]), stored_to_float<ST>(eb[i]));
                        if constexpr (P::MIX) {
                            f1[i] = f1[i] * isc1;
                            solda += fix24_stored<ST>(ea[i]);
                            soldb += fix24_stored<ST>(eb[i]);
                        }
                    }
                    const F2 s1p = mk2(kp.s1phi), c1 = mk2(1.0f - 0.5f * kp.s1phi), s2 = mk2(kp.s2), ncs2 = mk2(-kp.cs2);
                    auto relax = [&](F2 h, F2 he, F2 hF) { return fma2(c1, hF, h - s1p * (h - he)); };
                    hx = relax(f1[1] - f1[2], q1x, gx1);
                    hy = relax(f1[3] - f1[4], q1y, gy1);
                    hz = relax(f1[5] - f1[6], q1z, gz1);
#pragma unroll
                    for (int a = 0; a < 3; ++a) {
                        const F2 h = fma2(ncs2, h0, f1[1 + 2 * a] + f1[2 + 2 * a]);
                        hd[a] = h - s2 * (h - h2);
                    }
                }
                const F2 c0 = half * cs2 * hs;
                auto face = [&](F2 m1, F2 m2, F2 &fp, F2 &fm) {
                    const F2 e = fma2(half, m2, c0), o = half * m1;
                    fp = e + o;
                    fm = e - o;
                };
                face(hx, hd[0], f1[1], f1[2]);
                face(hy, hd[1], f1[3], f1[4]);
                face(hz, hd[2], f1[5], f1[6]);
                if constexpr (P::MIX) {
                    const F2 sc1 = mk2(kp.scale[0]);
                    const int k1 = Dm.p.klog2[0];
                    int bad = 0, badb = 0, na = 0, nb = 0;
                    // images of the stored values; the sums of magnitudes bound every
                    // value (and carry a NaN), so one test per cell finds the cells
                    // that may need saturating
                    ST qa_[6], qb_[6];
                    F2 mag = mk2(0.0f);
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        const F2 v = sc1 * f1[1 + i];
                        qa_[i] = Conv<P>::st(v.v.x, 1.0f);
                        qb_[i] = Conv<P>::st(v.v.y, 1.0f);
                        if constexpr (P::id == 3) {
                            qa_[i] = bf16_flush(qa_[i]);
                            qb_[i] = bf16_flush(qb_[i]);
                        }
                        const float a = stored_to_float<ST>(qa_[i]), b = stored_to_float<ST>(qb_[i]);
                        mag = mag + mk2(fabsf(a), fabsf(b));
                        const F2 w = mk2(16777216.0f) * mk2(a, b);
                        na += __float2int_rn(w.v.x);
                        nb += __float2int_rn(w.v.y);
                    }
                    if (!(mag.v.x < FIX24_LIMIT)) {
                        na = 0;
#pragma unroll
                        for (int i = 0; i < 6; ++i) na += fix24_sat<ST>(qa_[i], &bad);
                    }
                    if (!(mag.v.y < FIX24_LIMIT)) {
                        nb = 0;
#pragma unroll
                        for (int i = 0; i < 6; ++i) nb += fix24_sat<ST>(qb_[i], &badb);
                    }
#pragma unroll
                    for (int i = 0; i < 6; ++i) {
                        if (va) st_stream(fd + (1 + i) * plane + ida, qa_[i]);
                        if (vb) st_stream(fd + (1 + i) * plane + idb, qb_[i]);
                    }
                    // exact: the cell's populations sum to the phi k_phi3d left in rest
                    if (va) st_stream(rd + ida, ra - fix24_to_rest(na, k1));
                    if (vb) st_stream(rd + idb, rb - fix24_to_rest(nb, k1));
                    if ((va && bad) || (vb && badb)) atomicOr(A.flags, 2);
                } else {
                    f1[0] = fma2(mk2(1.0f - 3.0f * kp.cs2), hs, mk2(0.0f) - ((hd[0] + hd[1]) + hd[2]));
#pragma unroll
                    for (int i = 0; i < 7; ++i) {
                        if (va) st_stream(fd + i * plane + ida, f1[i].v.x);
                        if (vb) st_stream(fd + i * plane + idb, f1[i].v.y);
                    }
                }
            }
            // flow lattice (D3Q19)
            {
                const F2 c4r = mk2(kp.cs4 * kp.inv_1mcs2), ncs2 = mk2(-kp.cs2);
                const F2 c3 = mk2(1.0f - 3.0f * kp.cs2), tcs = mk2(2.0f * kp.cs2), nhalf = mk2(-0.5f);
                const F2 s2a = rcp2(inv_s2a), s2b = rcp2(inv_s2b), s0f = mk2(kp.s0);
                const F2 Mxx = fma2(two, uFx, fma2(tcs * ux, grx, fma2(c3, ugr, mk2(0.0f) - dSx)));
                const F2 Myy = fma2(two, uFy, fma2(tcs * uy, gry, fma2(c3, ugr, mk2(0.0f) - dSy)));
                const F2 Mzz = fma2(two, uFz, fma2(tcs * uz, grz, fma2(c3, ugr, mk2(0.0f) - dSz)));
                // symmetric products of two vectors: a_i b_j + b_i a_j
                auto sym = [](F2 a, F2 b, F2 c, F2 d) { return fma2(a, d, c * b); };
                const F2 sxy = sym(Sx, ux, Sy, uy), sxz = sym(Sx, ux, Sz, uz), syz = sym(Sy, uy, Sz, uz);
                const F2 pxy = sym(Spx, upx, Spy, upy), pxz = sym(Spx, upx, Spz, upz), pyz = sym(Spy, upy, Spz, upz);
                const F2 Mxy = fma2(cs2, sym(ux, grx, uy, gry), fma2(nhalf, sxy - pxy, sym(ux, Ftx, uy, Fty)));
                const F2 Mxz = fma2(cs2, sym(ux, grx, uz, grz), fma2(nhalf, sxz - pxz, sym(ux, Ftx, uz, Ftz)));
                const F2 Myz = fma2(cs2, sym(uy, gry, uz, grz), fma2(nhalf, syz - pyz, sym(uy, Fty, uz, Ftz)));
                const F2 nPc = ncs2 * Pr;
                const F2 q16 = nPc - c4r * Xz, q17 = nPc - c4r * Xy, q18 = nPc - c4r * Xx;
                const F2 g16 = mk2(0.0f) - c4r * Mzz, g17 = mk2(0.0f) - c4r * Myy, g18 = mk2(0.0f) - c4r * Mxx;
                F2 h[10], h16[3];
                h[0] = fma2(mk2(1.0f - 0.5f * kp.s0), ugr, mom.m0 - s0f * mom.m0);  // (heq = 0)
                // second order: h* = h - s (h - heq) + (1 - s/2) hF
                auto relax = [&](F2 v, F2 s, F2 he, F2 hF) { return fma2(fma2(nhalf, s, one), hF, v - s * (v - he)); };
                h[4] = relax(fma2(ncs2, mom.m0, mom.d[0]), s2a, Pr + Xx, Mxx);
                h[5] = relax(fma2(ncs2, mom.m0, mom.d[1]), s2a, Pr + Xy, Myy);
                h[6] = relax(fma2(ncs2, mom.m0, mom.d[2]), s2a, Pr + Xz, Mzz);
                h[7] = relax(mom.o[0], s2b, fma2(nhalf, sxy, rux * uy), Mxy);
                h[8] = relax(mom.o[1], s2b, fma2(nhalf, sxz, rux * uz), Mxz);
                h[9] = relax(mom.o[2], s2b, fma2(nhalf, syz, ruy * uz), Myz);
                if constexpr (UNIT) {
                    h[1] = fma2(half, Ftx, rux);
                    h[2] = fma2(half, Fty, ruy);
                    h[3] = fma2(half, Ftz, ruz);
                    h16[0] = fma2(half, g16, q16);
                    h16[1] = fma2(half, g17, q17);
                    h16[2] = fma2(half, g18, q18);
                    from_hermite19_pair(h, nullptr, h16, f2, cs2, cs4);
                } else {
                    const F2 s1 = mk2(kp.s1), s3 = mk2(kp.s3), s4 = mk2(kp.s4);
                    h[1] = relax(jx, s1, rux, Ftx);
                    h[2] = relax(jy, s1, ruy, Fty);
                    h[3] = relax(jz, s1, ruz, Ftz);
                    // (third-order moments: heq = hF = 0)
                    F2 th[6] = {(f2[7] - f2[8]) + (f2[9] - f2[10]),    (f2[11] - f2[12]) + (f2[13] - f2[14]),
                                (f2[7] - f2[8]) - (f2[9] - f2[10]),    (f2[15] - f2[16]) + (f2[17] - f2[18]),
                                (f2[11] - f2[12]) - (f2[13] - f2[14]), (f2[15] - f2[16]) - (f2[17] - f2[18])};
                    const F2 j[3] = {jx, jy, jz};
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const F2 v = fma2(ncs2, j[q / 2], th[q]);
                        th[q] = v - s3 * v;
                    }
                    auto fourth = [&](F2 e, F2 da, F2 db) { return fma2(cs4, mom.m0, fma2(ncs2, da + db, e)); };
                    h16[0] = relax(fourth(mom.exy, mom.d[0], mom.d[1]), s4, q16, g16);
                    h16[1] = relax(fourth(mom.exz, mom.d[0], mom.d[2]), s4, q17, g17);
                    h16[2] = relax(fourth(mom.eyz, mom.d[1], mom.d[2]), s4, q18, g18);
                    from_hermite19_pair(h, th, h16, f2, cs2, cs4);
                }
                const F2 sc2 = mk2(kp.scale[1]);
#pragma unroll
                for (int i = 0; i < 19; ++i) {
                    const F2 v = P::MIX ? sc2 * f2[i] : f2[i];
                    if (va) st_stream(fd + (7 + i) * plane + ida, Conv<P>::st(v.v.x, 1.0f));
                    if (vb) st_stream(fd + (7 + i) * plane + idb, Conv<P>::st(v.v.y, 1.0f));
                }
            }
            {
                const F2 out[7] = {ux, uy, uz, Sx, Sy, Sz, phi};
#pragma unroll
                for (int j = 0; j < 7; ++j) {
                    if (va) st_stream(ad + j * plane + ida, out[j].v.x);
                    if (vb) st_stream(ad + j * plane + idb, out[j].v.y);
                }
                // 0 * x is NaN for a non-finite x
                const F2 zero = mk2(0.0f);
                const F2 t = fma2(zero, phi, fma2(zero, ux, fma2(zero, uy, zero * uz)));
                if ((va && t.v.x != 0.0f) || (vb && t.v.y != 0.0f))
                    atomicOr(A.flags, 1);
            }
            // the next plane
            am = a0;
            a0 = ap;
            ap = znext(ap);
            bm = b0;
            b0 = bp;
            bp = znext(bp);
            sp = inc(sp, P3_PHI);
            s0 = inc(s0, P3_P0);
            sm = inc(sm, P3_MU);
            sT = inc(sT, P3_T);
        }
        cp_async_wait<0>();  // (the copies past the last plane)
    }
}

}  // namespace pf
