// S3: momentum predictor of Eqs. NS-num1 and rk3 on the staggered grid.
//
// u* = u^{k-1} + dt [zeta^k N^{k-1} + xi^k N^{k-2} - 2 alpha^k grad p^{k-1}
//                    + alpha^k div(tau^k + tau^{k-1})]
// N  = -div(uu) + mu_s lap(u) + f
//
// div(uu) by second-order central differences (products at centres and edges),
// the viscous term explicit with the advective weights, div(tau) at faces from
// centre tau with 4-point edge averages for the off-diagonal parts (div is linear,
// so the two stress levels are summed first).  Each thread computes the three
// faces (i+1/2, j, k), (i, j+1/2, k), (i, j, k+1/2) of its cell and marches along z;
// with walls the top y-face stays zero.
//
// momentum_point is the arithmetic of one cell.  What a cell shares with the cell
// above it (the fluxes and edge stresses half a plane up) travels along the march in
// registers, so that only planes k and k+1 are read.  Three kernels feed it:
//   momentum_tile      single precision: tiles, planes k, k+1 and k+2 (arriving)
//                      of u, v, w, p and of the summed stress S = tau^k + tau^{k-1}
//                      (written by the stress kernel) in a shared-memory ring;
//   momentum_column    double precision, bound by its FP64 instructions: neighbours
//                      straight through L1, threads numbered densely over the plane so
//                      that no lane idles on a ragged row;
//   momentum_soft_tile soft particles, where S is built from B^{k-1}, B^k and the solid
//                      fraction on the way.
#include "evp_internal.cuh"

namespace evp {

namespace {

__device__ __forceinline__ int pmod(int a, int n) {
    int r = a % n;
    return r < 0 ? r + n : r;
}
// a in [-n, 2n): one conditional wrap, no division
__device__ __forceinline__ int wrap1(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// 16-byte asynchronous copy (L2 only)
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}

template <typename T>
__device__ __forceinline__ void cp_async(T* smem, const T* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    if (sizeof(T) == 4)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(sa), "l"(gmem) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
// all but the most recently committed group have landed
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// Row ghost rules (walls): centred fields copy the nearest row; u and w take the odd
// mirror (no slip), v is zero outside the stored faces.  Periodic y wraps.  For row gy
// returns the source row and the factor (+1 copy, -1 negated copy, 0 zero) of velocity
// component q, or of a centred field for q = 3.
template <typename T>
__device__ __forceinline__ int row_rule(const Geo<T>& g, int gy, int q, int& src) {
    if (!g.walls) {
        src = pmod(gy, g.ny);
        return 1;
    }
    if (q == 3) {
        src = min(max(gy, 0), g.ny - 1);
        return 1;
    }
    const bool inside = gy >= 0 && gy < g.ny;
    if (q == 1) {
        src = inside ? gy : 0;
        return inside ? 1 : 0;
    }
    const int my = gy < 0 ? -1 - gy : (gy >= g.ny ? 2 * g.ny - 1 - gy : gy);
    src = min(max(my, 0), g.ny - 1);
    return (my >= 0 && my < g.ny) ? (inside ? 1 : -1) : 0;
}

// E elements from global (one 16-byte vector) into shared, times fac (-1 or 0)
template <typename T>
__device__ __forceinline__ void copy_scaled(T* dst, const T* src, int fac) {
    if constexpr (sizeof(T) == 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (fac) {
            v = __ldg(reinterpret_cast<const float4*>(src));
            v.x = -v.x; v.y = -v.y; v.z = -v.z; v.w = -v.w;
        }
        *reinterpret_cast<float4*>(dst) = v;
    } else {
        double2 v = make_double2(0.0, 0.0);
        if (fac) {
            v = __ldg(reinterpret_cast<const double2*>(src));
            v.x = -v.x; v.y = -v.y;
        }
        *reinterpret_cast<double2*>(dst) = v;
    }
}

// One rounding each, as written (no contraction choices left to the compiler: the three
// kernels below give the same bits)
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
// x a + y b + z c
template <typename T>
__device__ __forceinline__ T dot3(T x, T a, T y, T b, T z, T c) {
    return fma_rn(z, c, fma_rn(x, a, mul_rn(y, b)));
}

// What a cell at plane k takes over from plane k-1: the velocities there, the factors (twice
// the averages) of the fluxes u w and v w through its lower edges at k - 1/2, four times
// the flux w w there, and four times the edge stresses xz and yz.
template <typename T>
struct MomCarry {
    T um, vm, wm, uz, wx, vz, wy, fww, exz, eyz;
};

// The carry for plane k+1 from the planes k and k+1 that S gives (S as in momentum_point)
template <typename T, bool STRESS, typename Src>
__device__ __forceinline__ MomCarry<T> momentum_carry(const Src& S) {
    MomCarry<T> c;
    c.um = S.u(0, 0, 0);
    c.vm = S.v(0, 0, 0);
    c.wm = S.w(0, 0, 0);
    const T wz = c.wm + S.w(0, 0, 1);
    c.uz = c.um + S.u(0, 0, 1);
    c.wx = c.wm + S.w(1, 0, 0);
    c.vz = c.vm + S.v(0, 0, 1);
    c.wy = c.wm + S.w(0, 1, 0);
    c.fww = mul_rn(wz, wz);
    c.exz = c.eyz = T(0);
    if (STRESS) {
        c.exz = (S.s(2, 0, 0, 0) + S.s(2, 0, 0, 1)) + S.s(2, 1, 0, 1) + S.s(2, 1, 0, 0);
        c.eyz = (S.s(4, 0, 0, 0) + S.s(4, 0, 0, 1)) + S.s(4, 0, 1, 1) + S.s(4, 0, 1, 0);
    }
    return c;
}

// One cell (i, j, k): the momentum step at its three upper faces.  S gives the values
// around the cell at offsets di, dj in -1 .. 1 and planes k (dk = 0) and k+1 (dk = 1):
// S.u, S.v, S.w, S.p, S.s(component); wraps and wall ghosts are already applied.  c is
// the carry from plane k-1, replaced by the one for plane k+1; hist the history N^{k-2}.
// The halves of the averaged factors and the quarters of the edge averages are folded
// into the reciprocal spacings (powers of two: the same rounding).
template <typename T, bool STRESS, typename Src>
__device__ __forceinline__ void momentum_point(const Geo<T>& g, const ModelConst& mc, const MomentumArgs<T>& a,
                                               const Src& S, MomCarry<T>& c, const T (&hist)[3], int i, int j, int k,
                                               bool write) {
    const T qx = T(0.25) * g.idx, qy = T(0.25) * g.idy, qz = T(0.25) * g.idz;
    const T u0 = S.u(0, 0, 0), v0 = S.v(0, 0, 0), w0 = S.w(0, 0, 0);
    const T up = S.u(0, 0, 1), vp = S.v(0, 0, 1), wp = S.w(0, 0, 1);
    const T u10 = S.u(1, 0, 0), um0 = S.u(-1, 0, 0), u01 = S.u(0, 1, 0), u0m = S.u(0, -1, 0);
    const T v10 = S.v(1, 0, 0), vm0 = S.v(-1, 0, 0), v01 = S.v(0, 1, 0), v0m = S.v(0, -1, 0);
    const T w10 = S.w(1, 0, 0), wm0 = S.w(-1, 0, 0), w01 = S.w(0, 1, 0), w0m = S.w(0, -1, 0);

    // ---- div(uu) at the three faces: sums of neighbours, products four times the flux
    const T uxp = u0 + u10, uxm = um0 + u0, vyp = v0 + v01, vym = v0m + v0, wzp = w0 + wp;
    const T uy = u0 + u01, vx = v0 + v10, uz = u0 + up, wx = w0 + w10, vz = v0 + vp, wy = w0 + w01;
    const T uv = mul_rn(uy, vx), uw = mul_rn(uz, wx), vw = mul_rn(vz, wy);
    const T Ax = dot3(fma_rn(uxp, uxp, -mul_rn(uxm, uxm)), qx, fma_rn(-(u0m + u0), v0m + S.v(1, -1, 0), uv), qy,
                      fma_rn(-c.uz, c.wx, uw), qz);
    const T Ay = dot3(fma_rn(-(um0 + S.u(-1, 1, 0)), vm0 + v0, uv), qx, fma_rn(vyp, vyp, -mul_rn(vym, vym)), qy,
                      fma_rn(-c.vz, c.wy, vw), qz);
    const T Az = dot3(fma_rn(-(um0 + S.u(-1, 0, 1)), wm0 + w0, uw), qx, fma_rn(-(v0m + S.v(0, -1, 1)), w0m + w0, vw), qy,
                      fma_rn(wzp, wzp, -c.fww), qz);

    // ---- mu_s lap(u)
    const T idx2 = g.idx * g.idx, idy2 = g.idy * g.idy, idz2 = g.idz * g.idz;
    const T mu = kconst<T>(mc.mu_s, mc.f_mu_s);
    auto lap = [&](T f, T xp, T xm, T yp, T ym, T zp, T zm) {
        return dot3(fma_rn(T(-2), f, xp) + xm, idx2, fma_rn(T(-2), f, yp) + ym, idy2, fma_rn(T(-2), f, zp) + zm, idz2);
    };
    const T Lu = lap(u0, u10, um0, u01, u0m, up, c.um);
    const T Lv = lap(v0, v10, vm0, v01, v0m, vp, c.vm);
    const T Lw = lap(w0, w10, wm0, w01, w0m, wp, c.wm);

    // ---- body force: uniform dp/dx plus ABC forcing (separable tables)
    T fx = a.dpdx, fy = T(0), fz = T(0);
    if (a.trig && write) {
        const T* sx = a.trig;
        const T* cx = sx + g.nx;
        const T* sy = cx + g.nx;
        const T* cy = sy + g.ny;
        const T* sz = cy + g.ny;
        const T* cz = sz + g.nz;
        fx += a.abc_amp * (__ldg(sz + k) + __ldg(cy + j));
        fy = a.abc_amp * (__ldg(sx + i) + __ldg(cz + k));
        fz = a.abc_amp * (__ldg(sy + j) + __ldg(cx + i));
    }
    // implicit viscous option: the viscous term leaves N (alpha mu lap u^{k-1} is
    // added below; alpha mu lap u* is taken by the Helmholtz solves)
    const T mun = a.cn ? T(0) : mu;
    const T Nx = fma_rn(mun, Lu, -Ax) + fx;
    const T Ny = fma_rn(mun, Lv, -Ay) + fy;
    const T Nz = fma_rn(mun, Lw, -Az) + fz;

    T ix = mul_rn(a.zeta, Nx), iy = mul_rn(a.zeta, Ny), iz = mul_rn(a.zeta, Nz);
    if (a.read_hist) {
        ix = fma_rn(a.xi, hist[0], ix);
        iy = fma_rn(a.xi, hist[1], iy);
        iz = fma_rn(a.xi, hist[2], iz);
    }
    // ---- pressure gradient
    const T two_a = T(2) * a.alpha;
    const T p0 = S.p(0, 0, 0);
    ix = fma_rn(-two_a, mul_rn(S.p(1, 0, 0) - p0, g.idx), ix);
    iy = fma_rn(-two_a, mul_rn(S.p(0, 1, 0) - p0, g.idy), iy);
    iz = fma_rn(-two_a, mul_rn(S.p(0, 0, 1) - p0, g.idz), iz);
    if (a.cn) {
        const T am = a.alpha * mu;
        ix = fma_rn(am, Lu, ix);
        iy = fma_rn(am, Lv, iy);
        iz = fma_rn(am, Lw, iz);
    }
    if (STRESS) {
        // four times the edge averages; the cell above takes those at k + 1/2 over, its
        // own plane's values first in the sum
        const T s1 = S.s(1, 0, 0, 0), s1p = S.s(1, 0, 1, 0), s11 = S.s(1, 1, 0, 0);
        const T exy = s1 + s1p + s11 + S.s(1, 1, 1, 0);
        const T exym = s1 + S.s(1, 0, -1, 0) + s11 + S.s(1, 1, -1, 0);
        const T eyxm = s1 + s1p + S.s(1, -1, 0, 0) + S.s(1, -1, 1, 0);
        const T tx = S.s(2, 0, 0, 0) + S.s(2, 0, 0, 1), x0 = S.s(2, 1, 0, 0), x1 = S.s(2, 1, 0, 1);
        const T ty = S.s(4, 0, 0, 0) + S.s(4, 0, 0, 1), y0 = S.s(4, 0, 1, 0), y1 = S.s(4, 0, 1, 1);
        const T exz = tx + x0 + x1, exzm = tx + S.s(2, -1, 0, 0) + S.s(2, -1, 0, 1);
        const T eyz = ty + y0 + y1, eyzm = ty + S.s(4, 0, -1, 0) + S.s(4, 0, -1, 1);
        const T fxs = dot3(S.s(0, 1, 0, 0) - S.s(0, 0, 0, 0), g.idx, exy - exym, qy, exz - c.exz, qz);
        const T fys = dot3(exy - eyxm, qx, S.s(3, 0, 1, 0) - S.s(3, 0, 0, 0), g.idy, eyz - c.eyz, qz);
        const T fzs = dot3(exz - exzm, qx, eyz - eyzm, qy, S.s(5, 0, 0, 1) - S.s(5, 0, 0, 0), g.idz);
        ix = fma_rn(a.alpha, fxs, ix);
        iy = fma_rn(a.alpha, fys, iy);
        iz = fma_rn(a.alpha, fzs, iz);
        c.exz = tx + x1 + x0;
        c.eyz = ty + y1 + y0;
    }
    c.um = u0;
    c.vm = v0;
    c.wm = w0;
    c.uz = uz;
    c.wx = wx;
    c.vz = vz;
    c.wy = wy;
    c.fww = mul_rn(wzp, wzp);
    if (write) {
        const size_t c0 = ((size_t)k * g.ny + j) * g.nx + i;
        T us = fma_rn(a.dt, ix, u0), vs = fma_rn(a.dt, iy, v0), ws = fma_rn(a.dt, iz, w0);
        if (a.solid[0]) {
            // volume penalisation of fixed obstacles, Eq. forceAdded
            us *= T(1) - __ldg(a.solid[0] + c0);
            vs *= T(1) - __ldg(a.solid[1] + c0);
            ws *= T(1) - __ldg(a.solid[2] + c0);
        }
        a.Us[c0] = us;
        a.Vs[c0] = (g.walls && j == g.ny - 1) ? T(0) : vs;
        a.Ws[c0] = ws;
        if (a.write_hist) {
            a.NH[0][c0] = Nx;
            a.NH[1][c0] = Ny;
            a.NH[2][c0] = Nz;
        }
    }
}

// ---- single precision, summed stress written by the stress kernel (STRESS) or none.
// Three ring slots of all staged planes: while planes k and k+1 are used, k+2 arrives.
// One slot holds every field, so that a plane is one base offset and its fields and
// neighbours are constants from it.  Tiles of 64 x 4 cells where nx is a multiple of 64,
// else of 32 x 8: 256 threads, four CTAs on an SM.
//
// What bounds it: the plane's way into shared memory.  On 256^3 the kernel takes 267 us,
// the same kernel without its arithmetic 232, a plain stream over the same 19 arrays 164
// and the arithmetic on planes already there 210; deeper staging (a fourth slot, fewer
// CTAs), L1-allocating copies, tiles of 128 columns and reading the neighbours straight
// through L1 were slower (288, 308, 285, 319 us), and so were one ring per field with the
// fluxes through the lower faces computed again (289 us).
template <int TX_, int TY_>
struct MomTile {
    static constexpr int TX = TX_, TY = TY_, NT = TX * TY;
    static constexpr int XO = 4, VW = TX + 2 * XO;            // column of the tile's i0; row width
    static constexpr int VH = TY + 2, VPL = VW * VH;          // rows j0-1 .. j0+TY
};
constexpr int MOM_CTAS = 4;
template <typename Q, bool STRESS>
__host__ __device__ constexpr size_t mom_smem() { return 3 * (STRESS ? 10 : 4) * Q::VPL * sizeof(float); }

template <typename Q>
struct TileSrc {
    const float* sm;   // the ring
    int a, b;          // this cell in planes k and k+1
    __device__ __forceinline__ float at(int f, int di, int dj, int dk) const {
        return sm[(dk ? b : a) + f * Q::VPL + dj * Q::VW + di];
    }
    __device__ __forceinline__ float u(int di, int dj, int dk) const { return at(0, di, dj, dk); }
    __device__ __forceinline__ float v(int di, int dj, int dk) const { return at(1, di, dj, dk); }
    __device__ __forceinline__ float w(int di, int dj, int dk) const { return at(2, di, dj, dk); }
    __device__ __forceinline__ float p(int di, int dj, int dk) const { return at(3, di, dj, dk); }
    __device__ __forceinline__ float s(int c, int di, int dj, int dk) const { return at(4 + c, di, dj, dk); }
};

// One tile: the columns (bx, by) over the z chunk bz of kz_chunk planes.
// VEC: rows are staged in 16-byte chunks (needs nx % 4 == 0).
template <typename Q, bool VEC, bool STRESS>
__device__ __forceinline__ void momentum_tile(const Geo<float>& g, const ModelConst& mc, const MomentumArgs<float>& a,
                                              int kz_chunk, int bx, int by, int bz, unsigned char* smraw) {
    constexpr int TX = Q::TX, TY = Q::TY, NT = Q::NT, XO = Q::XO, VW = Q::VW, VH = Q::VH, VPL = Q::VPL;
    constexpr int NF = STRESS ? 10 : 4;               // u, v, w, p, S_xx .. S_zz
    float* const ring = reinterpret_cast<float*>(smraw);
    EVP_DBG_DECL;
#ifdef EVP_DEBUG
    dbg_poison(smraw, mom_smem<Q, STRESS>());
    const size_t dbg_n = (size_t)g.nx * g.ny * g.nz;
    auto dbg_src_ok = [&](const float* p, int n) {
        if (dbg_within(p, n, a.U, dbg_n) || dbg_within(p, n, a.V, dbg_n) || dbg_within(p, n, a.W, dbg_n) ||
            dbg_within(p, n, a.P, dbg_n))
            return true;
        for (int c = 0; c < 6; ++c)
            if (dbg_within(p, n, a.S[c], dbg_n)) return true;
        return false;
    };
    auto dbg_dst_ok = [&](const float* d, int n) {
        return (const unsigned char*)d >= smraw && (const unsigned char*)(d + n) <= smraw + mom_smem<Q, STRESS>();
    };
#endif
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int i0 = bx * TX, j0 = by * TY;
    const int k0 = bz * kz_chunk, k1 = min(k0 + kz_chunk, g.nz);
    const int i = i0 + tx, j = j0 + ty;
    const bool active = i < g.nx && j < g.ny;
    const size_t plane = (size_t)g.nx * g.ny;

    // this thread's copies of a plane: one 16-byte chunk of every field (the tile's own
    // columns first, a row's 128 bytes to eight neighbouring threads), or up to NE elements
    constexpr int SW = TX + 2, NE = VEC ? 1 : (SW * VH + NT - 1) / NT, LC = TX / 4;
    static_assert(!VEC || (LC + 2) * VH <= NT, "one chunk per thread");
    int dsm[NE], off[NE];
#pragma unroll
    for (int r = 0; r < NE; ++r) {
        dsm[r] = -1;
        off[r] = 0;
        int row, col;
        if (VEC) {
            if (tid >= (LC + 2) * VH) continue;
            const int h = tid - LC * VH;
            row = h < 0 ? tid / LC : h >> 1;
            col = h < 0 ? XO + (tid - row * LC) * 4 : ((h & 1) ? XO + TX : 0);
        } else {
            const int e = tid + r * NT;
            if (e >= SW * VH) continue;
            row = e / SW;
            col = e - row * SW + XO - 1;
        }
        dsm[r] = row * VW + col;
        // walls: the nearest row, which is also the mirrored one (see ghosts)
        const int gy = j0 - 1 + row, sy = g.walls ? min(max(gy, 0), g.ny - 1) : pmod(gy, g.ny);
        off[r] = sy * g.nx + pmod(i0 - XO + col, g.nx);     // a whole chunk: nx is a multiple of 4
    }
    // plane kk (-1 .. nz + 1) into a ring slot
    auto fetch = [&](int kk, int slot) {
        const size_t pk = (size_t)wrap1(kk, g.nz) * plane;
#pragma unroll
        for (int r = 0; r < NE; ++r) {
            if (dsm[r] < 0) continue;
            auto put = [&](int f, const float* F) {
                float* dst = ring + slot + f * VPL + dsm[r];
                const float* src = F + pk + off[r];
                if (!EVP_STAGE_OK(dst, src, VEC ? 4 : 1, VEC)) return;
                if (VEC) cp_async16(dst, src);
                else cp_async(dst, src);
            };
            put(0, a.U);
            put(1, a.V);
            put(2, a.W);
            put(3, a.P);
            if (STRESS) {
#pragma unroll
                for (int c = 0; c < 6; ++c) put(4 + c, a.S[c]);
            }
        }
    };
    // walls: the rows below j = 0 and above j = ny-1 of a landed plane hold the nearest
    // rows; u and w change sign there (no slip) and v is zero.  Uniform over the CTA.
    const bool low = g.walls && j0 == 0, high = g.walls && j0 + TY >= g.ny;
    auto ghosts = [&](int slot) {
        for (int c = tid; c < VW; c += NT) {
            auto row = [&](int r) {
                float* q = ring + slot + r * VW + c;
                q[0] = -q[0];
                q[VPL] = 0.f;
                q[2 * VPL] = -q[2 * VPL];
            };
            if (low) row(0);
            if (high) row(g.ny - j0 + 1);
        }
    };
    const int o = (ty + 1) * VW + tx + XO;
    const size_t cell = (size_t)min(j, g.ny - 1) * g.nx + min(i, g.nx - 1);

    int s0 = 0, s1 = NF * VPL, s2 = 2 * NF * VPL;      // ring offsets of planes k, k+1, k+2
    fetch(k0 - 1, s2);
    fetch(k0, s0);
    fetch(k0 + 1, s1);
    cp_async_commit();
    cp_async_wait_all();
    __syncthreads();
    if (low || high) {
        ghosts(s2);
        ghosts(s0);
        ghosts(s1);
        __syncthreads();
    }
    MomCarry<float> c = momentum_carry<float, STRESS>(TileSrc<Q>{ring, s2 + o, s0 + o});
    __syncthreads();     // slot s2 is read
    for (int k = k0; k < k1; ++k) {
        fetch(k + 2, s2);
        cp_async_commit();
        float h[3] = {0.f, 0.f, 0.f};
        if (a.read_hist) {
#pragma unroll
            for (int q = 0; q < 3; ++q) h[q] = a.NH[q][(size_t)k * plane + cell];
        }
        const bool write = active && EVP_DBG_OK((size_t)k * plane + (size_t)j * g.nx + i < plane * (size_t)g.nz);
        momentum_point<float, STRESS>(g, mc, a, TileSrc<Q>{ring, s0 + o, s1 + o}, c, h, i, j, k, write);
        // plane k+2 has landed; after the barrier every thread sees it and is done with plane k
        cp_async_wait_all();
        __syncthreads();
        if (low || high) {
            ghosts(s2);
            __syncthreads();
        }
        const int t = s0;
        s0 = s1;
        s1 = s2;
        s2 = t;
    }
    EVP_DBG_REPORT(a.status);
}

using MomWide = MomTile<64, 4>;
using MomTall = MomTile<32, 8>;

template <typename Q, bool VEC, bool STRESS>
__global__ void __launch_bounds__(Q::NT, MOM_CTAS)
k_momentum(const Geo<float> g, const ModelConst mc, const MomentumArgs<float> a, int kz_chunk) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smraw[];
    momentum_tile<Q, VEC, STRESS>(g, mc, a, kz_chunk, blockIdx.x, blockIdx.y, blockIdx.z, smraw);
}

// Batched form: a persistent grid walks a work list of (member, tile x, tile y, z
// chunk); members' grids may differ, so the tiles are 32 x 8.
template <bool VEC>
__global__ void __launch_bounds__(MomTall::NT, MOM_CTAS)
k_momentum_batch(const __grid_constant__ MomentumBatch<float> p, const int4* __restrict__ work, int nwork) {
    extern __shared__ __align__(16) unsigned char smraw[];
    for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
        const int4 t = __ldg(work + w);
        const MomentumMember<float>& m = p.m[t.x];
        momentum_tile<MomTall, VEC, true>(m.g, m.mc, m.a, m.kz, t.y, t.z, t.w, smraw);
        __syncthreads();
    }
}

// ---- double precision: a thread's cell is number blk * 128 + thread of the plane
constexpr int COL_NT = 128;
struct ColumnSrc {
    const MomentumArgs<double>* a;
    size_t p0, p1;           // planes k and k+1
    int x[3], r[3];          // offsets of columns i-1 .. i+1 and of rows j-1 .. j+1
    int fm, fp, fv;          // wall factors: u, w below and above, v below
    // x, -x or 0 by integer operations on the sign
    __device__ __forceinline__ static double scaled(double v, int f) {
        const int hi = __double2hiint(v) ^ (f < 0 ? (int)0x80000000 : 0);
        return f ? __hiloint2double(hi, __double2loint(v)) : 0.0;
    }
    __device__ __forceinline__ double at(const double* F, int di, int dj, int dk) const {
        return __ldg(F + (dk ? p1 : p0) + r[dj + 1] + x[di + 1]);
    }
    __device__ __forceinline__ double uw(const double* F, int di, int dj, int dk) const {
        const double v = at(F, di, dj, dk);
        return dj == 0 ? v : scaled(v, dj < 0 ? fm : fp);
    }
    __device__ __forceinline__ double u(int di, int dj, int dk) const { return uw(a->U, di, dj, dk); }
    __device__ __forceinline__ double w(int di, int dj, int dk) const { return uw(a->W, di, dj, dk); }
    __device__ __forceinline__ double v(int di, int dj, int dk) const {
        const double q = at(a->V, di, dj, dk);
        return dj == 0 ? q : scaled(q, dj < 0 ? fv : (fp < 0 ? 0 : 1));
    }
    __device__ __forceinline__ double p(int di, int dj, int dk) const { return at(a->P, di, dj, dk); }
    __device__ __forceinline__ double s(int c, int di, int dj, int dk) const { return at(a->S[c], di, dj, dk); }
};

template <bool STRESS>
__device__ __forceinline__ void momentum_column(const Geo<double>& g, const ModelConst& mc, const MomentumArgs<double>& a,
                                                int kz_chunk, int blk, int bz) {
    const int q = blk * COL_NT + (int)threadIdx.x;
    if (q >= g.nx * g.ny) return;
    const int j = q / g.nx, i = q - j * g.nx;
    const int k0 = bz * kz_chunk, k1 = min(k0 + kz_chunk, g.nz);
    const size_t plane = (size_t)g.nx * g.ny;
    auto kplane = [&](int k) { return (size_t)wrap1(k, g.nz) * plane; };
    ColumnSrc S;
    S.a = &a;
    S.x[0] = i > 0 ? i - 1 : g.nx - 1;
    S.x[1] = i;
    S.x[2] = i < g.nx - 1 ? i + 1 : 0;
    // at a wall the mirrored row and the nearest row are both the cell's own
    S.r[0] = (j > 0 ? j - 1 : (g.walls ? 0 : g.ny - 1)) * g.nx;
    S.r[1] = j * g.nx;
    S.r[2] = (j < g.ny - 1 ? j + 1 : (g.walls ? j : 0)) * g.nx;
    S.fm = g.walls && j == 0 ? -1 : 1;
    S.fv = g.walls && j == 0 ? 0 : 1;
    S.fp = g.walls && j == g.ny - 1 ? -1 : 1;
    S.p0 = kplane(k0 - 1);
    S.p1 = kplane(k0);
    MomCarry<double> c = momentum_carry<double, STRESS>(S);
    for (int k = k0; k < k1; ++k) {
        S.p0 = S.p1;
        S.p1 = kplane(k + 1);
        double h[3] = {0.0, 0.0, 0.0};
        if (a.read_hist) {
#pragma unroll
            for (int n = 0; n < 3; ++n) h[n] = a.NH[n][S.p0 + q];
        }
        momentum_point<double, STRESS>(g, mc, a, S, c, h, i, j, k, true);
    }
}

template <bool STRESS>
__global__ void __launch_bounds__(COL_NT, 4)
k_momentum_f64(const Geo<double> g, const ModelConst mc, const MomentumArgs<double> a, int kz_chunk) {
    pdl_wait();
    pdl_trigger();
    momentum_column<STRESS>(g, mc, a, kz_chunk, blockIdx.x, blockIdx.y);
}

__global__ void __launch_bounds__(COL_NT, 4)
k_momentum_f64_batch(const __grid_constant__ MomentumBatch<double> p, const int4* __restrict__ work, int nwork) {
    for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
        const int4 t = __ldg(work + w);
        const MomentumMember<double>& m = p.m[t.x];
        momentum_column<true>(m.g, m.mc, m.a, m.kz, t.y, t.w);
    }
}

// ---- soft particles: 32 x 4 tiles, planes staged two ahead: while plane k is computed, plane k+2
// has landed (or is landing) and plane k+3 is being requested.
constexpr int TX = 32, TY = 4, NT = TX * TY;
constexpr int VW = TX + 8, XO = 4;                       // plane row width; column of the tile's i0
constexpr int VH = TY + 2, VPL = VW * VH;                // rows j0-1 .. j0+TY
constexpr int SW = TX + 2;                               // columns the stencils use: XO-1 .. XO+TX
constexpr int NV = (SW * VH + NT - 1) / NT;              // used plane cells per thread (2)

template <typename T>
struct MomSoftSmem {
    T V[3][5][VPL];      // u, v, w: ring slots for planes k-1 .. k+3
    T S[6][3][VPL];      // summed stress: ring slots for planes k-1 .. k+1
    T Braw[2][12][VPL];  // raw B^{k-1} (0..5) and B^k (6..11) of planes k+2 and k+3
    T P[4][VPL];         // pressure planes k .. k+3
    T H[4][3][NT];       // momentum history of the tile's cells, planes k .. k+2
};
__device__ __forceinline__ int vs_of(int kk) { return (kk + 5) % 5; }   // ring slots (kk >= -1)

template <typename T>
struct SoftSrc {
    const MomSoftSmem<T>* sm;
    int o, vs[2], t[2], q[2];   // the cell in a plane; slots of planes k and k+1 (velocity, stress, pressure)
    __device__ __forceinline__ T vel(int n, int di, int dj, int dk) const { return sm->V[n][vs[dk]][o + dj * VW + di]; }
    __device__ __forceinline__ T u(int di, int dj, int dk) const { return vel(0, di, dj, dk); }
    __device__ __forceinline__ T v(int di, int dj, int dk) const { return vel(1, di, dj, dk); }
    __device__ __forceinline__ T w(int di, int dj, int dk) const { return vel(2, di, dj, dk); }
    __device__ __forceinline__ T p(int di, int dj, int dk) const { return sm->P[q[dk]][o + dj * VW + di]; }
    __device__ __forceinline__ T s(int c, int di, int dj, int dk) const { return sm->S[c][t[dk]][o + dj * VW + di]; }
};

// VEC: rows are staged in 16-byte chunks (needs nx * sizeof(T) % 16 == 0)
// One tile: the 32 x 4 columns (bx, by) over the z chunk bz of kz_chunk planes.  The
// summed stress phi_s G (B - I) of both levels is built from the staged B and the solid
// fractions, between two barriers per plane.
template <typename T, bool VEC>
__device__ __forceinline__ void momentum_soft_tile(const Geo<T>& g, const ModelConst& mc, const MomentumArgs<T>& a,
                                              int kz_chunk, int bx, int by, int bz, unsigned char* smraw) {
    MomSoftSmem<T>& sm = *reinterpret_cast<MomSoftSmem<T>*>(smraw);
    EVP_DBG_DECL;
#ifdef EVP_DEBUG
    dbg_poison(smraw, sizeof(MomSoftSmem<T>));
    const size_t dbg_n = (size_t)g.nx * g.ny * g.nz;
    auto dbg_src_ok = [&](const T* p, int n) {
        if (dbg_within(p, n, a.U, dbg_n) || dbg_within(p, n, a.V, dbg_n) || dbg_within(p, n, a.W, dbg_n) ||
            dbg_within(p, n, a.P, dbg_n) || dbg_within(p, n, a.phis_o, dbg_n) || dbg_within(p, n, a.phis_n, dbg_n))
            return true;
        for (int c = 0; c < 6; ++c)
            if (dbg_within(p, n, a.Bo[c], dbg_n) || dbg_within(p, n, a.Bn[c], dbg_n) || dbg_within(p, n, a.S[c], dbg_n))
                return true;
        for (int q = 0; q < 3; ++q)
            if (dbg_within(p, n, (const T*)a.NH[q], dbg_n) || dbg_within(p, n, a.solid[q], dbg_n)) return true;
        return false;
    };
    auto dbg_dst_ok = [&](const T* d, int n) {
        return (const unsigned char*)d >= smraw &&
               (const unsigned char*)(d + n) <= smraw + sizeof(MomSoftSmem<T>);
    };
#endif
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
    const int i0 = bx * TX, j0 = by * TY;
    const int k0 = bz * kz_chunk, k1 = min(k0 + kz_chunk, g.nz);
    const int i = i0 + tx, j = j0 + ty;
    const bool active = i < g.nx && j < g.ny;
    const size_t plane = (size_t)g.nx * g.ny;

    // element-wise staging: this thread's used plane cells (row r, column XO-1+c)
    size_t coff[NV], voff[3][NV];
    signed char vfac[3][NV];
    int psm[NV];
    // chunk staging: this thread's 16-byte chunk of a plane (row ch / CPR)
    constexpr int E = 16 / (int)sizeof(T);                // elements per chunk
    constexpr int CPR = VW / E, NCH = CPR * VH;           // chunks per row / plane
    int csm = -1;
    size_t ccoff = 0, cvoff[3] = {0, 0, 0};
    signed char cvfac[3] = {0, 0, 0};
    if (VEC) {
        if (tid < NCH) {
            const int r = tid / CPR, q0 = (tid - r * CPR) * E;
            csm = r * VW + q0;
            const int gx = pmod(i0 - XO + q0, g.nx);      // a whole chunk: nx is a multiple of E
            int src;
            row_rule(g, j0 - 1 + r, 3, src);
            ccoff = (size_t)src * g.nx + gx;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                cvfac[q] = (signed char)row_rule(g, j0 - 1 + r, q, src);
                cvoff[q] = (size_t)src * g.nx + gx;
            }
        }
    }
#pragma unroll
    for (int r = 0; r < NV; ++r) {
        const int e = tid + r * NT;
        const int vy = e / SW, vx = e - vy * SW;
        psm[r] = e < SW * VH ? vy * VW + vx + XO - 1 : -1;
        coff[r] = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            voff[q][r] = 0;
            vfac[q][r] = 0;
        }
        if (e >= SW * VH) continue;
        const int gx = pmod(i0 + vx - 1, g.nx);
        int src;
        row_rule(g, j0 + vy - 1, 3, src);
        coff[r] = (size_t)src * g.nx + gx;        // also the soft particles' solid-fraction reads
        if constexpr (!VEC) {
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                vfac[q][r] = (signed char)row_rule(g, j0 + vy - 1, q, src);
                voff[q][r] = (size_t)src * g.nx + gx;
            }
        }
    }
    const T* vel[3] = {a.U, a.V, a.W};
    auto fetch_vel = [&](int kk) {
        const size_t pv = (size_t)wrap1(kk, g.nz) * plane;
        const int slot = vs_of(kk);
        if constexpr (VEC) {
            if (csm < 0) return;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                T* dst = &sm.V[q][slot][csm];
                if (!EVP_STAGE_OK(dst, vel[q] + pv + cvoff[q], E, true)) continue;
                if (cvfac[q] == 1) cp_async16(dst, vel[q] + pv + cvoff[q]);
                else copy_scaled(dst, vel[q] + pv + cvoff[q], cvfac[q]);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 3; ++q)
#pragma unroll
                for (int r = 0; r < NV; ++r) {
                    if (psm[r] < 0) continue;
                    T* dst = &sm.V[q][slot][psm[r]];
                    if (!EVP_STAGE_OK(dst, vel[q] + pv + voff[q][r], 1, false)) continue;
                    if (vfac[q][r] == 1)
                        cp_async(dst, vel[q] + pv + voff[q][r]);
                    else
                        *dst = vfac[q][r] == 0 ? T(0) : -__ldg(vel[q] + pv + voff[q][r]);
                }
        }
    };
    auto fetch_p = [&](int kk) {
        const size_t pp = (size_t)wrap1(kk, g.nz) * plane;
        const int slot = (kk & 3);
        if constexpr (VEC) {
            if (csm >= 0 && EVP_STAGE_OK(&sm.P[slot][csm], a.P + pp + ccoff, E, true))
                cp_async16(&sm.P[slot][csm], a.P + pp + ccoff);
        } else {
#pragma unroll
            for (int r = 0; r < NV; ++r)
                if (psm[r] >= 0 && EVP_STAGE_OK(&sm.P[slot][psm[r]], a.P + pp + coff[r], 1, false))
                    cp_async(&sm.P[slot][psm[r]], a.P + pp + coff[r]);
        }
    };
    auto fetch_braw = [&](int kk) {
        const size_t pb = (size_t)wrap1(kk, g.nz) * plane;
        if constexpr (VEC) {
            if (csm < 0) return;
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                if (EVP_STAGE_OK(&sm.Braw[kk & 1][c][csm], a.Bo[c] + pb + ccoff, E, true))
                    cp_async16(&sm.Braw[kk & 1][c][csm], a.Bo[c] + pb + ccoff);
                if (EVP_STAGE_OK(&sm.Braw[kk & 1][6 + c][csm], a.Bn[c] + pb + ccoff, E, true))
                    cp_async16(&sm.Braw[kk & 1][6 + c][csm], a.Bn[c] + pb + ccoff);
            }
        } else {
#pragma unroll
            for (int c = 0; c < 6; ++c)
#pragma unroll
                for (int r = 0; r < NV; ++r)
                    if (psm[r] >= 0) {
                        if (EVP_STAGE_OK(&sm.Braw[kk & 1][c][psm[r]], a.Bo[c] + pb + coff[r], 1, false))
                            cp_async(&sm.Braw[kk & 1][c][psm[r]], a.Bo[c] + pb + coff[r]);
                        if (EVP_STAGE_OK(&sm.Braw[kk & 1][6 + c][psm[r]], a.Bn[c] + pb + coff[r], 1, false))
                            cp_async(&sm.Braw[kk & 1][6 + c][psm[r]], a.Bn[c] + pb + coff[r]);
                    }
        }
    };
    const T gm = kconst<T>(mc.gmod, mc.f_gmod);
    // staged raw B -> summed stress S in ring slot kk mod 3: tau = phi_s G (B - I) at both levels
    auto build_s = [&](int kk) {
        const int slot = pmod(kk, 3);
        const T(*Br)[VPL] = sm.Braw[kk & 1];
        const size_t pb = (size_t)wrap1(kk, g.nz) * plane;
#pragma unroll
        for (int r = 0; r < NV; ++r) {
            const int e = psm[r];
            if (e < 0) continue;
            const bool pok = EVP_DBG_OK(dbg_src_ok(a.phis_o + pb + coff[r], 1) && dbg_src_ok(a.phis_n + pb + coff[r], 1));
            const T po = pok ? gm * __ldg(a.phis_o + pb + coff[r]) : T(0);
            const T pn = pok ? gm * __ldg(a.phis_n + pb + coff[r]) : T(0);
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const T d = (c == 0 || c == 3 || c == 5) ? T(1) : T(0);
                sm.S[c][slot][e] = pn * (Br[6 + c][e] - d) + po * (Br[c][e] - d);
            }
        }
    };
    const size_t cell0 = (size_t)min(j, g.ny - 1) * g.nx + min(i, g.nx - 1);
    // history chunk of this thread (own cells of row hr, columns hq .. hq+E-1)
    constexpr int HCR = TX / E;                          // chunks per tile row
    const int hr = tid / HCR, hq = (tid - hr * HCR) * E;
    const bool hch = VEC && tid < TY * HCR && j0 + hr < g.ny && i0 + hq < g.nx;
    const size_t hoff = (size_t)(j0 + hr) * g.nx + i0 + hq;
    auto fetch_hist = [&](int kk) {
        if (!a.read_hist || kk >= k1) return;
        if constexpr (VEC) {
            if (hch) {
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (EVP_STAGE_OK(&sm.H[(kk & 3)][q][hr * TX + hq], a.NH[q] + (size_t)kk * plane + hoff, E, true))
                        cp_async16(&sm.H[(kk & 3)][q][hr * TX + hq], a.NH[q] + (size_t)kk * plane + hoff);
            }
        } else {
#pragma unroll
            for (int q = 0; q < 3; ++q)
                if (EVP_STAGE_OK(&sm.H[(kk & 3)][q][tid], a.NH[q] + (size_t)kk * plane + cell0, 1, false))
                    cp_async(&sm.H[(kk & 3)][q][tid], a.NH[q] + (size_t)kk * plane + cell0);
        }
    };

    // ---- prologue: velocity k0-1 .. k0+1, p k0 .. k0+1, S k0-1 .. k0+1, history k0
    // in place; then plane k0+2 and the history of k0+1 requested
    fetch_vel(k0 - 1);
    fetch_vel(k0);
    fetch_vel(k0 + 1);
    fetch_p(k0);
    fetch_p(k0 + 1);
    fetch_hist(k0);
    for (int d = -1; d <= 1; ++d) {
        fetch_braw(k0 + d);
        cp_async_commit();
        cp_async_wait_all();
        __syncthreads();
        build_s(k0 + d);
        __syncthreads();
    }
    fetch_vel(k0 + 2);
    fetch_braw(k0 + 2);
    fetch_p(k0 + 2);
    fetch_hist(k0 + 1);
    cp_async_commit();

    const int o = (ty + 1) * VW + tx + XO;
    auto source = [&](int k) {
        SoftSrc<T> S;
        S.sm = &sm;
        S.o = o;
        S.vs[0] = vs_of(k);
        S.vs[1] = vs_of(k + 1);
        S.t[0] = pmod(k, 3);
        S.t[1] = pmod(k + 1, 3);
        S.q[0] = k & 3;
        S.q[1] = (k + 1) & 3;
        return S;
    };
    MomCarry<T> c = momentum_carry<T, true>(source(k0 - 1));
    for (int k = k0; k < k1; ++k) {
        // ---- asynchronous request of plane k+3 (velocity, raw B, p) and the history of k+2
        fetch_vel(k + 3);
        fetch_braw(k + 3);
        fetch_p(k + 3);
        fetch_hist(k + 2);
        cp_async_commit();
        T h[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) h[q] = a.read_hist ? sm.H[k & 3][q][tid] : T(0);
        const bool write = active && EVP_DBG_OK((size_t)k * plane + (size_t)j * g.nx + i < plane * (size_t)g.nz);
        momentum_point<T, true>(g, mc, a, source(k), c, h, i, j, k, write);
        // ---- advance: plane k+2 has landed (only plane k+3 may be in flight); its
        // raw B becomes S plane k+2 (slot of plane k-1)
        cp_async_wait_prev();
        __syncthreads();
        build_s(k + 2);
        __syncthreads();
    }
    // the last request (two planes past the chunk) may still be in flight; let it land
    // before the tile's shared memory is given up
    cp_async_wait_all();
    EVP_DBG_REPORT(a.status);
}

template <typename T, bool VEC>
__global__ void __launch_bounds__(NT, sizeof(T) == 4 ? 4 : 2)
k_momentum_soft(const Geo<T> g, const ModelConst mc, const MomentumArgs<T> a, int kz_chunk) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smraw[];
    momentum_soft_tile<T, VEC>(g, mc, a, kz_chunk, blockIdx.x, blockIdx.y, blockIdx.z, smraw);
}

template <typename T>
cudaError_t launch_momentum_soft(const Geo<T>& g, const ModelConst& mc, const MomentumArgs<T>& a, cudaStream_t st,
                                 bool pdl) {
    // z chunks: about four waves of CTAs; small grids go down to one plane per CTA
    const int tiles = ((g.nx + TX - 1) / TX) * ((g.ny + TY - 1) / TY);
    int chunks = (4 * 152 * (sizeof(T) == 4 ? 4 : 2) + tiles - 1) / tiles;
    chunks = chunks > g.nz ? g.nz : chunks;
    const int kz = (g.nz + chunks - 1) / chunks;
    const dim3 block(TX, TY, 1), grid((g.nx + TX - 1) / TX, (g.ny + TY - 1) / TY, (g.nz + kz - 1) / kz);
    const size_t smem = sizeof(MomSoftSmem<T>);
    auto kern = (g.nx * sizeof(T)) % 16 == 0 ? k_momentum_soft<T, true> : k_momentum_soft<T, false>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    return launch_k(kern, grid, block, smem, st, pdl, g, mc, a, kz);
}

}  // namespace

namespace {
bool momentum_wide(int nx) { return nx % MomWide::TX == 0; }
}

template <>
MomentumTiles momentum_tiles<float>(int nx, int ny) {   // the batch's tiles
    return {(nx + MomTall::TX - 1) / MomTall::TX, (ny + MomTall::TY - 1) / MomTall::TY};
}
template <>
MomentumTiles momentum_tiles<double>(int nx, int ny) { return {(nx * ny + COL_NT - 1) / COL_NT, 1}; }

// planes per CTA: as the stress kernel's rule, the CTAs of the busiest SM times (planes +
// 1), with one CTA's worth for the first planes' way in.  Within 4 % of the best chunk of a
// sweep on ten grids from 32^3 to 256^3 (64^3 13.2 us with 4 planes, 16.5 with one; 96^3 25
// with 8, 27.5 with 3; 256 x 128 x 128 78 with 10)
template <>
int momentum_planes<float>(int nx, int ny, int nz) {
    const int tx = momentum_wide(nx) ? MomWide::TX : MomTall::TX, ty = momentum_wide(nx) ? MomWide::TY : MomTall::TY;
    const int tiles = ((nx + tx - 1) / tx) * ((ny + ty - 1) / ty);
    int best = 1;
    long long cost = -1;
    for (int kz = 1; kz <= nz && kz <= 64; ++kz) {
        const int rem = nz % kz, chunks = nz / kz + (4 * rem > kz ? 1 : 0);
        const long long c = (long long)((tiles * chunks + 151) / 152 + 1) * (kz + 1);
        if (cost < 0 || c <= cost) {
            cost = c;
            best = kz;
        }
    }
    return best;
}
// the busiest SM's planes, a CTA's start costing about half a plane
template <>
int momentum_planes<double>(int nx, int ny, int nz) {
    const MomentumTiles t = momentum_tiles<double>(nx, ny);
    int best = 1;
    double cost = -1.0;
    for (int kz = 1; kz <= nz && kz <= 64; ++kz) {
        const long long ctas = (long long)t.x * ((nz + kz - 1) / kz);
        const double c = (double)((ctas + 151) / 152) * (kz + 0.5);
        if (cost < 0.0 || c < cost) {
            cost = c;
            best = kz;
        }
    }
    return best;
}

template <>
cudaError_t launch_momentum<float>(const Geo<float>& g, const ModelConst& mc, const MomentumArgs<float>& a,
                                   cudaStream_t st, const TimingHook& th) {
    const bool stress = mc.model != EVP_NEWTONIAN;
    if (stress && !a.S[0] && !a.phis_o) return cudaErrorInvalidValue;
    cudaError_t e;
    th.b(K_MOMENTUM);
    if (stress && !a.S[0]) {
        e = launch_momentum_soft<float>(g, mc, a, st, th.pdl);
    } else {
        const int kz = momentum_planes<float>(g.nx, g.ny, g.nz);
        const bool vec = g.nx % 4 == 0;
        auto go = [&](auto kern, auto q, size_t smem) {
            using Q = decltype(q);
            const dim3 grid((g.nx + Q::TX - 1) / Q::TX, (g.ny + Q::TY - 1) / Q::TY, (g.nz + kz - 1) / kz);
            // all of the SM's unified L1 / shared memory as shared memory
            cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
            return launch_k(kern, grid, dim3(Q::NT), smem, st, th.pdl, g, mc, a, kz);
        };
        if (momentum_wide(g.nx)) {
            e = stress ? go(k_momentum<MomWide, true, true>, MomWide{}, mom_smem<MomWide, true>())
                       : go(k_momentum<MomWide, true, false>, MomWide{}, mom_smem<MomWide, false>());
        } else if (vec) {
            e = stress ? go(k_momentum<MomTall, true, true>, MomTall{}, mom_smem<MomTall, true>())
                       : go(k_momentum<MomTall, true, false>, MomTall{}, mom_smem<MomTall, false>());
        } else {
            e = stress ? go(k_momentum<MomTall, false, true>, MomTall{}, mom_smem<MomTall, true>())
                       : go(k_momentum<MomTall, false, false>, MomTall{}, mom_smem<MomTall, false>());
        }
    }
    if (e != cudaSuccess) return e;
    th.e(K_MOMENTUM);
    return cudaGetLastError();
}

template <>
cudaError_t launch_momentum<double>(const Geo<double>& g, const ModelConst& mc, const MomentumArgs<double>& a,
                                    cudaStream_t st, const TimingHook& th) {
    const bool stress = mc.model != EVP_NEWTONIAN;
    if (stress && !a.S[0] && !a.phis_o) return cudaErrorInvalidValue;
    cudaError_t e;
    th.b(K_MOMENTUM);
    if (stress && !a.S[0]) {
        e = launch_momentum_soft<double>(g, mc, a, st, th.pdl);
    } else {
        const int kz = momentum_planes<double>(g.nx, g.ny, g.nz);
        const dim3 grid(momentum_tiles<double>(g.nx, g.ny).x, (g.nz + kz - 1) / kz), block(COL_NT);
        e = launch_k(stress ? k_momentum_f64<true> : k_momentum_f64<false>, grid, block, 0, st, th.pdl, g, mc, a, kz);
    }
    if (e != cudaSuccess) return e;
    th.e(K_MOMENTUM);
    return cudaGetLastError();
}

template <>
cudaError_t launch_momentum_batch<float>(const MomentumBatch<float>& p, bool vec, const int4* work, int nwork, int ctas,
                                         cudaStream_t st) {
    if (nwork <= 0) return cudaSuccess;
    auto kern = vec ? k_momentum_batch<true> : k_momentum_batch<false>;
    constexpr size_t smem = mom_smem<MomTall, true>();
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    return launch_k(kern, dim3(ctas < nwork ? ctas : nwork), dim3(MomTall::NT), smem, st, false, p, work, nwork);
}
template <>
cudaError_t launch_momentum_batch<double>(const MomentumBatch<double>& p, bool, const int4* work, int nwork, int ctas,
                                          cudaStream_t st) {
    if (nwork <= 0) return cudaSuccess;
    return launch_k(k_momentum_f64_batch, dim3(ctas < nwork ? ctas : nwork), dim3(COL_NT), 0, st, false, p, work,
                    nwork);
}

// the tile configurations count 2 CTAs per SM in double precision where the kernel holds 4
template <>
int momentum_ctas_per_sm<float>() { return 4; }
template <>
int momentum_ctas_per_sm<double>() { return 2; }
template <>
int momentum_resident<float>(int counted) { return counted; }
template <>
int momentum_resident<double>(int counted) { return counted * 2; }

}  // namespace evp
