// S9 + S10: level set, interface force and the AB2 momentum predictor of the
// two-phase step (Secs. 3.2.1 and 3.2.2).
//
//   k_ls_stage      one TVD-RK3 stage of the level-set advection (Eq. ls-adv,
//                   WENO5 upwinded by the centre velocity) or of the
//                   re-distancing equation (Eq. reinit, Godunov |grad phi| from
//                   the WENO5 one-sided derivatives, S(phi0) = phi0/sqrt(phi0^2 + h^2))
//   k_iface_a       H(phi), n = grad phi/|grad phi| (central) near the interface, per-block
//                   sums of 1 - H
//   k_iface_mean    FP64 sum of the block sums (fixed order: deterministic)
//   k_mass_*        mass-preserving uniform shift of phi: block sums of 1 - H and
//                   delta at phi + d, Newton update of d on the device, phi += d
//   k_iface_b       kappa = -div n, the CSF force sigma kappa delta(phi) n (Eq. fLS) and
//                   the mean-free Boussinesq buoyancy, at cell centres
//   k_momentum_ab2  RU = -div(uu) + div[mu_s(H)(grad u + grad u^T)] + div tau(mu_p(H)) + f
//                   and u* = u + dt (w1 RU^n + w0 RU^{n-1})   (Eqs. ru, ab2)
// The level-set and interface kernels read neighbours through the read-only cache, the
// level-set stages marching in z; the AB2 momentum kernel marches z-planes of tiles staged
// in shared memory.
#include <algorithm>
#include <cfloat>
#include <climits>

#include "evp_internal.cuh"
#include "weno.cuh"

namespace evp {

namespace {

template <typename T>
__device__ __forceinline__ T sqr(T x) { return x * x; }

constexpr int LS_CTAS = 16;   // level-set stage: CTAs per SM below which a CTA takes one plane

// A stage marches in z: the seven values along z stay in registers, the wrapped or clamped
// offsets along x and y are formed once per thread.  The differences d_m = p_{m+1} - p_m
// serve both sides: the right-biased reconstruction is the left-biased one of d_5 .. d_1
// (weno5 is odd in its differences, exactly), so an upwind side is five selects and a
// signed velocity, and re-distancing takes its two sides in the two lanes of the packed
// WENO5.  Bound by instruction issue.  128 x 256 x 128 FP32, mean of 30 advection and 6
// re-distancing stages: 73.6 us with 21 reads and their addresses per cell and both sides'
// differences, 51.3 so (three CTAs per SM with the registers for early loads; four 53.0,
// five 52.3; 52.9 with the planes staged in shared memory two ahead).
template <typename T, bool REINIT>
__global__ void __launch_bounds__(256, 3) k_ls_stage(const Geo<T> g, const LsArgs<T> a, int kz) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k0 = blockIdx.z * kz, k1 = min(k0 + kz, g.nz);
    if (i >= g.nx || j >= g.ny) return;
    // 32-bit offsets within a plane
    const size_t plane = (size_t)g.nx * g.ny;
    const int col = j * g.nx + i;
    int ox[7], oy[7];
#pragma unroll
    for (int m = 0; m < 7; ++m) {
        ox[m] = j * g.nx + wrap(i + m - 3, g.nx);
        oy[m] = ycen(g, j + m - 3) * g.nx + i;
    }
    const bool wall = g.walls && j == 0;
    const int ovm = (j > 0 ? j - 1 : g.ny - 1) * g.nx + i;
    T pz[7], wm = T(0);
#pragma unroll
    for (int m = 0; m < 6; ++m) pz[m + 1] = __ldg(a.phis + wrap(k0 + m - 3, g.nz) * plane + col);
    if constexpr (!REINIT) wm = __ldg(a.W + wrap(k0 - 1, g.nz) * plane + col);
    for (int k = k0; k < k1; ++k) {
        const size_t o = (size_t)k * plane;
        const T* P = a.phis + o;
#pragma unroll
        for (int m = 0; m < 6; ++m) pz[m] = pz[m + 1];
        pz[6] = __ldg(a.phis + wrap(k + 3, g.nz) * plane + col);
        const T pc = pz[3];
        T d[3][6];
        {
            T px[7], py[7];
#pragma unroll
            for (int m = 0; m < 7; ++m) {
                px[m] = m == 3 ? pc : __ldg(P + ox[m]);
                py[m] = m == 3 ? pc : __ldg(P + oy[m]);
            }
#pragma unroll
            for (int m = 0; m < 6; ++m) {
                d[0][m] = px[m + 1] - px[m];
                d[1][m] = py[m + 1] - py[m];
                d[2][m] = pz[m + 1] - pz[m];
            }
        }
        T rhs;
        if constexpr (!REINIT) {
            // -u.grad(phi): upwind WENO5 per direction, velocity at the centre
            const T w0 = __ldg(a.W + o + col), vm = wall ? T(0) : __ldg(a.V + o + ovm);
            const T vel[3] = {T(0.5) * (__ldg(a.U + o + ox[2]) + __ldg(a.U + o + col)),
                              T(0.5) * (vm + __ldg(a.V + o + col)), T(0.5) * (wm + w0)};
            wm = w0;
            auto side = [&](int q, int m) { return vel[q] > T(0) ? d[q][m] : d[q][5 - m]; };
            const T sx = vel[0] * g.idx, sy = vel[1] * g.idy, sz = vel[2] * g.idz;
            const T az = weno5(side(2, 0), side(2, 1), side(2, 2), side(2, 3), side(2, 4), sz);
            if constexpr (sizeof(T) == 4) {
                auto xy = [&](int m) { return make_float2(side(0, m), side(1, m)); };
                const float2 sxy = weno5x2(xy(0), xy(1), xy(2), xy(3), xy(4), make_float2(sx, sy));
                rhs = -((sxy.x + sxy.y) + az);
            } else {
                T adv = weno5(side(0, 0), side(0, 1), side(0, 2), side(0, 3), side(0, 4), sx);
                adv += weno5(side(1, 0), side(1, 1), side(1, 2), side(1, 3), side(1, 4), sy);
                adv += az;
                rhs = -adv;
            }
        } else {
            const T f0 = __ldg(a.phi0 + o + col);
            const T sg = f0 / sqrt(fma(a.h, a.h, f0 * f0));
            const T ih[3] = {g.idx, g.idy, g.idz};
            T sum = T(0);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                T dl, dr;              // left- and right-biased derivatives
                if constexpr (sizeof(T) == 4) {
                    auto lr = [&](int m) { return make_float2(d[q][m], d[q][5 - m]); };
                    const float2 r = weno5x2<true>(lr(0), lr(1), lr(2), lr(3), lr(4), splat2(ih[q]));
                    dl = r.x;
                    dr = r.y;
                } else {
                    dl = weno5(d[q][0], d[q][1], d[q][2], d[q][3], d[q][4], ih[q]);
                    dr = weno5(d[q][5], d[q][4], d[q][3], d[q][2], d[q][1], ih[q]);
                }
                // Godunov: (max(dl, 0), min(dr, 0)) for S > 0, (min(dl, 0), max(dr, 0)) else
                const bool up = sg > T(0);
                const T l = up ? dl : -dl, r = up ? -dr : dr;
                // the square rounded on its own
                const T gr = fmax(fmax(l, r), T(0));
                if constexpr (sizeof(T) == 4) sum = __fadd_rn(sum, __fmul_rn(gr, gr));
                else sum = __dadd_rn(sum, __dmul_rn(gr, gr));
            }
            rhs = -sg * (sqrt(sum) - T(1));
        }
        // plain load: the third stage writes phi in place (each cell by its own thread)
        const T pn = a.pt_a != T(0) ? a.phin[o + col] : T(0);
        const T x = fma(a.dt, rhs, pc);
        a.out[o + col] = fma(a.pt_a, pn, a.pt_b * x);
    }
}

// The interface force in two passes, each one read of phi and little else: the unit
// normal is needed (and stored, and read back) only within one cell of the smoothing band
// |phi| <= eps, a few per cent of the cells; 1 - H is summed in integers, because an FP64
// add or a conversion per cell costs more on GB300 than the rest of the pass; and the
// mean's products are formed once instead of per cell.  128 x 256 x 128 FP32: 131 us
// with normals everywhere and FP64 sums, 47 us so.

// smoothed Heaviside of a centre
template <typename T>
__device__ __forceinline__ T heaviside(T ph, T eps) {
    if (ph < -eps) return T(0);
    if (ph > eps) return T(1);
    return T(0.5) * (T(1) + ph / eps + sin(T(3.14159265358979323846) * ph / eps) * T(0.31830988618379067154));
}

// 1 - H as a multiple of 2^-52 for |H| < 2, by the bits of the binary32 H: what lies
// below 2^-52 is dropped, as the rounding of 1 - double(H) does.  False for a larger or
// non-finite H.
__device__ __forceinline__ bool one_minus_fixed(float H, long long& fix) {
    const unsigned b = __float_as_uint(H);
    const int e = (int)((b >> 23) & 0xffu) - 98;          // |H| 2^52 = mantissa 2^e
    if (e > 29) return false;
    const long long m = (long long)((b & 0x7fffffu) | 0x800000u);
    const long long v = e >= 0 ? m << e : (e > -24 ? m >> -e : 0ll);
    fix += (1ll << 52) - ((int)b < 0 ? -v : v);
    return true;
}

constexpr int IF_KZ = 4;                        // planes per block of the first pass

// H, and the unit normal next to the band; per-block sums of (1 - H)
template <typename T>
__global__ void __launch_bounds__(256) k_iface_a(const Geo<T> g, const IfaceArgs<T> a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k0 = blockIdx.z * IF_KZ, k1 = min(k0 + IF_KZ, g.nz);
    long long fix = 0;
    double part = 0.0;
    bool bad = false;
    if (i < g.nx && j < g.ny) {
        const T eps = a.eps;
        const unsigned plane = g.nx * g.ny, row = j * g.nx;
        const unsigned c = row + i, xm = row + wrap(i - 1, g.nx), xp = row + wrap(i + 1, g.nx);
        const unsigned ym = ycen(g, j - 1) * g.nx + i, yp = ycen(g, j + 1) * g.nx + i;
        T below = __ldg(a.phi + wrap(k0 - 1, g.nz) * plane + c), ph = __ldg(a.phi + k0 * plane + c);
        for (int k = k0; k < k1; ++k) {
            const unsigned o = k * plane;
            const T above = __ldg(a.phi + wrap(k + 1, g.nz) * plane + c);
            const T pxm = __ldg(a.phi + o + xm), pxp = __ldg(a.phi + o + xp);
            const T pym = __ldg(a.phi + o + ym), pyp = __ldg(a.phi + o + yp);
            const T H = heaviside(ph, eps);
            a.H[o + c] = H;
            if constexpr (sizeof(T) == 4) {
                bad = !one_minus_fixed(H, fix) || bad;
            } else {
                part += 1.0 - H;
            }
            auto far = [&](T q) { return fabs(q) > eps; };      // false for a NaN
            if (!(far(ph) && far(pxm) && far(pxp) && far(pym) && far(pyp) && far(below) && far(above))) {
                const T gx = (pxp - pxm) * (T(0.5) * g.idx);
                const T gy = (pyp - pym) * (T(0.5) * g.idy);
                const T gz = (above - below) * (T(0.5) * g.idz);
                T mag = sqrt(gx * gx + gy * gy + gz * gz);
                mag = mag > T(1e-12) ? mag : T(1e-12);
                a.n[0][o + c] = gx / mag;
                a.n[1][o + c] = gy / mag;
                a.n[2][o + c] = gz / mag;
            }
            below = ph;
            ph = above;
        }
    }
    // fixed-shape block reduction -> one partial per block
    const int t = threadIdx.y * blockDim.x + threadIdx.x, warp = t >> 5, lane = t & 31;
    if constexpr (sizeof(T) == 4) {
        __shared__ long long red[8];
        __shared__ int rbad[8];
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) fix += __shfl_xor_sync(0xffffffffu, fix, s);
        const bool any = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            red[warp] = fix;
            rbad[warp] = any;
        }
        __syncthreads();
        if (t == 0) {
            long long s = 0;
            int nan = 0;
            for (int w = 0; w < 8; ++w) {
                s += red[w];
                nan |= rbad[w];
            }
            part = nan ? __longlong_as_double(0x7ff8000000000000ll) : (double)s * 0x1p-52;
        }
    } else {
        __shared__ double red[256];
        red[t] = part;
        __syncthreads();
        for (int s = 128; s > 0; s >>= 1) {
            if (t < s) red[t] += red[t + s];
            __syncthreads();
        }
        part = red[0];
    }
    if (t == 0) a.partials[(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = part;
}

// Domain mean of 1 - H, and what the cells need of it in their precision: T mean drho_g
// in out[1] (mean-free buoyancy) and the mean density in out[2] (density contrast)
template <typename T>
__global__ void __launch_bounds__(1024) k_iface_mean(const double* partials, int n, double scale, double drho_g,
                                                     double rho_ratio, double* out) {
    __shared__ double red[1024];
    double s = 0.0;
    for (int q = threadIdx.x; q < n; q += 1024) s += partials[q];
    red[threadIdx.x] = s;
    __syncthreads();
    for (int w = 512; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double m = red[0] * scale;
        out[0] = m;
        *reinterpret_cast<T*>(out + 1) = T(m * drho_g);
        *reinterpret_cast<T*>(out + 2) = T((1.0 - m) + rho_ratio * m);
    }
}

// Soft particles: the solid fraction advected like B, one thread per cell
template <typename T>
__global__ void __launch_bounds__(256) k_phis(const Geo<T> g, const PhisArgs<T> a) {
    pdl_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.nx || j >= g.ny) return;
    const size_t c0 = lin(g, i, j, k);
    // centre velocity: mean of the two faces of the cell
    const T uc = T(0.5) * (__ldg(a.U + c0) + ld_uw(g, a.U, i - 1, j, k));
    const T vc = T(0.5) * (__ldg(a.V + c0) + ld_v(g, a.V, i, j - 1, k));
    const T wc = T(0.5) * (__ldg(a.W + c0) + ld_uw(g, a.W, i, j, k - 1));
    const int sx = uc > T(0) ? 1 : -1, sy = vc > T(0) ? 1 : -1, sz = wc > T(0) ? 1 : -1;
    T p[3][6];
#pragma unroll
    for (int m = 0; m < 6; ++m) {
        p[0][m] = ld_c(g, a.phi, i + (m - 3) * sx, j, k);
        p[1][m] = ld_c(g, a.phi, i, j + (m - 3) * sy, k);
        p[2][m] = ld_c(g, a.phi, i, j, k + (m - 3) * sz);
    }
    const T adv = upwind_term(fabs(uc) * g.idx, p[0][0], p[0][1], p[0][2], p[0][3], p[0][4], p[0][5])
                  + upwind_term(fabs(vc) * g.idy, p[1][0], p[1][1], p[1][2], p[1][3], p[1][4], p[1][5])
                  + upwind_term(fabs(wc) * g.idz, p[2][0], p[2][1], p[2][2], p[2][3], p[2][4], p[2][5]);
    const T R = -adv;
    T inc = a.dt_zeta * R;
    if (a.read_hist) inc += a.dt_xi * a.hist[c0];
    a.phin[c0] = __ldg(a.phi + c0) + inc;
    if (a.write_hist) a.hist[c0] = R;
}

// Mass correction: per-block FP64 sums of 1 - H(phi + d) and delta(phi + d)
template <typename T>
__global__ void __launch_bounds__(256) k_mass_partials(const Geo<T> g, const MassArgs<T> a, int np) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    double v = 0.0, ar = 0.0;
    if (i < g.nx && j < g.ny) {
        const T ph = __ldg(a.phi + lin(g, i, j, k)) + T(*a.d);
        const T eps = a.eps;
        T H, D;
        if (ph < -eps) {
            H = T(0);
            D = T(0);
        } else if (ph > eps) {
            H = T(1);
            D = T(0);
        } else {
            const T x = T(3.14159265358979323846) * ph / eps;
            H = T(0.5) * (T(1) + ph / eps + sin(x) * T(0.31830988618379067154));
            D = T(0.5) / eps * (T(1) + cos(x));
        }
        v = 1.0 - double(H);
        ar = double(D);
    }
    __shared__ double rv[256], ra[256];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    rv[t] = v;
    ra[t] = ar;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (t < w) {
            rv[t] += rv[t + w];
            ra[t] += ra[t + w];
        }
        __syncthreads();
    }
    if (t == 0) {
        const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        a.partials[b] = rv[0];
        a.partials[np + b] = ra[0];
    }
}

// Mass correction: sum the block partials (fixed order) and either record the
// volume (mode 0) or take one Newton step d += (V - v0)/A (mode 1)
__global__ void __launch_bounds__(256) k_mass_newton(const double* partials, int np, double dv, double* v0,
                                                     double* d, int mode) {
    __shared__ double rv[256], ra[256];
    double v = 0.0, ar = 0.0;
    for (int q = threadIdx.x; q < np; q += 256) {
        v += partials[q];
        ar += partials[np + q];
    }
    rv[threadIdx.x] = v;
    ra[threadIdx.x] = ar;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) {
            rv[threadIdx.x] += rv[threadIdx.x + w];
            ra[threadIdx.x] += ra[threadIdx.x + w];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double V = rv[0] * dv, A = ra[0] * dv;
        if (mode == 0) *v0 = V;
        else if (A > 0.0) *d += (V - *v0) / A;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_mass_shift(T* phi, size_t n, const double* d) {
    const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c < n) phi[c] += T(*d);
}

// CSF force sigma kappa delta(phi) n plus buoyancy (1 - H - mean(1 - H)) drho_g e_y: two
// cells of a row per thread (nx is even), the force itself in the band only
template <typename T>
__global__ void __launch_bounds__(256) k_iface_b(const Geo<T> g, const IfaceArgs<T> a) {
    const int i2 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i2 >= g.nx || j >= g.ny) return;
    const size_t c0 = lin(g, i2, j, k);
    const T eps = a.eps;
    const T mean = *reinterpret_cast<const T*>(a.mean_1mH + 1);
    T f[3][2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int i = i2 + q;
        const T ph = __ldg(a.phi + c0 + q);
        f[0][q] = T(0);
        f[1][q] = (T(1) - __ldg(a.H + c0 + q)) * a.drho_g - mean;
        f[2][q] = T(0);
        if (ph != ph) {
            f[0][q] = f[2][q] = ph;             // a NaN, as f[1] is by H
        } else if (fabs(ph) <= eps) {
            const T kap = -((ld_c(g, a.n[0], i + 1, j, k) - ld_c(g, a.n[0], i - 1, j, k)) * (T(0.5) * g.idx)
                            + (ld_c(g, a.n[1], i, j + 1, k) - ld_c(g, a.n[1], i, j - 1, k)) * (T(0.5) * g.idy)
                            + (ld_c(g, a.n[2], i, j, k + 1) - ld_c(g, a.n[2], i, j, k - 1)) * (T(0.5) * g.idz));
            const T dl = T(0.5) / eps * (T(1) + cos(T(3.14159265358979323846) * ph / eps));
            const T s = a.sigma * kap * dl;
            f[0][q] = s * __ldg(a.n[0] + c0 + q);
            f[1][q] += s * __ldg(a.n[1] + c0 + q);
            f[2][q] = s * __ldg(a.n[2] + c0 + q);
        }
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        if constexpr (sizeof(T) == 4) *reinterpret_cast<float2*>(a.f[q] + c0) = make_float2(f[q][0], f[q][1]);
        else *reinterpret_cast<double2*>(a.f[q] + c0) = make_double2(f[q][0], f[q][1]);
    }
}

// tau component c at a centre from B^n (b: the six components there) with the
// mixture polymer viscosity mu_p(H) (Table 1 inverted)
template <typename T, int MODEL>
__device__ __forceinline__ T tau_value(const MomAB2Args<T>& a, int c, const T* b, T H) {
    const T gm = (a.mu_p1 * H + a.mu_p2 * (T(1) - H)) * a.inv_lam;
    const bool diag = (c == 0 || c == 3 || c == 5);
    if (MODEL == EVP_FENE_P) {
        const T tr = b[0] + b[3] + b[5];
        const T F = a.L2 / (a.L2 - tr);
        return gm * (F * b[c] - (diag ? a.a_fene : T(0)));
    }
    if (MODEL == EVP_NEO_HOOKEAN) return gm * b[c];
    return gm * (b[c] - (diag ? T(1) : T(0)));
}

// One cell (i, j, k) of the AB2 momentum step.  S gives the staged values around
// the cell at offsets (di, dj, dk) in -1 .. 1: S.u, S.v, S.w (faces), S.H, S.tau(c)
// and S.f(q) (centres); the wraps and wall ghost rules were applied when staging.
template <typename T, int MODEL, typename Src>
__device__ __forceinline__ void momentum_ab2_cell(const Geo<T>& g, const MomAB2Args<T>& a, int i, int j, int k,
                                                  const Src& S) {
    const size_t c0 = lin(g, i, j, k);
    auto u = [&](int di, int dj, int dk) { return S.u(di, dj, dk); };
    auto v = [&](int di, int dj, int dk) { return S.v(di, dj, dk); };
    auto w = [&](int di, int dj, int dk) { return S.w(di, dj, dk); };
    auto mu = [&](int di, int dj, int dk) {
        const T H = S.H(di, dj, dk);
        return a.mu_s1 * H + a.mu_s2 * (T(1) - H);
    };
    // viscosity averaged over the 4 centres (0 or d1) x (0 or d2), shifted by (si, sj, sk)
    auto mue = [&](int si, int sj, int sk, int di, int dj, int dk) {
        int a1i = 0, a1j = 0, a1k = 0, a2i = 0, a2j = 0, a2k = 0;
        if (di) {
            a1i = di;
            if (dj) a2j = dj; else a2k = dk;
        } else {
            a1j = dj;
            a2k = dk;
        }
        return T(0.25) * (mu(si, sj, sk) + mu(si + a2i, sj + a2j, sk + a2k) + mu(si + a1i, sj + a1j, sk + a1k)
                          + mu(si + a1i + a2i, sj + a1j + a2j, sk + a1k + a2k));
    };
    auto tau = [&](int c, int di, int dj, int dk) { return S.tau(c, di, dj, dk); };
    // average of tau_c over (0 or d1) x (0 or d2) around the cell; offsets as in the RK3 kernel
    auto tau_e4 = [&](int c, int di, int dj, int dk) {
        int a1i = 0, a1j = 0, a1k = 0, a2i = 0, a2j = 0, a2k = 0;
        if (di) {
            a1i = di;
            if (dj) a2j = dj; else a2k = dk;
        } else {
            a1j = dj;
            a2k = dk;
        }
        return T(0.25) * (tau(c, 0, 0, 0) + tau(c, a2i, a2j, a2k) + tau(c, a1i, a1j, a1k)
                          + tau(c, a1i + a2i, a1j + a2j, a1k + a2k));
    };
    const T h = T(0.5);
    const T u0 = u(0, 0, 0), v0 = v(0, 0, 0), w0 = w(0, 0, 0);
    const T ix = g.idx, iy = g.idy, iz = g.idz;

    // ---- div(uu) (same discretisation as the RK3 predictor)
    const T Ax = (sqr(h * (u0 + u(1, 0, 0))) - sqr(h * (u(-1, 0, 0) + u0))) * ix
                 + (h * (u0 + u(0, 1, 0)) * h * (v0 + v(1, 0, 0)) - h * (u(0, -1, 0) + u0) * h * (v(0, -1, 0) + v(1, -1, 0))) * iy
                 + (h * (u0 + u(0, 0, 1)) * h * (w0 + w(1, 0, 0)) - h * (u(0, 0, -1) + u0) * h * (w(0, 0, -1) + w(1, 0, -1))) * iz;
    const T Ay = (h * (u0 + u(0, 1, 0)) * h * (v0 + v(1, 0, 0)) - h * (u(-1, 0, 0) + u(-1, 1, 0)) * h * (v(-1, 0, 0) + v0)) * ix
                 + (sqr(h * (v0 + v(0, 1, 0))) - sqr(h * (v(0, -1, 0) + v0))) * iy
                 + (h * (v0 + v(0, 0, 1)) * h * (w0 + w(0, 1, 0)) - h * (v(0, 0, -1) + v0) * h * (w(0, 0, -1) + w(0, 1, -1))) * iz;
    const T Az = (h * (u0 + u(0, 0, 1)) * h * (w0 + w(1, 0, 0)) - h * (u(-1, 0, 0) + u(-1, 0, 1)) * h * (w(-1, 0, 0) + w0)) * ix
                 + (h * (v0 + v(0, 0, 1)) * h * (w0 + w(0, 1, 0)) - h * (v(0, -1, 0) + v(0, -1, 1)) * h * (w(0, -1, 0) + w0)) * iy
                 + (sqr(h * (w0 + w(0, 0, 1))) - sqr(h * (w(0, 0, -1) + w0))) * iz;

    // ---- div[mu (grad u + grad u^T)], normal stresses at centres, shear at edges
    auto sxx = [&](int di) { return T(2) * mu(di, 0, 0) * (u(di, 0, 0) - u(di - 1, 0, 0)) * ix; };
    auto syy = [&](int dj) { return T(2) * mu(0, dj, 0) * (v(0, dj, 0) - v(0, dj - 1, 0)) * iy; };
    auto szz = [&](int dk) { return T(2) * mu(0, 0, dk) * (w(0, 0, dk) - w(0, 0, dk - 1)) * iz; };
    // shear stress at the xy edge (i+si+1/2, j+sj+1/2), etc.
    auto sxy = [&](int si, int sj) {
        return mue(si, sj, 0, 1, 1, 0) * ((u(si, sj + 1, 0) - u(si, sj, 0)) * iy + (v(si + 1, sj, 0) - v(si, sj, 0)) * ix);
    };
    auto sxz = [&](int si, int sk) {
        return mue(si, 0, sk, 1, 0, 1) * ((u(si, 0, sk + 1) - u(si, 0, sk)) * iz + (w(si + 1, 0, sk) - w(si, 0, sk)) * ix);
    };
    auto syz = [&](int sj, int sk) {
        return mue(0, sj, sk, 0, 1, 1) * ((v(0, sj, sk + 1) - v(0, sj, sk)) * iz + (w(0, sj + 1, sk) - w(0, sj, sk)) * iy);
    };
    const T Vx = (sxx(1) - sxx(0)) * ix + (sxy(0, 0) - sxy(0, -1)) * iy + (sxz(0, 0) - sxz(0, -1)) * iz;
    const T Vy = (sxy(0, 0) - sxy(-1, 0)) * ix + (syy(1) - syy(0)) * iy + (syz(0, 0) - syz(0, -1)) * iz;
    const T Vz = (sxz(0, 0) - sxz(-1, 0)) * ix + (syz(0, 0) - syz(-1, 0)) * iy + (szz(1) - szz(0)) * iz;

    // ---- div tau^n with mu_p(H)
    T dtx = T(0), dty = T(0), dtz = T(0);
    if (MODEL != EVP_NEWTONIAN) {
        dtx = (tau(0, 1, 0, 0) - tau(0, 0, 0, 0)) * ix + (tau_e4(1, 1, 1, 0) - tau_e4(1, 1, -1, 0)) * iy
              + (tau_e4(2, 1, 0, 1) - tau_e4(2, 1, 0, -1)) * iz;
        dty = (tau_e4(1, 1, 1, 0) - tau_e4(1, -1, 1, 0)) * ix + (tau(3, 0, 1, 0) - tau(3, 0, 0, 0)) * iy
              + (tau_e4(4, 0, 1, 1) - tau_e4(4, 0, 1, -1)) * iz;
        dtz = (tau_e4(2, 1, 0, 1) - tau_e4(2, -1, 0, 1)) * ix + (tau_e4(4, 0, 1, 1) - tau_e4(4, 0, -1, 1)) * iy
              + (tau(5, 0, 0, 1) - tau(5, 0, 0, 0)) * iz;
    }

    // ---- interface force: mean of the two centres next to each face
    const T Fx = h * (S.f(0, 0, 0, 0) + S.f(0, 1, 0, 0));
    const T Fy = h * (S.f(1, 0, 0, 0) + S.f(1, 0, 1, 0));
    const T Fz = h * (S.f(2, 0, 0, 0) + S.f(2, 0, 0, 1));

    T Nx, Ny, Nz;
    if (a.rho_ratio > T(0)) {
        // density contrast: 1/rho on the stress terms, (1 - rho_bar/rho) g per unit mass
        auto rho = [&](int di, int dj, int dk) {
            const T Hc = S.H(di, dj, dk);
            return Hc + a.rho_ratio * (T(1) - Hc);
        };
        const T r0 = rho(0, 0, 0);
        const T rfx = h * (r0 + rho(1, 0, 0)), rfy = h * (r0 + rho(0, 1, 0)), rfz = h * (r0 + rho(0, 0, 1));
        const T rbar = *reinterpret_cast<const T*>(a.mean_1mH + 2);
        Nx = -Ax + (Vx + dtx + Fx) / rfx;
        Ny = -Ay + (Vy + dty + Fy) / rfy + (T(1) - rbar / rfy) * (-a.gravity);
        Nz = -Az + (Vz + dtz + Fz) / rfz;
    } else {
        Nx = -Ax + Vx + dtx + Fx;
        Ny = -Ay + Vy + dty + Fy;
        Nz = -Az + Vz + dtz + Fz;
    }
    T ux = a.w1dt * Nx, uy = a.w1dt * Ny, uz = a.w1dt * Nz;
    if (a.read_hist) {
        ux += a.w0dt * a.NH[0][c0];
        uy += a.w0dt * a.NH[1][c0];
        uz += a.w0dt * a.NH[2][c0];
    }
    a.Us[c0] = u0 + ux;
    a.Vs[c0] = (g.walls && j == g.ny - 1) ? T(0) : v0 + uy;
    a.Ws[c0] = w0 + uz;
    a.NH[0][c0] = Nx;
    a.NH[1][c0] = Ny;
    a.NH[2][c0] = Nz;
}

// z-marching tiles of the AB2 momentum step: a 32 x 4 tile walks a chunk of z planes.
// Planes k-1, k, k+1 of u, v, w, H and tau (built once per staged cell from B^n and H,
// instead of once per stencil use) and planes k, k+1 of the interface force sit in
// shared memory with a one-cell halo in x and y, staged with the periodic wraps and the
// wall ghost rules; the raw values of plane k+2 are loaded into registers before plane k
// is computed.  A staged cell's offset and its wall ghost (the nearest row, u and w
// negated, v zero) are found once per thread.  Bound by instruction issue and
// shared-memory reads, about 45 a cell.  128 x 256 x 128 FP32: 154 us with wraps and ghost
// rules at each of the 13 reads of a staged cell, 144 so (32 x 8 tiles 150, 32 x 16 160).
constexpr int AB_TX = 32, AB_TY = 4, AB_NT = AB_TX * AB_TY;
constexpr int AB_W = AB_TX + 2, AB_PL = AB_W * (AB_TY + 2);
constexpr int AB_NE = (AB_PL + AB_NT - 1) / AB_NT;          // staged cells per thread

template <typename T>
struct Ab2Smem {
    static constexpr int RES = sizeof(T) == 4 ? 4 : 3;      // CTAs per SM that the registers leave
    T U[3][AB_PL], V[3][AB_PL], W[3][AB_PL], H[3][AB_PL];    // ring slot = plane mod 3
    T TAU[6][3][AB_PL];
    T F[3][2][AB_PL];                                       // slot = plane mod 2
};

template <typename T>
struct Ab2Src {
    const Ab2Smem<T>* sm;
    int o;          // the cell in a plane tile
    int sl[3];      // slots of planes k-1, k, k+1
    int fs[2];      // force slots of planes k, k+1
    __device__ __forceinline__ int at(int di, int dj) const { return o + dj * AB_W + di; }
    __device__ __forceinline__ T u(int di, int dj, int dk) const { return sm->U[sl[1 + dk]][at(di, dj)]; }
    __device__ __forceinline__ T v(int di, int dj, int dk) const { return sm->V[sl[1 + dk]][at(di, dj)]; }
    __device__ __forceinline__ T w(int di, int dj, int dk) const { return sm->W[sl[1 + dk]][at(di, dj)]; }
    __device__ __forceinline__ T H(int di, int dj, int dk) const { return sm->H[sl[1 + dk]][at(di, dj)]; }
    __device__ __forceinline__ T tau(int c, int di, int dj, int dk) const {
        return sm->TAU[c][sl[1 + dk]][at(di, dj)];
    }
    __device__ __forceinline__ T f(int q, int di, int dj, int dk) const { return sm->F[q][fs[dk]][at(di, dj)]; }
};

template <typename T, int MODEL>
__global__ void __launch_bounds__(AB_NT, Ab2Smem<T>::RES)
k_momentum_ab2(const Geo<T> g, const MomAB2Args<T> a, int kz_chunk) {
    extern __shared__ __align__(16) unsigned char smraw[];
    Ab2Smem<T>& sm = *reinterpret_cast<Ab2Smem<T>*>(smraw);
    const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * AB_TX + tx;
    const int i0 = blockIdx.x * AB_TX, j0 = blockIdx.y * AB_TY;
    const int k0 = blockIdx.z * kz_chunk, k1 = min(k0 + kz_chunk, g.nz);
    const int i = i0 + tx, j = j0 + ty;
    const bool active = i < g.nx && j < g.ny;
    constexpr bool STRESS = MODEL != EVP_NEWTONIAN;
    const size_t plane = (size_t)g.nx * g.ny;
    // raw values of one staged plane for this thread's cells, their offsets in a plane
    T ru[AB_NE], rv[AB_NE], rw[AB_NE], rH[AB_NE], rB[6][AB_NE], rf[3][AB_NE];
    int off[AB_NE];
    bool ghost[AB_NE];
#pragma unroll
    for (int r = 0; r < AB_NE; ++r) {
        const int e = min(tid + r * AB_NT, AB_PL - 1), ly = e / AB_W, lx = e - ly * AB_W;
        // the halo of a ragged tile may reach past the ghosts: any cell does there
        const int gi = min(i0 - 1 + lx, g.nx), gj = min(j0 - 1 + ly, g.ny);
        off[r] = ycen(g, gj) * g.nx + wrap(gi, g.nx);
        ghost[r] = g.walls && (gj < 0 || gj >= g.ny);
    }
    auto load = [&](int q) {
        const size_t o = (size_t)wrap(q, g.nz) * plane;
#pragma unroll
        for (int r = 0; r < AB_NE; ++r) {
            if (tid + r * AB_NT >= AB_PL) continue;
            const int c0 = off[r];
            ru[r] = __ldg(a.U + o + c0);
            rv[r] = __ldg(a.V + o + c0);
            rw[r] = __ldg(a.W + o + c0);
            rH[r] = __ldg(a.H + o + c0);
#pragma unroll
            for (int c = 0; c < 6; ++c) rB[c][r] = STRESS ? __ldg(a.B[c] + o + c0) : T(0);
#pragma unroll
            for (int c = 0; c < 3; ++c) rf[c][r] = __ldg(a.f[c] + o + c0);
        }
    };
    auto store = [&](int q) {
        const int s3 = (q + 3) % 3, s2 = q & 1;
#pragma unroll
        for (int r = 0; r < AB_NE; ++r) {
            const int e = tid + r * AB_NT;
            if (e >= AB_PL) continue;
            sm.U[s3][e] = ghost[r] ? -ru[r] : ru[r];
            sm.V[s3][e] = ghost[r] ? T(0) : rv[r];
            sm.W[s3][e] = ghost[r] ? -rw[r] : rw[r];
            sm.H[s3][e] = rH[r];
            if (STRESS) {
                T b[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) b[c] = rB[c][r];
#pragma unroll
                for (int c = 0; c < 6; ++c) sm.TAU[c][s3][e] = tau_value<T, MODEL>(a, c, b, rH[r]);
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) sm.F[c][s2][e] = rf[c][r];
        }
    };
    for (int q = k0 - 1; q <= k0 + 1; ++q) {
        load(q);
        store(q);
    }
    __syncthreads();
    Ab2Src<T> src;
    src.sm = &sm;
    src.o = (ty + 1) * AB_W + tx + 1;
    for (int k = k0; k < k1; ++k) {
        const bool more = k + 2 <= k1;
        if (more) load(k + 2);
        src.sl[0] = (k + 2) % 3;
        src.sl[1] = k % 3;
        src.sl[2] = (k + 1) % 3;
        src.fs[0] = k & 1;
        src.fs[1] = (k + 1) & 1;
        if (active) momentum_ab2_cell<T, MODEL>(g, a, i, j, k, src);
        __syncthreads();
        if (more) store(k + 2);
        __syncthreads();
    }
}

// density at a centre from the Heaviside: rho_1 = 1 (H = 1), rho_2 = rho_ratio
template <typename T>
__device__ __forceinline__ T rho_c(const Geo<T>& g, const SplitArgs<T>& a, int i, int j, int k) {
    const T H = ld_c(g, a.H, i, j, k);
    return H + a.rho_ratio * (T(1) - H);
}

// p_hat = 2 p^n - p^{n-1} at a centre
template <typename T>
__device__ __forceinline__ T phat(const Geo<T>& g, const SplitArgs<T>& a, int i, int j, int k) {
    return T(2) * ld_c(g, a.P, i, j, k) - ld_c(g, a.Pold, i, j, k);
}

// r = div[(1 - rho_0/rho_f) grad p_hat] + (rho_0/dt) div u*   (Eq. poisson-LS)
template <typename T>
__global__ void __launch_bounds__(256) k_split_rhs(const Geo<T> g, const SplitArgs<T> a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    if (i >= g.nx || j >= g.ny) return;
    const size_t c0 = lin(g, i, j, k);
    const T r0 = rho_c(g, a, i, j, k), p0 = phat(g, a, i, j, k);
    // flux (1 - rho_0/rho_f) d p_hat / dn through the +1/2 face of (i, j, k) offset by (di, dj, dk)
    auto fx = [&](int di) {
        const T ra = rho_c(g, a, i + di, j, k), rb = rho_c(g, a, i + di + 1, j, k);
        return (T(1) - a.rho0 / (T(0.5) * (ra + rb))) * (phat(g, a, i + di + 1, j, k) - phat(g, a, i + di, j, k)) * g.idx;
    };
    auto fy = [&](int dj) {
        const int jf = j + dj;
        if (g.walls && (jf < 0 || jf >= g.ny - 1)) return T(0);   // no flux through the walls
        const T ra = rho_c(g, a, i, jf, k), rb = rho_c(g, a, i, jf + 1, k);
        return (T(1) - a.rho0 / (T(0.5) * (ra + rb))) * (phat(g, a, i, jf + 1, k) - phat(g, a, i, jf, k)) * g.idy;
    };
    auto fz = [&](int dk) {
        const T ra = rho_c(g, a, i, j, k + dk), rb = rho_c(g, a, i, j, k + dk + 1);
        return (T(1) - a.rho0 / (T(0.5) * (ra + rb))) * (phat(g, a, i, j, k + dk + 1) - phat(g, a, i, j, k + dk)) * g.idz;
    };
    (void)r0;
    (void)p0;
    const T divf = (fx(0) - fx(-1)) * g.idx + (fy(0) - fy(-1)) * g.idy + (fz(0) - fz(-1)) * g.idz;
    const T du = __ldg(a.Us + c0) - ld_uw(g, a.Us, i - 1, j, k);
    const T dv = __ldg(a.Vs + c0) - ld_v(g, a.Vs, i, j - 1, k);
    const T dw = __ldg(a.Ws + c0) - ld_uw(g, a.Ws, i, j, k - 1);
    a.R[c0] = divf + a.rho0 / a.dt * (du * g.idx + dv * g.idy + dw * g.idz);
}

// u^{n+1} = u* - dt [grad p^{n+1}/rho_0 + (1/rho_f - 1/rho_0) grad p_hat]   (Eq. projection-LS)
template <typename T>
__global__ void __launch_bounds__(256) k_split_correct(const Geo<T> g, const SplitArgs<T> a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    const int j = blockIdx.y * blockDim.y + threadIdx.y;
    const int k = blockIdx.z;
    unsigned bits = 0;
    if (i < g.nx && j < g.ny) {
        const size_t c0 = lin(g, i, j, k);
        const T ir0 = T(1) / a.rho0;
        // corrected face value of component d at the +1/2 face of (ii, jj, kk)
        auto face = [&](int d, int ii, int jj, int kk) {
            int oi = d == 0, oj = d == 1, ok = d == 2;
            if (d == 1 && g.walls && (jj < 0 || jj >= g.ny - 1)) return T(0);
            const T* S = d == 0 ? a.Us : (d == 1 ? a.Vs : a.Ws);
            const T us = d == 1 ? ld_v(g, S, ii, jj, kk) : ld_uw(g, S, ii, jj, kk);
            const T h = d == 0 ? g.idx : (d == 1 ? g.idy : g.idz);
            const T ra = rho_c(g, a, ii, jj, kk), rb = rho_c(g, a, ii + oi, jj + oj, kk + ok);
            const T rf = T(0.5) * (ra + rb);
            const T gp = (ld_c(g, a.R, ii + oi, jj + oj, kk + ok) - ld_c(g, a.R, ii, jj, kk)) * h;
            const T gh = (phat(g, a, ii + oi, jj + oj, kk + ok) - phat(g, a, ii, jj, kk)) * h;
            return us - a.dt * (gp * ir0 + (T(1) / rf - ir0) * gh);
        };
        const T Un = face(0, i, j, k), Vn = face(1, i, j, k), Wn = face(2, i, j, k);
        a.U[c0] = Un;
        a.V[c0] = Vn;
        a.W[c0] = Wn;
        if (!isfinite(Un + Vn + Wn)) bits |= EVP_BIT_NONFINITE;
    }
    bits = __reduce_or_sync(0xffffffffu, bits);
    if ((threadIdx.x & 31) == 0 && bits) atomicOr(a.status, bits);
}

}  // namespace

template <typename T>
cudaError_t launch_split_rhs(const Geo<T>& g, const SplitArgs<T>& a, cudaStream_t st, const TimingHook& th) {
    dim3 block(32, 8, 1), grid((g.nx + 31) / 32, (g.ny + 7) / 8, g.nz);
    th.b(K_DIV_FFTX);
    k_split_rhs<T><<<grid, block, 0, st>>>(g, a);
    th.e(K_DIV_FFTX);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_split_correct(const Geo<T>& g, const SplitArgs<T>& a, cudaStream_t st, const TimingHook& th) {
    dim3 block(32, 8, 1), grid((g.nx + 31) / 32, (g.ny + 7) / 8, g.nz);
    th.b(K_CORRECT);
    k_split_correct<T><<<grid, block, 0, st>>>(g, a);
    th.e(K_CORRECT);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_ls_stage(const Geo<T>& g, const LsArgs<T>& a, bool reinit, cudaStream_t st,
                            const TimingHook& th) {
    // planes per CTA: a chunk costs six reads more to start with, a small grid needs CTAs:
    // up to eight planes, one below LS_CTAS CTAs per SM (128 x 256 x 128, times for
    // LS_CTAS = 4, 8, 16, 32: 53.9, 54.0, 53.0, 56.0 us)
    const dim3 block(32, 8, 1), tiles((g.nx + 31) / 32, (g.ny + 7) / 8, 1);
    const long long items = (long long)tiles.x * tiles.y * g.nz;
    const int kz = (int)std::min<long long>(8, std::max<long long>(1, items / (LS_CTAS * 152)));
    const dim3 grid(tiles.x, tiles.y, (g.nz + kz - 1) / kz);
    th.b(K_LEVELSET);
    if (reinit)
        k_ls_stage<T, true><<<grid, block, 0, st>>>(g, a, kz);
    else
        k_ls_stage<T, false><<<grid, block, 0, st>>>(g, a, kz);
    th.e(K_LEVELSET);
    return cudaGetLastError();
}

template <typename T>
size_t iface_partials(const Geo<T>& g) {
    return (size_t)((g.nx + 31) / 32) * ((g.ny + 7) / 8) * g.nz;
}

template <typename T>
cudaError_t launch_interface(const Geo<T>& g, const IfaceArgs<T>& a, cudaStream_t st, const TimingHook& th) {
    const dim3 block(32, 8, 1), ga((g.nx + 31) / 32, (g.ny + 7) / 8, (g.nz + IF_KZ - 1) / IF_KZ);
    const dim3 gb((g.nx / 2 + 31) / 32, (g.ny + 7) / 8, g.nz);
    th.b(K_INTERFACE);
    k_iface_a<T><<<ga, block, 0, st>>>(g, a);
    k_iface_mean<T><<<1, 1024, 0, st>>>(a.partials, (int)(ga.x * ga.y * ga.z), 1.0 / (double(g.nx) * g.ny * g.nz),
                                        (double)a.drho_g, a.rho_ratio, a.mean_1mH);
    k_iface_b<T><<<gb, block, 0, st>>>(g, a);
    th.e(K_INTERFACE);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_phis(const Geo<T>& g, const PhisArgs<T>& a, cudaStream_t st, const TimingHook& th) {
    dim3 block(32, 8, 1), grid((g.nx + 31) / 32, (g.ny + 7) / 8, g.nz);
    th.b(K_LEVELSET);
    k_phis<T><<<grid, block, 0, st>>>(g, a);
    th.e(K_LEVELSET);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_mass_correct(const Geo<T>& g, const MassArgs<T>& a, int mode, int iters, cudaStream_t st,
                                const TimingHook& th) {
    dim3 block(32, 8, 1), grid((g.nx + 31) / 32, (g.ny + 7) / 8, g.nz);
    const int np = (int)iface_partials(g);
    const size_t n = (size_t)g.nx * g.ny * g.nz;
    th.b(K_LEVELSET);
    cudaError_t e = cudaMemsetAsync(a.d, 0, sizeof(double), st);
    if (e != cudaSuccess) return e;
    if (mode == 0) {
        k_mass_partials<T><<<grid, block, 0, st>>>(g, a, np);
        k_mass_newton<<<1, 256, 0, st>>>(a.partials, np, a.dv, a.v0, a.d, 0);
    } else {
        for (int it = 0; it < iters; ++it) {
            k_mass_partials<T><<<grid, block, 0, st>>>(g, a, np);
            k_mass_newton<<<1, 256, 0, st>>>(a.partials, np, a.dv, a.v0, a.d, 1);
        }
        k_mass_shift<T><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(a.phi, n, a.d);
    }
    th.e(K_LEVELSET);
    return cudaGetLastError();
}

template <typename T>
cudaError_t launch_momentum_ab2(const Geo<T>& g, int model, const MomAB2Args<T>& a, cudaStream_t st,
                                const TimingHook& th) {
    // planes per chunk: the least (waves of CTAs) x (planes + 2), two planes being what a
    // chunk's start costs
    const int gx = (g.nx + AB_TX - 1) / AB_TX, gy = (g.ny + AB_TY - 1) / AB_TY;
    int kz = 1;
    long long best = LLONG_MAX;
    for (int c = 1; c <= g.nz; ++c) {
        const long long ctas = (long long)gx * gy * ((g.nz + c - 1) / c), slots = 152 * Ab2Smem<T>::RES;
        const long long cost = (ctas + slots - 1) / slots * (c + 2);
        if (cost < best) {
            best = cost;
            kz = c;
        }
    }
    const dim3 block(AB_TX, AB_TY, 1), grid(gx, gy, (g.nz + kz - 1) / kz);
    const size_t smem = sizeof(Ab2Smem<T>);
    auto go = [&](auto kern) {
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kern<<<grid, block, smem, st>>>(g, a, kz);
    };
    th.b(K_MOMENTUM);
    switch (model) {
        case EVP_NEWTONIAN: go(k_momentum_ab2<T, EVP_NEWTONIAN>); break;
        case EVP_OLDROYD_B: go(k_momentum_ab2<T, EVP_OLDROYD_B>); break;
        case EVP_FENE_P: go(k_momentum_ab2<T, EVP_FENE_P>); break;
        case EVP_SARAMITO: go(k_momentum_ab2<T, EVP_SARAMITO>); break;
        case EVP_NEO_HOOKEAN: go(k_momentum_ab2<T, EVP_NEO_HOOKEAN>); break;
        default: return cudaErrorInvalidValue;
    }
    th.e(K_MOMENTUM);
    return cudaGetLastError();
}

#define EVP_INST(T)                                                                                           \
    template cudaError_t launch_ls_stage<T>(const Geo<T>&, const LsArgs<T>&, bool, cudaStream_t,              \
                                            const TimingHook&);                                               \
    template size_t iface_partials<T>(const Geo<T>&);                                                         \
    template cudaError_t launch_interface<T>(const Geo<T>&, const IfaceArgs<T>&, cudaStream_t,                \
                                             const TimingHook&);                                              \
    template cudaError_t launch_mass_correct<T>(const Geo<T>&, const MassArgs<T>&, int, int, cudaStream_t,    \
                                                const TimingHook&);                                           \
    template cudaError_t launch_phis<T>(const Geo<T>&, const PhisArgs<T>&, cudaStream_t, const TimingHook&);  \
    template cudaError_t launch_momentum_ab2<T>(const Geo<T>&, int, const MomAB2Args<T>&, cudaStream_t,       \
                                                const TimingHook&);                                           \
    template cudaError_t launch_split_rhs<T>(const Geo<T>&, const SplitArgs<T>&, cudaStream_t, const TimingHook&); \
    template cudaError_t launch_split_correct<T>(const Geo<T>&, const SplitArgs<T>&, cudaStream_t,            \
                                                 const TimingHook&);
EVP_INST(float)
EVP_INST(double)
#undef EVP_INST

}  // namespace evp
