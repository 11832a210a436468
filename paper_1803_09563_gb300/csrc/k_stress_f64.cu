// Stress kernel (S1 + S2) in double precision: the equations of k_stress.cuh
//
// RT = (a I - F B)/lambda - (u.grad B - B.grad u - grad u^T.B)     (Eq. rt / RK-rt)
//      [+ kappa_ad lap B where det B < 0 or, FENE-P, tr B >= 0.95 L^2  (Sec. 3.1)]
// B^k = B^{k-1} + dt (zeta^k RT^{k-1} + xi^k RT^{k-2})            (Eq. rk3tau)
//
// arranged for GB300's FP64 pipe, which takes 64 cycles per warp instruction and
// scheduler (2 lanes per clock and SM): the kernel's time is its count of FP64-pipe
// instructions, while loads, shared memory and integer work have that many cycles to
// hide in.  So
//   * the second differences of B and the third-difference part of the smoothness
//     indicators, which up to four cells of a line use, are formed once per grid
//     point (x and y: in shared memory for the tile's plane; z: in a register window
//     that moves with the plane) instead of once per reconstruction;
//   * a WENO5 reconstruction is the upwind first difference plus weighted second
//     differences, with one reciprocal refined from the hardware's approximation:
//     29 FP64 instructions instead of 52;
//   * tests and conversions that would run on the FP64 pipe are integer operations,
//     and the determinant's sign is settled in single precision unless it is close;
//   * the tile's shape is chosen for the grid (stress_shape): an inactive lane costs
//     as much as an active one, and 32-wide tiles leave a quarter of the lanes idle
//     on a 72-point row.
#include "evp_internal.cuh"
#include "refined.cuh"

namespace evp {

namespace {

constexpr int NT = 128;    // threads of a CTA, one cell each

__device__ __forceinline__ constexpr int symi(int a, int b) {
    return a <= b ? (a == 0 ? b : (a == 1 ? 2 + b : 5)) : (b == 0 ? a : (b == 1 ? 2 + a : 5));
}
__device__ __forceinline__ constexpr int row_of(int c) { return c < 3 ? 0 : (c < 5 ? 1 : 2); }
__device__ __forceinline__ constexpr int col_of(int c) { return c == 0 ? 0 : ((c == 1 || c == 3) ? 1 : 2); }
__device__ __forceinline__ constexpr bool is_diag(int c) { return c == 0 || c == 3 || c == 5; }

__device__ __forceinline__ int pmod(int a, int n) {
    const int r = a % n;
    return r < 0 ? r + n : r;
}

__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
// x > 0 by integer compare (true for a positive NaN, whose products are NaN anyway)
__device__ __forceinline__ bool positive_bits(double x) { return __double_as_longlong(x) > 0; }
// x, -x or 0 for f = 1, -1, 0 without an FP64 instruction
__device__ __forceinline__ double scaled(double x, int f) {
    const int hi = __double2hiint(x) ^ (f < 0 ? (int)0x80000000 : 0);
    return f ? __hiloint2double(hi, __double2loint(x)) : 0.0;
}

// Third-difference part of a smoothness indicator: (13/3) a^2 + 4 eps, so that
// 4 (eps + S) = b^2 + this with S = 13/12 a^2 + 1/4 b^2 (Jiang-Shu)
__device__ __forceinline__ double smooth_a(double a) { return fma(a * (13.0 / 3.0), a, 4.0e-6); }

// Upwind WENO5 undivided derivative (weno.cuh's, in second differences D of the
// field, ordered from far upwind: D_{-2}, D_{-1}, D_0, D_{+1}) from the upwind first
// difference v3.  With e = -D the candidates are q_k = v3 + P_k/6,
// P = (5 D_{-1} - 2 D_{-2}, D_{-1} + 2 D_0, 4 D_0 - D_{+1}); A1..A3 = smooth_a of the
// third differences between neighbouring D.  The denominator is above 1e-21 and leaves
// rcp_refined's range only where it is about to overflow (differences of B near 1e38).
__device__ __forceinline__ double weno_shared(double dm2, double dm1, double d0, double dp1, double A1, double A2,
                                              double A3, double v3) {
    const double b1 = fma(3.0, dm1, -dm2), b2 = dm1 + d0, b3 = fma(3.0, d0, -dp1);
    double s1 = fma(b1, b1, A1), s2 = fma(b2, b2, A2), s3 = fma(b3, b3, A3);
    s1 *= s1;
    s2 *= s2;
    s3 *= s3;
    const double w1 = s2 * s3, w2 = 6.0 * (s1 * s3), w3 = 3.0 * (s1 * s2);   // weights 1, 6, 3 over s_k^2
    const double den = (w1 + w2) + w3;
    const double num = fma(w3, b3 + d0, fma(w2, b2 + d0, w1 * fma(2.0, b1, -dm1)));
    return fma(num * rcp_refined(den), 1.0 / 6.0, v3);
}

__device__ __forceinline__ void cp_async8(double* smem, const double* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Shared memory of a tw x th tile, in doubles: two planes of B with a 3-cell halo;
// second differences along x (columns -2 .. tw+1) and y (rows -2 .. th+1) and smooth_a
// at the half points between them
__host__ __device__ constexpr int tile_doubles(int tw, int th) {
    return 12 * (tw + 6) * (th + 6) + 12 * (tw + 4) * th + 12 * tw * (th + 4);
}
// The tiles that stress_shape chooses from: TW_MIN .. TW_MAX columns and the rows that
// NT threads hold.  The largest one's bytes are the kernels' limit of dynamic shared
// memory: the limit belongs to a kernel, not to a launch, and host threads with states on
// different grids launch the same kernel, so a limit set to each launch's own size could
// be lowered by another thread before the launch.
constexpr int TW_MIN = 8, TW_MAX = 64;
constexpr int largest_tile_bytes() {
    int most = 0;
    for (int tw = TW_MIN; tw <= TW_MAX; ++tw) {
        const int d = tile_doubles(tw, NT / tw);
        most = d > most ? d : most;
    }
    return most * (int)sizeof(double);
}
static_assert(2 * (largest_tile_bytes() + 1024) <= 228 * 1024, "two CTAs on an SM");
template <typename K>
cudaError_t raise_smem_limit(K kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, largest_tile_bytes());
}

// MODE: 0 = right-hand side only, 1 = update without history read, 2 = update reading
// and writing the history, 3 = update reading the history without writing it.
// One tile: tw x th columns (tile bx, by) over the z chunk bz of kz_chunk planes.
template <int MODEL, int MODE, bool DIFF>
__device__ __forceinline__ void stress_tile(const Geo<double>& g, const ModelConst& mc, const StressArgs<double>& a,
                                            int tw, int th, int kz_chunk, int bx, int by, int bz, double* sm) {
    constexpr bool RHS_ONLY = MODE == 0, READ_H = MODE >= 2, WRITE_H = MODE == 1 || MODE == 2;
    const int bw = tw + 6, bh = th + 6, BPL = bw * bh;
    const int dw = tw + 4, DXN = dw * th, DYN = tw * (th + 4);
    double* const smB = sm;                       // [2][6][BPL]
    double* const DX = smB + 12 * BPL;            // [6][DXN]
    double* const AX = DX + 6 * DXN;
    double* const DY = AX + 6 * DXN;              // [6][DYN]
    double* const AY = DY + 6 * DYN;
    EVP_DBG_DECL;
#ifdef EVP_DEBUG
    dbg_poison(reinterpret_cast<unsigned char*>(sm), (size_t)tile_doubles(tw, th) * sizeof(double));
    const size_t dbg_n = (size_t)g.nx * g.ny * g.nz;
    auto dbg_src_ok = [&](const double* p, int n) {
        for (int c = 0; c < 6; ++c)
            if (dbg_within(p, n, a.B[c], dbg_n)) return true;
        return dbg_within(p, n, a.H, dbg_n);
    };
    auto dbg_dst_ok = [&](const double* d, int n) { return d >= sm && d + n <= sm + tile_doubles(tw, th); };
#endif
    const int tid = threadIdx.x;
    const int i0 = bx * tw, j0 = by * th;
    const int k0 = bz * kz_chunk, k1 = min(k0 + kz_chunk, g.nz);
    const int ly = tid / tw, lx = tid - ly * tw;
    const bool own = ly < th;                     // threads beyond tw x th only help with the differences
    const int i = i0 + lx, j = j0 + ly;
    const bool active = own && i < g.nx && j < g.ny;
    const size_t plane = (size_t)g.nx * g.ny;
    auto kplane = [&](int k) { return (size_t)(k < 0 ? k + g.nz : (k >= g.nz ? k - g.nz : k)) * plane; };

    // ---- neighbours of the thread's cell (a ragged thread takes a cell of the grid, its results are not used)
    const int iw = i < g.nx ? i : pmod(i, g.nx);
    const int jw = j < g.ny ? j : (g.walls ? g.ny - 1 : pmod(j, g.ny));
    const int im = iw > 0 ? iw - 1 : g.nx - 1, ip = iw < g.nx - 1 ? iw + 1 : 0;
    // rows j-1, j+1 of u and w (odd mirror at walls) and row j-1 of v (zero below the wall)
    int jm = jw - 1, jp = jw + 1, fm = 1, fp = 1, fv = 1;
    if (jm < 0) {
        jm = g.walls ? 0 : g.ny - 1;
        fm = g.walls ? -1 : 1;
        fv = g.walls ? 0 : 1;
    }
    if (jp >= g.ny) {
        jp = g.walls ? g.ny - 1 : 0;
        fp = g.walls ? -1 : 1;
    }
    const int rc = jw * g.nx, rm = jm * g.nx, rp = jp * g.nx;
    const size_t col = (size_t)rc + iw;

    // plane kk of B with its halo into buffer kk & 1
    auto fetch = [&](int kk) {
        const size_t pb = kplane(kk);
        double* dst = smB + (kk & 1) * 6 * BPL;
        for (int e = tid; e < BPL; e += NT) {
            const int ry = e / bw, rx = e - ry * bw;
            const int gy = j0 + ry - 3;
            const int sy = g.walls ? min(max(gy, 0), g.ny - 1) : pmod(gy, g.ny);
            const size_t o = pb + (size_t)sy * g.nx + pmod(i0 + rx - 3, g.nx);
#pragma unroll
            for (int c = 0; c < 6; ++c)
                if (EVP_STAGE_OK(dst + c * BPL + e, a.B[c] + o, 1, false)) cp_async8(dst + c * BPL + e, a.B[c] + o);
        }
    };

    fetch(k0);
    cp_async_commit();

    // ---- z window of the cell's column: second differences at planes k-2 .. k+2,
    // smooth_a at the half planes between them, the last first difference
    double Dz[6][5], Az[6][4], vz[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        double q[7];
#pragma unroll
        for (int m = 0; m < 7; ++m) q[m] = __ldg(a.B[c] + kplane(k0 + m - 3) + col);
        double v = q[1] - q[0];
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const double vn = q[m + 2] - q[m + 1];
            Dz[c][m] = vn - v;
            v = vn;
        }
        vz[c] = v;
#pragma unroll
        for (int m = 0; m < 4; ++m) Az[c][m] = smooth_a(Dz[c][m + 1] - Dz[c][m]);
    }
    cp_async_wait_all();
    __syncthreads();

    const double qx = 0.25 * g.idx, qy = 0.25 * g.idy, qz = 0.25 * g.idz;
    const double inv_lam = mc.inv_lam;
    const int ob = (ly + 3) * bw + lx + 3;        // the cell in a plane of B
    unsigned bits = 0;

    for (int k = k0; k < k1; ++k) {
        if (k + 1 < k1) {
            fetch(k + 1);
            cp_async_commit();
        }
        const double* Bk = smB + (k & 1) * 6 * BPL;

        // ---- differences of the plane along x: runs of 8 columns of one row and component
        {
            const int nseg = (dw + 7) / 8;
            for (int q = tid; q < 6 * th * nseg; q += NT) {
                const int seg = q % nseg, line = q / nseg, c = line / th, r = line - c * th;
                const double* F = Bk + c * BPL + (r + 3) * bw;     // F[p .. p+2]: centre of column p is F[p+1]
                double* D = DX + c * DXN + r * dw;
                double* A = AX + c * DXN + r * dw;
                const int p0 = seg * 8;
                double v = F[p0 + 2] - F[p0 + 1];
                double d = v - (F[p0 + 1] - F[p0]);
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    const int p = p0 + m;
                    if (p < dw) D[p] = d;
                    if (p < dw - 1) {
                        const double vn = F[p + 3] - F[p + 2], dn = vn - v;
                        A[p] = smooth_a(dn - d);
                        v = vn;
                        d = dn;
                    }
                }
            }
        }
        // ---- along y: runs of 4 rows of one column and component
        {
            const int nrow = th + 4, nblk = (nrow + 3) / 4;
            for (int q = tid; q < 6 * tw * nblk; q += NT) {
                const int x = q % tw, t = q / tw, c = t / nblk, blk = t - c * nblk;
                const double* F = Bk + c * BPL + x + 3;            // rows p .. p+2: centre of row p is F[(p+1) bw]
                double* D = DY + c * DYN + x;
                double* A = AY + c * DYN + x;
                const int p0 = blk * 4;
                double v = F[(p0 + 2) * bw] - F[(p0 + 1) * bw];
                double d = v - (F[(p0 + 1) * bw] - F[p0 * bw]);
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    const int p = p0 + m;
                    if (p < nrow) D[p * tw] = d;
                    if (p < nrow - 1) {
                        const double vn = F[(p + 3) * bw] - F[(p + 2) * bw], dn = vn - v;
                        A[p * tw] = smooth_a(dn - d);
                        v = vn;
                        d = dn;
                    }
                }
            }
        }
        __syncthreads();

        if (own) {
            // ---- S1: centre velocity (doubled) and gradient (Reading 5)
            const size_t p0 = kplane(k), pm = kplane(k - 1), pp = kplane(k + 1);
            auto ld = [](const double* F, size_t p, int r, int x) { return __ldg(F + p + r + x); };
            const double Uc = ld(a.U, p0, rc, iw), Um = ld(a.U, p0, rc, im);
            const double Vc = ld(a.V, p0, rc, iw), Vm = scaled(ld(a.V, p0, rm, iw), fv);
            const double Wc = ld(a.W, p0, rc, iw), Wm = ld(a.W, pm, rc, iw);
            const double su = Um + Uc, sv = Vm + Vc, sw = Wm + Wc;
            double L[3][3];
            L[0][0] = (Uc - Um) * g.idx;
            L[1][1] = (Vc - Vm) * g.idy;
            L[2][2] = (Wc - Wm) * g.idz;
            L[0][1] = ((scaled(ld(a.U, p0, rp, im), fp) + scaled(ld(a.U, p0, rp, iw), fp))
                       - (scaled(ld(a.U, p0, rm, im), fm) + scaled(ld(a.U, p0, rm, iw), fm))) * qy;
            L[0][2] = ((ld(a.U, pp, rc, im) + ld(a.U, pp, rc, iw)) - (ld(a.U, pm, rc, im) + ld(a.U, pm, rc, iw))) * qz;
            L[1][0] = ((scaled(ld(a.V, p0, rm, ip), fv) + ld(a.V, p0, rc, ip))
                       - (scaled(ld(a.V, p0, rm, im), fv) + ld(a.V, p0, rc, im))) * qx;
            L[1][2] = ((scaled(ld(a.V, pp, rm, iw), fv) + ld(a.V, pp, rc, iw))
                       - (scaled(ld(a.V, pm, rm, iw), fv) + ld(a.V, pm, rc, iw))) * qz;
            L[2][0] = ((ld(a.W, pm, rc, ip) + ld(a.W, p0, rc, ip)) - (ld(a.W, pm, rc, im) + ld(a.W, p0, rc, im))) * qx;
            L[2][1] = ((scaled(ld(a.W, pm, rp, iw), fp) + scaled(ld(a.W, p0, rp, iw), fp))
                       - (scaled(ld(a.W, pm, rm, iw), fm) + scaled(ld(a.W, p0, rm, iw), fm))) * qy;
            const bool xpos = positive_bits(su), ypos = positive_bits(sv), zpos = positive_bits(sw);
            const double vx = fabs(su) * (0.5 * g.idx), vy = fabs(sv) * (0.5 * g.idy), vw = fabs(sw) * (0.5 * g.idz);

            // ---- B^{k-1} of the cell and the Table 1 closure
            double b0[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) b0[c] = Bk[c * BPL + ob];
            double F = 1.0, av = 1.0;
            if (MODEL == EVP_NEO_HOOKEAN) {
                F = 0.0;
                av = 0.0;
            } else if (MODEL == EVP_FENE_P) {
                const double d = mc.L2 - (b0[0] + b0[3] + b0[5]);
                F = refinable(d) ? div_refined(mc.L2, d) : mc.L2 / d;
                av = mc.a_fene;
            } else if (MODEL == EVP_SARAMITO) {
                double gm = mc.gmod;
                if (a.H) {
                    // two-phase mixture: polymer viscosity mu_p(H) of the cell
                    const double* hp = a.H + p0 + col;
                    const double Hc = EVP_DBG_OK(dbg_src_ok(hp, 1)) ? __ldg(hp) : 0.0;
                    gm = (a.mu_p1 * Hc + a.mu_p2 * (1.0 - Hc)) * inv_lam;
                }
                const double t0 = b0[0] - 1.0, t3 = b0[3] - 1.0, t5 = b0[5] - 1.0;
                const double tr3 = (t0 + t3 + t5) * (1.0 / 3.0);
                const double d0 = t0 - tr3, d3 = t3 - tr3, d5 = t5 - tr3;
                double m2 = fma(d5, d5, fma(d3, d3, d0 * d0)) * 0.5;
                m2 = fma(b0[4], b0[4], fma(b0[2], b0[2], fma(b0[1], b0[1], m2)));
                const double mag2 = (gm * gm) * m2;
                if (refinable(mag2)) {
                    const double f = fma(-mc.tau_y, rsqrt_refined(mag2), 1.0);
                    F = f > 0.0 ? f : 0.0;
                } else if (mag2 > 0.0) {
                    const double f = 1.0 - mc.tau_y / sqrt(mag2);
                    F = f > 0.0 ? f : 0.0;
                } else {
                    F = mc.tau_y > 0.0 ? 0.0 : 1.0;
                }
                av = F;
            }

            // ---- local artificial diffusion (Sec. 3.1): selected from B^{k-1} of the cell
            double kad = 0.0;
            if constexpr (DIFF) {
                const double det0 = b0[0] * (b0[3] * b0[5] - b0[4] * b0[4]) - b0[1] * (b0[1] * b0[5] - b0[4] * b0[2])
                                    + b0[2] * (b0[1] * b0[4] - b0[3] * b0[2]);
                bool hit = det0 < 0.0;
                if (MODEL == EVP_FENE_P) hit = hit || (b0[0] + b0[3] + b0[5] >= 0.95 * mc.L2);
                kad = hit ? mc.art_diff : 0.0;
            }

            // ---- advection, upper-convected terms, source and update per component
            const int sx = xpos ? 1 : -1, sy = ypos ? tw : -tw, sbx = xpos ? 1 : -1, sby = ypos ? bw : -bw;
            const int ox = ly * dw + lx + 2, oy = (ly + 2) * tw + lx;
            const int ax = ox + (xpos ? -2 : 1), ay = oy + (ypos ? -2 * tw : tw);
            const size_t up = (zpos ? pm : pp) + col;
            const size_t cell = p0 + col;
            const bool wr = active && EVP_DBG_OK(cell < plane * (size_t)g.nz);
            const double Fl = F * inv_lam, al = av * inv_lam;
            double bn[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const double* P = Bk + c * BPL + ob;
                const double* D = DX + c * DXN;
                const double* A = AX + c * DXN;
                const double tx = weno_shared(D[ox - 2 * sx], D[ox - sx], D[ox], D[ox + sx], A[ax], A[ax + sx], A[ax + 2 * sx],
                                              b0[c] - P[-sbx]);
                const double* E = DY + c * DYN;
                const double* Q = AY + c * DYN;
                const double ty = weno_shared(E[oy - 2 * sy], E[oy - sy], E[oy], E[oy + sy], Q[ay], Q[ay + sy], Q[ay + 2 * sy],
                                              b0[c] - P[-sby]);
                const double tz = weno_shared(zpos ? Dz[c][0] : Dz[c][4], zpos ? Dz[c][1] : Dz[c][3], Dz[c][2],
                                              zpos ? Dz[c][3] : Dz[c][1], zpos ? Az[c][0] : Az[c][3],
                                              zpos ? Az[c][1] : Az[c][2], zpos ? Az[c][2] : Az[c][1],
                                              b0[c] - __ldg(a.B[c] + up));
                const int ra = row_of(c), cb = col_of(c);
                double rt;
                if (is_diag(c)) {
                    double u = L[ra][0] * b0[symi(0, ra)];
                    u = fma(L[ra][1], b0[symi(1, ra)], u);
                    u = fma(L[ra][2], b0[symi(2, ra)], u);
                    rt = fma(2.0, u, fma(-Fl, b0[c], al));
                } else {
                    rt = -Fl * b0[c];
#pragma unroll
                    for (int q = 0; q < 3; ++q)
                        rt = fma(b0[symi(ra, q)], L[cb][q], fma(L[ra][q], b0[symi(q, cb)], rt));
                }
                rt = fma(-vw, tz, fma(-vy, ty, fma(-vx, tx, rt)));
                if (DIFF && kad != 0.0)
                    rt += kad * (D[ox] * (g.idx * g.idx) + E[oy] * (g.idy * g.idy) + Dz[c][2] * (g.idz * g.idz));
                if (RHS_ONLY) {
                    if (wr) a.RT[c][cell] = rt;
                } else {
                    double inc = a.dt_zeta * rt;
                    if (READ_H) inc = fma(a.dt_xi, wr ? a.RT[c][cell] : 0.0, inc);
                    bn[c] = b0[c] + inc;
                    if (wr) {
                        a.Bn[c][cell] = bn[c];
                        if (WRITE_H) a.RT[c][cell] = rt;
                    }
                }
            }
            if (wr && !RHS_ONLY) {
                bool fin = true;
                float s[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) {
                    fin = fin && finite_bits(bn[c]);
                    s[c] = narrow_f64(bn[c]);
                }
                if (!fin) bits |= EVP_BIT_NONFINITE;
                // trace limit and sign of det B: in single precision where its rounding (below
                // 1e-6 of the sum of the terms' magnitudes) leaves no doubt, else in double
                if (MODEL == EVP_FENE_P) {
                    const float tr32 = s[0] + s[3] + s[5], trm = fabsf(s[0]) + fabsf(s[3]) + fabsf(s[5]);
                    if (!(fmaf(1e-6f, trm, tr32) < (1.0f - 1e-6f) * mc.f_L2) && bn[0] + bn[3] + bn[5] >= mc.L2)
                        bits |= EVP_BIT_TRACE_LIMIT;
                }
                const float p35 = s[3] * s[5], p44 = s[4] * s[4], p15 = s[1] * s[5], p42 = s[4] * s[2], p14 = s[1] * s[4],
                            p32 = s[3] * s[2];
                const float det32 = s[0] * (p35 - p44) - s[1] * (p15 - p42) + s[2] * (p14 - p32);
                const float mag = fabsf(s[0]) * (fabsf(p35) + p44) + fabsf(s[1]) * (fabsf(p15) + fabsf(p42))
                                  + fabsf(s[2]) * (fabsf(p14) + fabsf(p32));
                if (!(det32 > 2e-6f * mag && mag < 1e37f && mag > 1e-25f)) {
                    const double det = bn[0] * (bn[3] * bn[5] - bn[4] * bn[4]) - bn[1] * (bn[1] * bn[5] - bn[4] * bn[2])
                                       + bn[2] * (bn[1] * bn[4] - bn[3] * bn[2]);
                    if (det < 0.0) bits |= EVP_BIT_DET_NEG;
                }
                if (a.S[0]) {
                    // summed polymer stress tau(B^k) + tau(B^{k-1}) of the cell (Table 1),
                    // the divergence term of the momentum step
                    const double gm = mc.gmod;
                    if (MODEL == EVP_FENE_P) {
                        const double dn = mc.L2 - (bn[0] + bn[3] + bn[5]);
                        const double Fn = refinable(dn) ? div_refined(mc.L2, dn) : mc.L2 / dn;
#pragma unroll
                        for (int c = 0; c < 6; ++c) {
                            const double d = is_diag(c) ? mc.a_fene : 0.0;
                            a.S[c][cell] = is_diag(c) ? gm * fma(Fn, bn[c], -d) + gm * fma(F, b0[c], -d)
                                                      : gm * (Fn * bn[c]) + gm * (F * b0[c]);
                        }
                    } else if (MODEL == EVP_NEO_HOOKEAN) {
#pragma unroll
                        for (int c = 0; c < 6; ++c) a.S[c][cell] = gm * bn[c] + gm * b0[c];
                    } else {
#pragma unroll
                        for (int c = 0; c < 6; ++c)
                            a.S[c][cell] = is_diag(c) ? gm * (bn[c] - 1.0) + gm * (b0[c] - 1.0) : gm * bn[c] + gm * b0[c];
                    }
                }
            }
        }

        // ---- next plane: move the z window; plane k+1 of B has landed, and every thread is
        // done with this plane's differences
        if (k + 1 < k1) {
            const size_t a3 = kplane(k + 3) + col, a4 = kplane(k + 4) + col;
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                const double vn = __ldg(a.B[c] + a4) - __ldg(a.B[c] + a3), dn = vn - vz[c];
                vz[c] = vn;
                const double An = smooth_a(dn - Dz[c][4]);
#pragma unroll
                for (int m = 0; m < 4; ++m) Dz[c][m] = Dz[c][m + 1];
                Dz[c][4] = dn;
#pragma unroll
                for (int m = 0; m < 3; ++m) Az[c][m] = Az[c][m + 1];
                Az[c][3] = An;
            }
            cp_async_wait_all();
            __syncthreads();
        }
    }
    if (bits) atomicOr(a.status, bits);
    EVP_DBG_REPORT(a.status);
}

template <int MODEL, int MODE, bool DIFF>
__global__ void __launch_bounds__(NT, 2)
k_stress(const Geo<double> g, const ModelConst mc, const StressArgs<double> a, int tw, int th, int kz_chunk) {
    pdl_wait();
    pdl_trigger();
    extern __shared__ __align__(16) unsigned char smraw[];
    stress_tile<MODEL, MODE, DIFF>(g, mc, a, tw, th, kz_chunk, blockIdx.x, blockIdx.y, blockIdx.z,
                                   reinterpret_cast<double*>(smraw));
}

// Batched form: a persistent grid over a work list of (member, tile x, tile y, z chunk)
template <int MODEL, int MODE>
__global__ void __launch_bounds__(NT, 2)
k_stress_batch(const __grid_constant__ StressBatch<double> p, const int4* __restrict__ work, int nwork) {
    extern __shared__ __align__(16) unsigned char smraw[];
    for (int w = blockIdx.x; w < nwork; w += gridDim.x) {
        const int4 t = __ldg(work + w);
        const StressMember<double>& m = p.m[t.x];
        stress_tile<MODEL, MODE, false>(m.g, m.mc, m.a, m.tw, m.th, m.kz, t.y, t.z, t.w,
                                        reinterpret_cast<double*>(smraw));
        __syncthreads();
    }
}

// FP64 instructions per thread and plane of a tw x th tile: the cell's own (about 665)
// and its share of the differences along x (43 per run of 8) and y (23 per run of 4)
int plane_cost(int tw, int th) {
    const int rx = (6 * th * ((tw + 4 + 7) / 8) + NT - 1) / NT, ry = (6 * tw * ((th + 4 + 3) / 4) + NT - 1) / NT;
    return 665 + 43 * rx + 23 * ry;
}

}  // namespace

// Tile shape of at most 128 cells with the fewest FP64 instructions over an nx x ny
// plane: ragged edges count as full tiles, small tiles pay for their halo.  72 x 54
// takes 18 x 7 (32 tiles) where 32 x 4 tiles would leave a quarter of the lanes idle
// (42 tiles of 32 x 4); a multiple of 32 in x keeps 32 x 4.
template <>
StressShape stress_shape<double>(int nx, int ny) {
    StressShape best{32, 4};
    long long cost = -1;
    for (int tw = TW_MIN; tw <= TW_MAX; ++tw) {
        int th = NT / tw;
        th = th > ny ? ny : th;
        const long long c = (long long)((nx + tw - 1) / tw) * ((ny + th - 1) / th) * plane_cost(tw, th);
        if (cost < 0 || c < cost || (c == cost && tw == 32)) {
            cost = c;
            best = {tw, th};
        }
    }
    return best;
}

// Planes per z chunk.  In units of FP64 instructions per thread a CTA costs its planes
// plus about 260 to start (its first plane's z window and the latency of its first
// loads); CTAs are handed out two to an SM and share its pipe, and one alone keeps the
// pipe 81 % busy.  The chunk with the smallest such time measured within 8 % of the best
// of a sweep on seven grids from 24 x 36 x 48 to 128 x 96 x 64.
template <>
int stress_planes<double>(int nx, int ny, int nz) {
    const StressShape s = stress_shape<double>(nx, ny);
    const long long tiles = (long long)((nx + s.tw - 1) / s.tw) * ((ny + s.th - 1) / s.th);
    const int pc = plane_cost(s.tw, s.th);
    int best = 1;
    double cost = -1.0;
    for (int kz = 1; kz <= nz && kz <= 64; ++kz) {
        const long long ctas = tiles * ((nz + kz - 1) / kz);
        const double c = ctas <= 152 ? 1.24 * kz * pc + 260.0 : 2.0 * ((ctas + 303) / 304) * (kz * pc + 260.0);
        if (cost < 0.0 || c < cost) {
            cost = c;
            best = kz;
        }
    }
    return best;
}

template <>
int stress_ctas_per_sm<double>() { return 1; }
template <>
int stress_cta_factor<double>() { return 2; }

template <>
cudaError_t launch_stress<double>(const Geo<double>& g, const ModelConst& mc, const StressArgs<double>& a,
                                  cudaStream_t st, const TimingHook& th) {
    const StressShape s = stress_shape<double>(g.nx, g.ny);
    const int kz = stress_planes<double>(g.nx, g.ny, g.nz);
    const dim3 grid((g.nx + s.tw - 1) / s.tw, (g.ny + s.th - 1) / s.th, (g.nz + kz - 1) / kz), block(NT);
    const size_t smem = (size_t)tile_doubles(s.tw, s.th) * sizeof(double);
    auto go = [&](auto kern) {
        if (cudaError_t e = raise_smem_limit(kern)) return e;
        return launch_k(kern, grid, block, smem, st, th.pdl, g, mc, a, s.tw, s.th, kz);
    };
    const int mode = a.rhs_only ? 0 : (!a.read_hist ? 1 : (a.write_hist ? 2 : 3));
    const int diff = mc.art_diff > 0.0 ? 1 : 0;
    cudaError_t e;
    th.b(K_STRESS);
    switch ((mc.model * 4 + mode) * 2 + diff) {
#define EVP_S(M, MD)                                                  \
    case (M * 4 + MD) * 2 + 0: e = go(k_stress<M, MD, false>); break; \
    case (M * 4 + MD) * 2 + 1: e = go(k_stress<M, MD, true>); break;
#define EVP_SM(M) EVP_S(M, 0) EVP_S(M, 1) EVP_S(M, 2) EVP_S(M, 3)
        EVP_SM(EVP_OLDROYD_B)
        EVP_SM(EVP_FENE_P)
        EVP_SM(EVP_SARAMITO)
        EVP_SM(EVP_NEO_HOOKEAN)
#undef EVP_SM
#undef EVP_S
        default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    th.e(K_STRESS);
    return cudaGetLastError();
}

template <>
cudaError_t launch_stress_batch<double>(const StressBatch<double>& p, int model, int mode, bool, const int4* work,
                                        int nwork, int ctas, size_t smem, cudaStream_t st) {
    if (nwork <= 0) return cudaSuccess;
    const dim3 grid(ctas < nwork ? ctas : nwork), block(NT);
    auto go = [&](auto kern) {
        if (cudaError_t e = raise_smem_limit(kern)) return e;
        return launch_k(kern, grid, block, smem, st, false, p, work, nwork);
    };
    switch (model * 4 + mode) {
#define EVP_S(M, MD) \
    case M * 4 + MD: return go(k_stress_batch<M, MD>);
#define EVP_SM(M) EVP_S(M, 1) EVP_S(M, 2) EVP_S(M, 3)
        EVP_SM(EVP_OLDROYD_B)
        EVP_SM(EVP_FENE_P)
        EVP_SM(EVP_SARAMITO)
#undef EVP_SM
#undef EVP_S
        default: return cudaErrorInvalidValue;
    }
}

// dynamic shared memory of a tile (the batch launches with its members' largest)
template <>
size_t stress_smem<double>(int nx, int ny) {
    const StressShape s = stress_shape<double>(nx, ny);
    return (size_t)tile_doubles(s.tw, s.th) * sizeof(double);
}

}  // namespace evp
