// Monitoring reductions of evp_diagnostics: kinetic energy, det B and tr B, the
// cells the Saramito closure of Table 1 leaves yielded (F > 0), and non-finite
// cells, all as FP64 evaluates them on the stored values.
//
//   k_diag        one (32 x 8 patch, z plane) work item after another per block
//                 (grid-stride over all items), one partial record per block;
//                 k_diag_f32 for single-precision states
//   k_diag_final  one block folds the partial records in index order
//
// Both reductions run in a fixed order (thread-local sums, then a fixed shuffle
// tree, then the warps in index order, then the blocks in index order), so a
// repeated call on the same fields returns the same bits.  Not on the step's
// path: a monitoring call of 9 words a cell, bound by instruction issue in single
// precision and by the FP64 pipe in double.
#include "evp_internal.cuh"

namespace evp {

namespace {

struct Acc {
    double ke, dmin, tmax;
    unsigned long long yielded, bad;
};

__device__ __forceinline__ void fold(Acc& a, const Acc& b) {
    a.ke += b.ke;
    a.dmin = fmin(a.dmin, b.dmin);   // fmin/fmax skip a NaN operand
    a.tmax = fmax(a.tmax, b.tmax);
    a.yielded += b.yielded;
    a.bad += b.bad;
}

__device__ __forceinline__ Acc shfl(const Acc& a, int o) {
    Acc r;
    r.ke = __shfl_xor_sync(0xffffffffu, a.ke, o);
    r.dmin = __shfl_xor_sync(0xffffffffu, a.dmin, o);
    r.tmax = __shfl_xor_sync(0xffffffffu, a.tmax, o);
    r.yielded = __shfl_xor_sync(0xffffffffu, a.yielded, o);
    r.bad = __shfl_xor_sync(0xffffffffu, a.bad, o);
    return r;
}

// Fold the block's 256 accumulators; thread 0 returns the result.
__device__ __forceinline__ Acc block_fold(Acc a) {
    __shared__ Acc red[8];
    const int t = threadIdx.y * blockDim.x + threadIdx.x, lane = t & 31, warp = t >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) fold(a, shfl(a, o));
    if (lane == 0) red[warp] = a;
    __syncthreads();
    if (t == 0) {
        a = red[0];
        for (int q = 1; q < 8; ++q) fold(a, red[q]);
    }
    return a;
}

__device__ __forceinline__ Acc acc_zero() {
    Acc a;
    a.ke = 0.0;
    a.dmin = __longlong_as_double(0x7ff0000000000000ll);    // +inf
    a.tmax = __longlong_as_double((long long)0xfff0000000000000ull);   // -inf
    a.yielded = 0ull;
    a.bad = 0ull;
    return a;
}

// det of the symmetric B (xx, xy, xz, yy, yz, zz) by cofactor expansion along the
// first row; each product and sum rounded in the written order (no contraction)
__device__ __forceinline__ double det_sym(const double b[6]) {
    const double c0 = __dsub_rn(__dmul_rn(b[3], b[5]), __dmul_rn(b[4], b[4]));
    const double c1 = __dsub_rn(__dmul_rn(b[1], b[5]), __dmul_rn(b[4], b[2]));
    const double c2 = __dsub_rn(__dmul_rn(b[1], b[4]), __dmul_rn(b[3], b[2]));
    return __dadd_rn(__dsub_rn(__dmul_rn(b[0], c0), __dmul_rn(b[1], c1)), __dmul_rn(b[2], c2));
}

// |tau^d| > tau_y for tau = gm (B - I), |tau^d|^2 = 1/2 tau^d_ij tau^d_ij (Table 1,
// Saramito row), rounded in the written order
__device__ __forceinline__ bool yielded_cell(const double b[6], double gm, double tau_y) {
    double t[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) t[c] = __dmul_rn(gm, (c == 0 || c == 3 || c == 5) ? __dsub_rn(b[c], 1.0) : b[c]);
    const double tr3 = __ddiv_rn(__dadd_rn(__dadd_rn(t[0], t[3]), t[5]), 3.0);
    const double d0 = __dsub_rn(t[0], tr3), d3 = __dsub_rn(t[3], tr3), d5 = __dsub_rn(t[5], tr3);
    double m2 = __dmul_rn(0.5, __dadd_rn(__dadd_rn(__dmul_rn(d0, d0), __dmul_rn(d3, d3)), __dmul_rn(d5, d5)));
    m2 = __dadd_rn(m2, __dmul_rn(t[1], t[1]));
    m2 = __dadd_rn(m2, __dmul_rn(t[2], t[2]));
    m2 = __dadd_rn(m2, __dmul_rn(t[4], t[4]));
    return __dsqrt_rn(m2) > tau_y;
}

// A float as an unsigned integer of the same order (a NaN beyond the infinities)
__device__ __forceinline__ unsigned order_key(float x) {
    const unsigned b = __float_as_uint(x);
    return b ^ ((int)b < 0 ? 0xffffffffu : 0x80000000u);
}

// A thread's extreme value so far as an interval [lo, hi] that its single-precision form
// and the form's error bound leave, with the cell's values for the exact one
template <int N>
struct Kept {
    float lo, hi, b[N];
};
// Offer a cell of interval [lo, hi] (MIN: the smallest is kept, else the largest).  Returns
// false where the intervals overlap, so that neither cell can be dropped.
template <bool MIN, int N>
__device__ __forceinline__ bool offer(Kept<N>& k, float lo, float hi, const float (&b)[N]) {
    const bool worse = MIN ? lo > k.hi : hi < k.lo, better = MIN ? hi < k.lo : lo > k.hi;
    if (better) {
        k.lo = lo;
        k.hi = hi;
#pragma unroll
        for (int c = 0; c < N; ++c) k.b[c] = b[c];
    }
    return worse || better;
}

// The same reductions of single-precision states.  In FP64 throughout a cell costs about
// 95 instructions of GB300's FP64 pipe (64 cycles each per scheduler): 630 us on 256 x 128
// x 128, where reading the nine fields takes 22.  Here a cell is settled in single
// precision where its error bound leaves no doubt: each thread keeps the cell of its
// smallest determinant and of its largest trace and evaluates in FP64, as k_diag does,
// only cells whose intervals overlap, at the end those that the block's bounds leave, and
// deviators within their error of the yield stress.  The results are k_diag's, bit for
// bit, except the kinetic energy's order of sums; the squares are summed in FP64, widened
// by integer operations.  79 us, bound by instruction issue (about 300 a warp and item).
// Where every cell ties (a fluid at rest with B = I) each is evaluated in both forms: the
// whole evp_diagnostics call takes 350 us on 256 x 128 x 128 then, 910 in FP64 throughout.
__global__ void __launch_bounds__(256) k_diag_f32(const Geo<float> g, const DiagArgs<float> a,
                                                  DiagPart* __restrict__ parts) {
    __shared__ unsigned best[2];       // keys: upper bound of the smallest det, lower bound of the largest trace
    // 32-bit work items (16 cells or more each, so that a device's memory holds far fewer
    // than 2^31): 79 us against 94 with their division in 64 bits
    const unsigned tx = (g.nx + 31) / 32, tiles = tx * ((g.ny + 7) / 8), items = tiles * g.nz;
    const size_t plane = (size_t)g.nx * g.ny;
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        best[0] = 0xffffffffu;
        best[1] = 0u;
    }
    __syncthreads();
    const float inf = __int_as_float(0x7f800000);
    Kept<6> kd;
    Kept<3> kt;
    kd.lo = kd.hi = inf;               // nothing kept yet
    kt.lo = kt.hi = -inf;
    Acc acc = acc_zero();
    const float ty2 = (float)a.tau_y * (float)a.tau_y;
    const bool ty_ok = ty2 > 1e-30f && ty2 < 1e30f;
    for (unsigned w = blockIdx.x; w < items; w += gridDim.x) {
        const unsigned k = w / tiles, t = w - k * tiles, ty = t / tx;
        const int i = (t - ty * tx) * 32 + threadIdx.x, j = ty * 8 + threadIdx.y;
        const bool in = i < g.nx && j < g.ny;
        const size_t o = in ? (size_t)k * plane + (size_t)j * g.nx + i : 0;
        const float u = __ldg(a.U + o), v = __ldg(a.V + o), wv = __ldg(a.W + o);
        float b[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
        if (a.B[0]) {
#pragma unroll
            for (int c = 0; c < 6; ++c) b[c] = __ldg(a.B[c] + o);
        }
        bool bad = !isfinite(u) || !isfinite(v) || !isfinite(wv);
        if (in) {
            const double ud = widen_f32(u), vd = widen_f32(v), wd = widen_f32(wv);
            acc.ke = fma(wd, wd, fma(vd, vd, fma(ud, ud, acc.ke)));
        }
        if (a.B[0]) {
#pragma unroll
            for (int c = 0; c < 6; ++c) bad = bad || !isfinite(b[c]);
            // ---- det B and tr B with the sums of their terms' magnitudes: the errors are below
            // 16 roundings of 2^-24 of those (1e-6)
            const float p35 = b[3] * b[5], p44 = b[4] * b[4], p15 = b[1] * b[5], p42 = b[4] * b[2], p14 = b[1] * b[4],
                        p32 = b[3] * b[2];
            const float det = b[0] * (p35 - p44) - b[1] * (p15 - p42) + b[2] * (p14 - p32);
            const float dm = fabsf(b[0]) * (fabsf(p35) + p44) + fabsf(b[1]) * (fabsf(p15) + fabsf(p42))
                             + fabsf(b[2]) * (fabsf(p14) + fabsf(p32));
            const float tr = b[0] + b[3] + b[5], tm = fabsf(b[0]) + fabsf(b[3]) + fabsf(b[5]);
            const bool dok = dm > 1e-25f && dm < 1e30f, tok = tm < 1e30f;
            const float de = 1e-6f * dm, te = 1e-6f * tm, diag[3] = {b[0], b[3], b[5]};
            const bool need_d = in && !(dok && offer<true>(kd, det - de, det + de, b));
            const bool need_t = in && !(tok && offer<false>(kt, tr - te, tr + te, diag));
            // ---- the yield test, by the squares
            bool y = a.yield_mode == 1, need_y = false;
            if (a.yield_mode == 2) {
                const float gm = a.H ? (float)a.mp1 * __ldg(a.H + o) * (float)a.inv_lam : (float)a.gm;
                const float t0 = gm * (b[0] - 1.f), t3 = gm * (b[3] - 1.f), t5 = gm * (b[5] - 1.f);
                const float t1 = gm * b[1], t2 = gm * b[2], t4 = gm * b[4];
                const float t13 = (t0 + t3 + t5) * (1.f / 3.f), d0 = t0 - t13, d3 = t3 - t13, d5 = t5 - t13;
                const float off = t1 * t1 + t2 * t2 + t4 * t4, ts = fabsf(t0) + fabsf(t3) + fabsf(t5);
                const float m2 = 0.5f * (d0 * d0 + d3 * d3 + d5 * d5) + off;
                const float err = 4e-6f * (fmaf(ts, ts, off) + ty2);
                y = m2 - ty2 > err;
                need_y = in && !(ty_ok && (y || ty2 - m2 > err));
                if (a.tau_y == 0.0) {
                    y = true;
                    need_y = false;
                }
            }
            if (need_d || need_t || need_y) {
                double bd[6];
#pragma unroll
                for (int c = 0; c < 6; ++c) bd[c] = (double)b[c];
                if (need_d) acc.dmin = fmin(acc.dmin, det_sym(bd));
                if (need_t) acc.tmax = fmax(acc.tmax, __dadd_rn(__dadd_rn(bd[0], bd[3]), bd[5]));
                if (need_y) {
                    const double gm = a.H ? __dmul_rn(__dmul_rn(a.mp1, (double)__ldg(a.H + o)), a.inv_lam) : a.gm;
                    y = yielded_cell(bd, gm, a.tau_y);
                }
            }
            acc.yielded += in && y ? 1ull : 0ull;
        }
        acc.bad += in && bad ? 1ull : 0ull;
    }
    // ---- the kept cells: the block's bounds first, then what they leave in FP64
    if (a.B[0]) {
        const unsigned du = __reduce_min_sync(0xffffffffu, order_key(kd.hi));
        const unsigned tl = __reduce_max_sync(0xffffffffu, order_key(kt.lo));
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&best[0], du);
            atomicMax(&best[1], tl);
        }
        __syncthreads();
        if (kd.lo < inf && order_key(kd.lo) <= best[0]) {
            double bd[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) bd[c] = (double)kd.b[c];
            acc.dmin = fmin(acc.dmin, det_sym(bd));
        }
        if (kt.hi > -inf && order_key(kt.hi) >= best[1])
            acc.tmax = fmax(acc.tmax, __dadd_rn(__dadd_rn((double)kt.b[0], (double)kt.b[1]), (double)kt.b[2]));
    }
    acc = block_fold(acc);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        DiagPart p;
        p.ke = acc.ke;
        p.min_det = acc.dmin;
        p.max_tr = acc.tmax;
        p.yielded = acc.yielded;
        p.nonfinite = acc.bad;
        parts[blockIdx.x] = p;
    }
}

template <typename T>
__global__ void __launch_bounds__(256) k_diag(const Geo<T> g, const DiagArgs<T> a, DiagPart* __restrict__ parts) {
    const int tx = (g.nx + 31) / 32;
    const long long tiles = (long long)tx * ((g.ny + 7) / 8);
    const long long items = tiles * g.nz;
    const size_t plane = (size_t)g.nx * g.ny;
    Acc acc = acc_zero();
    for (long long w = blockIdx.x; w < items; w += gridDim.x) {
        const int t = (int)(w % tiles), k = (int)(w / tiles);
        const int i = (t % tx) * 32 + threadIdx.x, j = (t / tx) * 8 + threadIdx.y;
        if (i >= g.nx || j >= g.ny) continue;
        const size_t o = (size_t)k * plane + (size_t)j * g.nx + i;
        const double u = (double)__ldg(a.U + o), v = (double)__ldg(a.V + o), wv = (double)__ldg(a.W + o);
        bool bad = !isfinite(u) || !isfinite(v) || !isfinite(wv);
        acc.ke += u * u + v * v + wv * wv;
        if (a.B[0]) {
            double b[6];
#pragma unroll
            for (int c = 0; c < 6; ++c) {
                b[c] = (double)__ldg(a.B[c] + o);
                bad = bad || !isfinite(b[c]);
            }
            acc.dmin = fmin(acc.dmin, det_sym(b));
            acc.tmax = fmax(acc.tmax, __dadd_rn(__dadd_rn(b[0], b[3]), b[5]));
            bool y = a.yield_mode == 1;
            if (a.yield_mode == 2) {
                const double gm = a.H ? __dmul_rn(__dmul_rn(a.mp1, (double)__ldg(a.H + o)), a.inv_lam) : a.gm;
                y = a.tau_y == 0.0 || yielded_cell(b, gm, a.tau_y);
            }
            acc.yielded += y ? 1ull : 0ull;
        }
        acc.bad += bad ? 1ull : 0ull;
    }
    acc = block_fold(acc);
    if (threadIdx.x == 0 && threadIdx.y == 0) {
        DiagPart p;
        p.ke = acc.ke;
        p.min_det = acc.dmin;
        p.max_tr = acc.tmax;
        p.yielded = acc.yielded;
        p.nonfinite = acc.bad;
        parts[blockIdx.x] = p;
    }
}

__global__ void __launch_bounds__(256) k_diag_final(const DiagPart* __restrict__ parts, int nparts,
                                                    const unsigned long long* __restrict__ maxdiv,
                                                    DiagResult* __restrict__ out) {
    Acc acc = acc_zero();
    for (int q = threadIdx.x; q < nparts; q += blockDim.x) {
        Acc b;
        b.ke = parts[q].ke;
        b.dmin = parts[q].min_det;
        b.tmax = parts[q].max_tr;
        b.yielded = parts[q].yielded;
        b.bad = parts[q].nonfinite;
        fold(acc, b);
    }
    acc = block_fold(acc);
    if (threadIdx.x == 0) {
        out->p.ke = acc.ke;
        out->p.min_det = acc.dmin;
        out->p.max_tr = acc.tmax;
        out->p.yielded = acc.yielded;
        out->p.nonfinite = acc.bad;
        out->maxdiv = *maxdiv;
    }
}

}  // namespace

template <typename T>
cudaError_t launch_diag(const Geo<T>& g, const DiagArgs<T>& a, DiagPart* parts, const unsigned long long* maxdiv,
                        DiagResult* out, cudaStream_t st) {
    const long long items = (long long)((g.nx + 31) / 32) * ((g.ny + 7) / 8) * g.nz;
    const int nb = (int)(items < DIAG_BLOCKS ? items : DIAG_BLOCKS);
    if constexpr (sizeof(T) == 4) k_diag_f32<<<nb, dim3(32, 8, 1), 0, st>>>(g, a, parts);
    else k_diag<T><<<nb, dim3(32, 8, 1), 0, st>>>(g, a, parts);
    k_diag_final<<<1, 256, 0, st>>>(parts, nb, maxdiv, out);
    return cudaGetLastError();
}

template cudaError_t launch_diag<float>(const Geo<float>&, const DiagArgs<float>&, DiagPart*, const unsigned long long*,
                                        DiagResult*, cudaStream_t);
template cudaError_t launch_diag<double>(const Geo<double>&, const DiagArgs<double>&, DiagPart*,
                                         const unsigned long long*, DiagResult*, cudaStream_t);

}  // namespace evp
