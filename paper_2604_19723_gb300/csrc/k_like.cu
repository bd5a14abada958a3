// Per-particle update messages iota~ and nu~ (Supplementary Sec. S-V); the PF message
// kappa~ is in k_kappa.cu.
//
// Every message is a complex Gaussian whose quadratic form is evaluated in
// its variational (regularised least-squares) form,
//     e^H (eta I + M M^H)^-1 e = min_y |e - M y|^2/eta + |y|^2,
// with the residual r = e - M y* formed element by element.  In this form
// the FP32 error of the result is relative to the residual energy (the
// noise floor) rather than to the signal energy, and errors in y* enter
// only at second order.
//
//  iota~(x^p) for every p, summed over j (columns sqrt(pi (gamma + |mu|^2 (1 - pi))) psi_s):
//     log iota = -|r|^2/eta_bar - |y|^2 - log det(I + D G D/eta_bar) - Nz log(pi eta_bar).
//  nu~(eta^(j,p)) for every (j, p) through the tridiagonal form of G = M^H M.
//
// Steering vectors psi_s^(j,p) = lambda/(4 pi d) e^{-i 2 pi d/lambda} (b kron a_y kron a_z)
// (eq. array-response, unit-modulus-array-response) are rebuilt in FP32 from the
// per-(p, s, j) geometry records of k_geom (FP64 distance and direction).
#include "bp_internal.cuh"
#include "bp_kernels.cuh"

namespace bp {

// ---------------------------------------------------------------- iota (warp per particle)
// Fast path in FP32: factors from the geometry records, g = Psi^H z, the Gram
// G = Psi^H Psi from the Kronecker factors, Cholesky of eta_bar I + D G D,
// solves, and the element-wise residual (squared sums in FP64).  The FP32
// log det loses accuracy when a pivot cancels, i.e. when a column nearly lies
// in the span of the previous ones (1 - |rho|^2 small, e.g. a fresh birth PF
// next to a real component): each pivot's ratio A_kk / L_kk^2 measures that
// loss, and particles with sqrt(sum ratio^2) > IOTA_RATIO_MAX are queued for
// k_iota_blk, which recomputes them with a float-float Gram and factorisation.
// The FP32 log det error per pivot is about 8 eps ratio (measured), so the
// bound keeps unrepaired particles within ~5e-5 in log-likelihood.
constexpr float IOTA_RATIO_MAX = 100.0f;
constexpr double LOG_PI = 1.14472988584940017414;   // log(pi)

__device__ inline int tri(int i, int j) { return i * (i + 1) / 2 + j; }
__device__ inline void tri_ab(int t, int& a, int& b) {
    a = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((a + 1) * (a + 2) / 2 <= t) ++a;
    while (a * (a + 1) / 2 > t) --a;
    b = t - a * (a + 1) / 2;
}

// per-warp shared memory of the FP32 path (float2 units)
__host__ __device__ inline size_t iota32_warp_f2(int S, int nfac, int Nf) {
    return (size_t)S * nfac + 4 * (size_t)S + (size_t)S * (S + 1) / 2 + (size_t)S * Nf + (size_t)S;
}

__global__ void k_iota(DevGeom G, DevParams Pm, DevState D, int S, const float* z) {
    extern __shared__ float2 sm32[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int wpb = blockDim.x >> 5;
    const int P = Pm.P, J = G.J, Nz = G.Nz, Nm = G.My * G.Mz, Nf = G.Nf;
    const int nfac = Nf + G.My + G.Mz;
    float2* zs = sm32;                                                    // [Nz]
    float2* base = zs + Nz + wib * iota32_warp_f2(S, nfac, Nf);
    float2* fac = base;                                                   // [S][nfac]
    float2* cS = fac + (size_t)S * nfac;                                  // [S] carrier*amplitude
    float2* cmS = cS + S;                                                 // [S] pi mu, then w
    float2* gS = cmS + S;                                                 // [S] g, rhs, solution
    float2* dS = gS + S;                                                  // [S] (d, A_kk)
    float2* Am = dS + S;                                                  // [S(S+1)/2] packed lower
    float2* gpart = Am + (size_t)S * (S + 1) / 2;                         // [S][Nf] partial g
    const int p = blockIdx.x * wpb + wib;
    const bool act = p < P;
    const int pp = act ? p : 0;
    const float* phi = D.phi[D.cur];
    __shared__ double lg_eb[J_MAX], inv_eb[J_MAX];
    if (threadIdx.x < J) { lg_eb[threadIdx.x] = log(D.eta_bar[threadIdx.x]); inv_eb[threadIdx.x] = 1.0 / D.eta_bar[threadIdx.x]; }
    double total = 0.0;
    float ratio2 = 0.f;
    for (int j = 0; j < J; ++j) {
        __syncthreads();
        for (int k = threadIdx.x; k < Nz; k += blockDim.x)
            zs[k] = make_float2(z[2 * (j * Nz + k)], z[2 * (j * Nz + k) + 1]);
        __syncthreads();
        const double eb = D.eta_bar[j];
        const float ebf = (float)eb;
        // 1. factors and coefficients, lanes over s
        for (int s = lane; s < S; s += 32) {
            const float* ph = phi + (size_t)s * 6 * P;
            float2* fs = fac + (size_t)s * nfac;
            const size_t gi = ((size_t)s * J + j) * P + pp;
            cS[s] = factors_from_geo(G, D.geo[gi], D.geo_lo[gi], fs, fs + Nf, fs + Nf + G.My, 1);
            const float pi = (float)(D.zeta[s * J + j] * D.W[s]);
            const float gm = ph[3 * P + pp], mr = ph[4 * P + pp], mi = ph[5 * P + pp];
            dS[s] = make_float2(sqrtf(fmaxf(pi * (gm + (mr * mr + mi * mi) * (1.0f - pi)), 0.0f)), 0.f);
            cmS[s] = make_float2(pi * mr, pi * mi);
        }
        __syncwarp();
        // 2. g_s = psi_s^H z: tasks (s, f) contract over the antennas, then sum over f
        for (int t = lane; t < S * Nf; t += 32) {
            const int s = t / Nf, f = t - s * Nf;
            const float2* fs = fac + (size_t)s * nfac;
            float2 accy = make_float2(0.f, 0.f);
            for (int y = 0; y < G.My; ++y) {
                float2 accm = make_float2(0.f, 0.f);
                for (int m = 0; m < G.Mz; ++m) {
                    const float2 u = cmulc(fs[Nf + G.My + m], zs[f * Nm + y * G.Mz + m]);
                    accm.x += u.x; accm.y += u.y;
                }
                const float2 u = cmulc(fs[Nf + y], accm);
                accy.x += u.x; accy.y += u.y;
            }
            gpart[t] = cmulc(fs[f], accy);
        }
        // 3. Gram (packed lower) from the Kronecker factors
        const int npair = S * (S + 1) / 2;
        for (int t = lane; t < npair; t += 32) {
            int a, b;
            tri_ab(t, a, b);
            const float2* fa = fac + (size_t)a * nfac;
            const float2* fb2 = fac + (size_t)b * nfac;
            float2 sf = make_float2(0.f, 0.f), sy = sf, sz = sf;
            for (int f = 0; f < Nf; ++f) { const float2 u = cmulc(fa[f], fb2[f]); sf.x += u.x; sf.y += u.y; }
            for (int y = Nf; y < Nf + G.My; ++y) { const float2 u = cmulc(fa[y], fb2[y]); sy.x += u.x; sy.y += u.y; }
            for (int m = Nf + G.My; m < nfac; ++m) { const float2 u = cmulc(fa[m], fb2[m]); sz.x += u.x; sz.y += u.y; }
            Am[t] = cmul(cmulc(cS[a], cS[b]), cmul(sf, cmul(sy, sz)));
        }
        __syncwarp();
        for (int s = lane; s < S; s += 32) {
            float2 acc = make_float2(0.f, 0.f);
            for (int f = 0; f < Nf; ++f) { acc.x += gpart[s * Nf + f].x; acc.y += gpart[s * Nf + f].y; }
            gS[s] = cmulc(cS[s], acc);
        }
        __syncwarp();
        // 4. rhs_a = d_a (g_a - sum_b G_ab cm_b)
        for (int a = lane; a < S; a += 32) {
            float2 acc = gS[a];
            for (int b = 0; b < S; ++b) {
                const float2 gab = (b <= a) ? Am[tri(a, b)] : make_float2(Am[tri(b, a)].x, -Am[tri(b, a)].y);
                const float2 u = cmul(gab, cmS[b]);
                acc.x -= u.x; acc.y -= u.y;
            }
            gS[a] = make_float2(dS[a].x * acc.x, dS[a].x * acc.y);
        }
        __syncwarp();
        // 5. A = eta_bar I + D G D, keep the original diagonal; Cholesky in place
        for (int t = lane; t < npair; t += 32) {
            int a, b;
            tri_ab(t, a, b);
            const float dd = dS[a].x * dS[b].x;
            const float2 v = Am[t];
            Am[t] = make_float2(dd * v.x + (a == b ? ebf : 0.f), dd * v.y);
            if (a == b) dS[a].y = dd * v.x + ebf;
        }
        __syncwarp();
        ffexp det{ff{1.f, 0.f}, 0};
        for (int k = 0; k < S; ++k) {
            const float piv = fmaxf(Am[tri(k, k)].x, 1e-30f);
            const float dk = sqrtf(piv);
            ffexp_mul(det, ff{piv, 0.f});
            const float rk = dS[k].y / piv;
            ratio2 += rk * rk;
            __syncwarp();
            for (int i = k + 1 + lane; i < S; i += 32) {
                const float2 v = Am[tri(i, k)];
                Am[tri(i, k)] = make_float2(v.x / dk, v.y / dk);
            }
            if (lane == 0) Am[tri(k, k)] = make_float2(dk, 0.f);
            __syncwarp();
            const int n = S - k - 1;
            for (int t = lane; t < n * (n + 1) / 2; t += 32) {
                int a, c;
                tri_ab(t, a, c);
                const int i = k + 1 + a, cc = k + 1 + c;
                const float2 u = cmul(Am[tri(i, k)], make_float2(Am[tri(cc, k)].x, -Am[tri(cc, k)].y));
                Am[tri(i, cc)].x -= u.x; Am[tri(i, cc)].y -= u.y;
            }
            __syncwarp();
        }
        // 6. solve L L^H y = rhs
        for (int i = 0; i < S; ++i) {
            float2 acc = make_float2(0.f, 0.f);
            for (int b = lane; b < i; b += 32) { const float2 u = cmul(Am[tri(i, b)], gS[b]); acc.x += u.x; acc.y += u.y; }
            acc.x = warp_sum_f(acc.x); acc.y = warp_sum_f(acc.y);
            if (lane == 0) { const float dd = Am[tri(i, i)].x; gS[i] = make_float2((gS[i].x - acc.x) / dd, (gS[i].y - acc.y) / dd); }
            __syncwarp();
        }
        for (int i = S - 1; i >= 0; --i) {
            float2 acc = make_float2(0.f, 0.f);
            for (int b = i + 1 + lane; b < S; b += 32) { const float2 u = cmulc(Am[tri(b, i)], gS[b]); acc.x += u.x; acc.y += u.y; }
            acc.x = warp_sum_f(acc.x); acc.y = warp_sum_f(acc.y);
            if (lane == 0) { const float dd = Am[tri(i, i)].x; gS[i] = make_float2((gS[i].x - acc.x) / dd, (gS[i].y - acc.y) / dd); }
            __syncwarp();
        }
        // 7. w = cm + d y; |y|^2 (exact squares, float-float sums)
        ff yy{0.f, 0.f};
        for (int a = lane; a < S; a += 32) {
            const float2 y = gS[a];
            ff_acc_sq(yy, y);
            cmS[a] = make_float2(cmS[a].x + dS[a].x * y.x, cmS[a].y + dS[a].x * y.y);
        }
        yy = warp_sum_ff(yy);
        __syncwarp();
        // 8. residual z - sum_s w_s psi_s, element-wise
        ff rr{0.f, 0.f};
        for (int k = lane; k < Nz; k += 32) {
            const int f = k / Nm, ym = k - f * Nm, y = ym / G.Mz, m = ym - y * G.Mz;
            float2 acc = zs[k];
            for (int s = 0; s < S; ++s) {
                const float2* fs = fac + (size_t)s * nfac;
                const float2 u = cmul(cmul(cmS[s], cS[s]), cmul(fs[f], cmul(fs[Nf + y], fs[Nf + G.My + m])));
                acc.x -= u.x; acc.y -= u.y;
            }
            ff_acc_sq(rr, acc);
        }
        rr = warp_sum_ff(rr);
        const double lg = lg_eb[j];
        total += -(ff_to_d(rr) * inv_eb[j] + ff_to_d(yy)) - (ffexp_log(det) - S * lg) - Nz * (LOG_PI + lg);
    }
    if (act && lane == 0) {
        D.lw_x[p] = total;
        if (sqrtf(ratio2) > IOTA_RATIO_MAX) {
            const int slot = atomicAdd(&D.flags[0], 1);
            if (bp_in_range(slot, P, D.kerr)) D.flags[1 + slot] = p;
        }
    }
}

// ---------------------------------------------------------------- iota, float-float Gram and Cholesky
// For the particles the FP32 path flags (or for every particle when S is large):
// the same log-likelihood with the pivots of eta_bar I + D G D kept to ~44 bits,
// so that nearly coinciding columns lose nothing.  One block per
// particle; the lower triangle of A (S <= 64) lives in registers, distributed as
// row pairs (rp, 63 - rp) x column groups c = NCG q + cg (32 NCG threads), so that
// every thread holds about S(S+1)/(64 NCG) entries and every row's scaled column
// entry is formed by NCG threads only.
//  - Gram: G'_ab = (sum_f conj(b'_af) b'_bf)(sum_y ..)(sum_m ..) of the unit-modulus
//    factors, each sum exact to ~2^-40 (products split on a fixed 2^-16 grid,
//    remainders by FMA); A_ab = A_a d_a A_b d_b G'_ab + eta_bar delta_ab in float-float.
//  - Right-looking Cholesky, one barrier per pivot: step k scales column k by
//    1/pivot, subtracts the rank-one term from the trailing entries, and the owners
//    of column k+1 publish it (and its pivot with the reciprocal) for step k+1.
//  - Forward/back solves with the FP32 parts of L, residual in FP32 with FP64 sums
//    (both enter the variational form only at second order).
constexpr int IB_SMAX = 64;
constexpr int IOTA_BLK_NCG = 8;   // column groups: 256 threads, 12 register slots per thread

__device__ inline cff fx_dotc(const float2* x, const float2* y, int n) {
    // sum_k conj(x_k) y_k for |x_k|, |y_k| <= 1 + O(eps), n <= 127: fmaf(a, b, M) - M
    // rounds a*b to a multiple of 2^-16 (M = 1.5 * 2^7), so the grid parts add
    // exactly while |sum| < 256, and fmaf(a, b, -grid part) is the remainder.
    const float M = 192.0f;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    for (int k = 0; k < n; ++k) {
        const float2 a = x[k], b = y[k];
        float t = __fsub_rn(fmaf(a.x, b.x, M), M);
        rh = __fadd_rn(rh, t); rl = __fadd_rn(rl, fmaf(a.x, b.x, -t));
        t = __fsub_rn(fmaf(a.y, b.y, M), M);
        rh = __fadd_rn(rh, t); rl = __fadd_rn(rl, fmaf(a.y, b.y, -t));
        t = __fsub_rn(fmaf(a.x, b.y, M), M);
        ih = __fadd_rn(ih, t); il = __fadd_rn(il, fmaf(a.x, b.y, -t));
        t = __fsub_rn(fmaf(-a.y, b.x, M), M);
        ih = __fadd_rn(ih, t); il = __fadd_rn(il, fmaf(-a.y, b.x, -t));
    }
    cff r;
    two_sum(rh, rl, r.re.hi, r.re.lo);
    two_sum(ih, il, r.im.hi, r.im.lo);
    return r;
}

__device__ inline ff ff_recip(ff x) {
    const float r = __frcp_rn(x.hi);
    const float e = __fsub_rn(fmaf(-x.hi, r, 1.0f), __fmul_rn(x.lo, r));   // 1 - x r
    ff o;
    fast_two_sum(r, __fmul_rn(r, e), o.hi, o.lo);
    return o;
}

// One trailing entry (i, c) of the factorisation, held as an exact multiple of a
// per-entry grid (h) plus an FP32 remainder (l).  With 2^E >= 4 sqrt(A_ii A_cc),
// every partial Schur complement and every product l_ik conj(l_ck) is below 2^(E-2)
// in modulus (Cauchy-Schwarz for the positive definite A), so fmaf(x, y, M) - M
// (M = 1.5 * 2^E) rounds a product onto the multiples of 2^(E-23), the grid parts
// subtract exactly, and the remainders (exact to 2^(E-48) by FMA) collect in l.
// The row factor enters in float-float, the column factor rounded to FP32: the log
// determinant then stays within ~1e-5 of exact on 64 near-collinear columns.
struct gent { float hr, lr, hi, li, M; };
__device__ inline gent gent_make(const cff& a, float bound) {
    int e;
    frexpf(4.0f * bound, &e);   // 2^e > 4 bound
    gent g;
    g.M = ldexpf(1.5f, e);
    g.hr = __fsub_rn(__fadd_rn(a.re.hi, g.M), g.M);
    g.lr = __fadd_rn(__fsub_rn(a.re.hi, g.hr), a.re.lo);
    g.hi = __fsub_rn(__fadd_rn(a.im.hi, g.M), g.M);
    g.li = __fadd_rn(__fsub_rn(a.im.hi, g.hi), a.im.lo);
    return g;
}
__device__ inline void grid_sub(float& h, float& l, ff x, float y, float M) {   // h + l -= x y
    const float ph = __fsub_rn(fmaf(x.hi, y, M), M);
    h = __fsub_rn(h, ph);
    l = __fsub_rn(l, fmaf(x.lo, y, fmaf(x.hi, y, -ph)));
}
__device__ inline void gent_sub_mulc(gent& g, const cff& x, float2 a) {   // A_ic -= x conj(a)
    grid_sub(g.hr, g.lr, x.re, a.x, g.M);
    grid_sub(g.hr, g.lr, x.im, a.y, g.M);
    grid_sub(g.hi, g.li, x.im, a.x, g.M);
    grid_sub(g.hi, g.li, ff_neg(x.re), a.y, g.M);
}
__device__ inline cff gent_value(const gent& g) {
    cff v;
    two_sum(g.hr, g.lr, v.re.hi, v.re.lo);
    two_sum(g.hi, g.li, v.im.hi, v.im.lo);
    return v;
}

// shared memory of k_iota_blk (bytes): colbuf [2][64] cff, colh [2][64] float2, pivbuf [2][2] ff, red [16]
// double, A packed lower [S(S+1)/2] cff, then float2 z [Nz], factors [S][nfac | 1], cm [S], g [S], L packed [S(S+1)/2]
// (also the partial sums g [S][Nf] before the Gram), then float amplitude [S],
// A d [S], d [S], 1/L_kk [64], pivots [64] ff
__host__ __device__ inline size_t iota_blk_lsize(int S, int Nf) {
    const size_t a = (size_t)S * (S + 1) / 2, b = (size_t)S * Nf;
    return a > b ? a : b;
}
__host__ __device__ inline size_t iota_blk_smem(int S, int nfac, int Nf, int Nz) {
    return 2 * IB_SMAX * 16 + 2 * IB_SMAX * 8 + 4 * 8 + 16 * 8 + (size_t)S * (S + 1) / 2 * 16 +
           ((size_t)Nz + (size_t)S * (nfac | 1) + 2 * (size_t)S + iota_blk_lsize(S, Nf)) * 8 + 3 * (size_t)S * 4 + IB_SMAX * 4 +
           IB_SMAX * 8 +
           // residual: alignment slack, cis table [256] (float4), low parts of the factors [S][nfac | 1]
           16 + 256 * 16 + (size_t)S * (nfac | 1) * 8;
}

// blocks per SM: two 256-thread blocks at 128 registers (67 KB shared each).  Three
// (capped at 80 registers, 112 B spilled) measured 127 ms against 120 ms at 64 x 100k:
// the extra warps against the per-pivot barriers do not pay for the spills
constexpr int IOTA_BLK_PER_SM = 2;

template <int NCG>
__global__ void __launch_bounds__(32 * NCG, IOTA_BLK_PER_SM) k_iota_blk(DevGeom G, DevParams Pm, DevState D, int S, const float* z, int all) {
    constexpr int IB_T = 32 * NCG;
    constexpr int QA = 32 / NCG, QB = 64 / NCG;   // register slots of rows ra (< 32) and rb (>= 32)
    extern __shared__ float4 smb[];
    cff* colbuf = reinterpret_cast<cff*>(smb);                    // [2][IB_SMAX] published column (row side)
    float2* colh = reinterpret_cast<float2*>(colbuf + 2 * IB_SMAX);   // [2][IB_SMAX] same, rounded (column side)
    ff* pivbuf = reinterpret_cast<ff*>(colh + 2 * IB_SMAX);       // [2][piv, 1/piv]
    double* red = reinterpret_cast<double*>(pivbuf + 4);          // [16]: yy, then per-warp |r|^2 at 8 + warp
    const int P = Pm.P, J = G.J, Nz = G.Nz, Nm = G.My * G.Mz, Nf = G.Nf;
    const int nfac = (Nf + G.My + G.Mz) | 1;   // factor row stride, odd in float2 against bank conflicts
    cff* Apk = reinterpret_cast<cff*>(red + 16);                   // [S(S+1)/2] float-float A
    float2* zs = reinterpret_cast<float2*>(Apk + (size_t)S * (S + 1) / 2);   // [Nz]
    float2* fac = zs + Nz;                                        // [S][nfac]: b', a_y, a_z
    float2* cmS = fac + (size_t)S * nfac;                         // [S] pi mu, then A (pi mu + d y)
    float2* gS = cmS + S;                                         // [S] g, rhs, solution
    float2* Lsm = gS + S;                                         // FP32 G, then L (packed lower)
    float2* gpart = Lsm;                                          // [S][Nf] (before the Gram)
    float* amp = reinterpret_cast<float*>(Lsm + iota_blk_lsize(S, Nf));     // [S]
    float* adS = amp + S;                                         // [S] A d
    float* dS = adS + S;                                          // [S] d
    float* ild = dS + S;                                          // [IB_SMAX] 1 / L_kk
    ff* pivs = reinterpret_cast<ff*>(ild + IB_SMAX);              // [IB_SMAX] pivots
    // [256] e^{i 2 pi n / 256} (hi, lo), on a 16-byte boundary (the float arrays above end on 4)
    float4* ctab = reinterpret_cast<float4*>((reinterpret_cast<uintptr_t>(pivs + IB_SMAX) + 15) & ~(uintptr_t)15);
    float2* flo = reinterpret_cast<float2*>(ctab + 256);          // [S][nfac] low parts of the factors
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int cg = lane % NCG;
    const int rp = wid * (32 / NCG) + lane / NCG;
    const int ra = rp, rb = IB_SMAX - 1 - rp;
    const float* phi = D.phi[D.cur];
    __shared__ double lg_eb[J_MAX], inv_eb[J_MAX];
    if (tid < J) { lg_eb[tid] = log(D.eta_bar[tid]); inv_eb[tid] = 1.0 / D.eta_bar[tid]; }
    cis_table_fill(ctab, tid, IB_T);
    const int count = all ? P : D.flags[0];
    for (int w = blockIdx.x; w < count; w += gridDim.x) {
        const int pp = all ? w : D.flags[1 + w];
        double total = 0.0;
        for (int j = 0; j < J; ++j) {
            __syncthreads();
            for (int k = tid; k < Nz; k += IB_T) zs[k] = make_float2(z[2 * (j * Nz + k)], z[2 * (j * Nz + k) + 1]);
            const double eb = D.eta_bar[j];
            const float ebf = (float)eb;
            const ff ebff = ff{ebf, (float)(eb - (double)ebf)};
            for (int s = tid; s < S; s += IB_T) {
                const float* ph = phi + (size_t)s * 6 * P;
                float2* fs = fac + (size_t)s * nfac;
                const size_t gi = ((size_t)s * J + j) * P + pp;
                const float A = factors_from_geo_pairs(G, ctab, D.geo[gi], D.geo_lo[gi], fs, flo + (size_t)s * nfac);
                const float pi = (float)(D.zeta[s * J + j] * D.W[s]);
                const float gm = ph[3 * P + pp], mr = ph[4 * P + pp], mi = ph[5 * P + pp];
                const float d = sqrtf(fmaxf(pi * (gm + (mr * mr + mi * mi) * (1.0f - pi)), 0.0f));
                amp[s] = A;
                dS[s] = d;
                adS[s] = A * d;
                cmS[s] = make_float2(pi * mr, pi * mi);
            }
            __syncthreads();
            // g_s = psi_s^H z: tasks (s, f) contract over the antennas
            for (int t = tid; t < S * Nf; t += IB_T) {
                const int f = t / S, s = t - f * S;   // lanes over s: z_f broadcast
                const float2* fs = fac + (size_t)s * nfac;
                float2 accy = make_float2(0.f, 0.f);
                for (int y = 0; y < G.My; ++y) {
                    float2 accm = make_float2(0.f, 0.f);
                    for (int m = 0; m < G.Mz; ++m) {
                        const float2 u = cmulc(fs[Nf + G.My + m], zs[f * Nm + y * G.Mz + m]);
                        accm.x += u.x; accm.y += u.y;
                    }
                    const float2 u = cmulc(fs[Nf + y], accm);
                    accy.x += u.x; accy.y += u.y;
                }
                gpart[s * Nf + f] = cmulc(fs[f], accy);
            }
            __syncthreads();
            for (int s = tid; s < S; s += IB_T) {
                float2 acc = make_float2(0.f, 0.f);
                for (int f = 0; f < Nf; ++f) { acc.x += gpart[s * Nf + f].x; acc.y += gpart[s * Nf + f].y; }
                gS[s] = make_float2(amp[s] * acc.x, amp[s] * acc.y);
            }
            __syncthreads();
            // Gram, one packed entry per task (a >= b), into shared memory
            for (int t = tid; t < S * (S + 1) / 2; t += IB_T) {
                int a, b;
                tri_ab(t, a, b);
                const float2* fa = fac + (size_t)a * nfac;
                const float2* fb = fac + (size_t)b * nfac;
                const cff sf = fx_dotc(fa, fb, Nf);
                const cff sy = fx_dotc(fa + Nf, fb + Nf, G.My);
                const cff sz = fx_dotc(fa + Nf + G.My, fb + Nf + G.My, G.Mz);
                const cff gu = cff_mul(sf, cff_mul(sy, sz));
                const float aa = amp[a] * amp[b];
                Lsm[t] = make_float2(aa * (gu.re.hi + gu.re.lo), aa * (gu.im.hi + gu.im.lo));
                const ff sc = ff_prod(adS[a], adS[b]);
                cff v{ff_mul(gu.re, sc), ff_mul(gu.im, sc)};
                if (a == b) { v.re = ff_add(v.re, ebff); v.im = ff{0.f, 0.f}; }
                Apk[t] = v;
                if (b == 0) { colbuf[a] = v; colh[a] = make_float2(v.re.hi, v.im.hi); }
                if (t == 0) { pivbuf[0] = v.re; pivbuf[1] = ff_recip(v.re); }
            }
            __syncthreads();
            // this thread's slots (rows ra: q < 8, rb: q < 16) into registers
            gent Ar[QA], Br[QB];
            unsigned liveA = 0u, liveB = 0u;   // slots of the lower triangle; cleared as columns finish
            {
                const float sa = (ra < S) ? sqrtf(Apk[tri(ra, ra)].re.hi) : 0.f;
                const float sb = (rb < S) ? sqrtf(Apk[tri(rb, rb)].re.hi) : 0.f;
                #pragma unroll
                for (int q = 0; q < QA; ++q) {
                    const int c = NCG * q + cg;
                    if (c <= ra && ra < S) { Ar[q] = gent_make(Apk[tri(ra, c)], sa * sqrtf(Apk[tri(c, c)].re.hi)); liveA |= 1u << q; }
                }
                #pragma unroll
                for (int q = 0; q < QB; ++q) {
                    const int c = NCG * q + cg;
                    if (c <= rb && rb < S) { Br[q] = gent_make(Apk[tri(rb, c)], sb * sqrtf(Apk[tri(c, c)].re.hi)); liveB |= 1u << q; }
                }
            }
            // rhs_a = d_a (g_a - sum_b G_ab pi_b mu_b), FP32
            float2 rhs = make_float2(0.f, 0.f);
            const int fst = tid - 64;   // forward-substitution row of this thread (warps 2-3)
            if (fst >= 0 && fst < S) {
                const int a = fst;
                float2 acc = gS[a];
                for (int b = 0; b < S; ++b) {
                    const float2 e = (b <= a) ? Lsm[tri(a, b)] : make_float2(Lsm[tri(b, a)].x, -Lsm[tri(b, a)].y);
                    const float2 u = cmul(e, cmS[b]);
                    acc.x -= u.x; acc.y -= u.y;
                }
                rhs = make_float2(dS[a] * acc.x, dS[a] * acc.y);
            }
            __syncthreads();
            // Cholesky with exactly accumulated trailing entries; log det from the
            // float-float product of the pivots (exponent kept apart)
            for (int k = 0; k < S; ++k) {
                const int cur = k & 1, nxt = cur ^ 1;
                const cff* col = colbuf + cur * IB_SMAX;
                const float2* colr = colh + cur * IB_SMAX;
                cff* ncol = colbuf + nxt * IB_SMAX;
                float2* ncolr = colh + nxt * IB_SMAX;
                ff piv = pivbuf[2 * cur];
                ff inv = pivbuf[2 * cur + 1];
                if (!(piv.hi > 0.f)) { piv = ff{1e-30f, 0.f}; inv = ff{1e30f, 0.f}; }
                // FP32 factor for the (variational) solves: 1/L_kk by the fast reciprocal square root
                const float il = rsqrtf(piv.hi + piv.lo);
                const float lkk = (piv.hi + piv.lo) * il;
                // column c = NCG q + cg takes updates while c > k: the slot of column k retires
                const int kc = k - cg;
                if (kc >= 0 && kc % NCG == 0) { liveA &= ~(1u << (kc / NCG)); liveB &= ~(1u << (kc / NCG)); }
                if (tid == 0) {
                    pivs[k] = piv;
                    Lsm[tri(k, k)] = make_float2(lkk, 0.f);
                    ild[k] = il;
                }
                // forward substitution L u = rhs, one column behind the factorisation:
                // row i takes column k-1 (published last step), then row k yields u_k
                if (fst >= k && fst < S) {
                    if (k > 0) {
                        const float2 u = cmul(Lsm[tri(fst, k - 1)], gS[k - 1]);
                        rhs.x -= u.x; rhs.y -= u.y;
                    }
                    if (fst == k) gS[k] = make_float2(rhs.x * il, rhs.y * il);
                }
                {   // FP32 column k of L for the solves (warps 4-5)
                    const int i = k + 1 + (tid - 128);
                    if (tid >= 128 && i < S) {
                        const cff v = col[i];
                        Lsm[tri(i, k)] = make_float2((v.re.hi + v.re.lo) * il, (v.im.hi + v.im.lo) * il);
                    }
                }
                cff la{}, lb{};
                if (ra > k && ra < S) { const cff v = col[ra]; la = cff{ff_mul(v.re, inv), ff_mul(v.im, inv)}; }
                if (rb > k && rb < S) { const cff v = col[rb]; lb = cff{ff_mul(v.re, inv), ff_mul(v.im, inv)}; }
                #pragma unroll
                for (int q = 0; q < QA; ++q) {
                    const int c = NCG * q + cg;
                    if (liveA & (1u << q)) {
                        gent_sub_mulc(Ar[q], la, colr[c]);
                        if (NCG * q == kc + 1) {
                            const cff v = gent_value(Ar[q]);
                            ncol[ra] = v;
                            ncolr[ra] = make_float2(v.re.hi, v.im.hi);
                            if (ra == c) { pivbuf[2 * nxt] = v.re; pivbuf[2 * nxt + 1] = ff_recip(v.re); }
                        }
                    }
                }
                #pragma unroll
                for (int q = 0; q < QB; ++q) {
                    const int c = NCG * q + cg;
                    if (liveB & (1u << q)) {
                        gent_sub_mulc(Br[q], lb, colr[c]);
                        if (NCG * q == kc + 1) {
                            const cff v = gent_value(Br[q]);
                            ncol[rb] = v;
                            ncolr[rb] = make_float2(v.re.hi, v.im.hi);
                            if (rb == c) { pivbuf[2 * nxt] = v.re; pivbuf[2 * nxt + 1] = ff_recip(v.re); }
                        }
                    }
                }
                __syncthreads();
            }
            // back substitution L^H y = u (warp 0; lane owns rows lane and lane + 32); log det
            // from the float-float product of the pivots (exponents apart)
            if (wid == 0) {
                ffexp det{ff{1.f, 0.f}, 0};
                for (int k = lane; k < S; k += 32) ffexp_mul(det, pivs[k]);
                #pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const ff om{__shfl_xor_sync(0xffffffffu, det.m.hi, o), __shfl_xor_sync(0xffffffffu, det.m.lo, o)};
                    const int oe = __shfl_xor_sync(0xffffffffu, det.e, o);
                    ffexp_mul(det, om);
                    det.e += oe;
                }
                if (lane == 0) red[1] = ffexp_log(det);
                float2 r0 = (lane < S) ? gS[lane] : make_float2(0.f, 0.f);
                float2 r1 = (lane + 32 < S) ? gS[lane + 32] : make_float2(0.f, 0.f);
                const float i0 = (lane < S) ? ild[lane] : 0.f, i1 = (lane + 32 < S) ? ild[lane + 32] : 0.f;
                for (int k = S - 1; k >= 0; --k) {
                    const float2 lr0 = (lane < k) ? Lsm[tri(k, lane)] : make_float2(0.f, 0.f);
                    const float2 lr1 = (lane + 32 < k) ? Lsm[tri(k, lane + 32)] : make_float2(0.f, 0.f);
                    const bool hi_row = k >= 32;
                    const float2 own = hi_row ? r1 : r0;
                    const float io = hi_row ? i1 : i0;
                    const float2 yk = make_float2(__shfl_sync(0xffffffffu, own.x * io, k & 31),
                                                  __shfl_sync(0xffffffffu, own.y * io, k & 31));
                    if (lane == (k & 31)) { if (hi_row) r1 = yk; else r0 = yk; }
                    if (lane < k) { const float2 u = cmulc(lr0, yk); r0.x -= u.x; r0.y -= u.y; }
                    if (lane + 32 < k) { const float2 u = cmulc(lr1, yk); r1.x -= u.x; r1.y -= u.y; }
                }
                ff yy{0.f, 0.f};
                if (lane < S) {
                    ff_acc_sq(yy, r0);
                    const float2 c = cmS[lane];
                    cmS[lane] = make_float2(amp[lane] * (c.x + dS[lane] * r0.x), amp[lane] * (c.y + dS[lane] * r0.y));
                }
                if (lane + 32 < S) {
                    ff_acc_sq(yy, r1);
                    const float2 c = cmS[lane + 32];
                    cmS[lane + 32] = make_float2(amp[lane + 32] * (c.x + dS[lane + 32] * r1.x),
                                                 amp[lane + 32] * (c.y + dS[lane + 32] * r1.y));
                }
                yy = warp_sum_ff(yy);
                if (lane == 0) red[0] = ff_to_d(yy);
            }
            __syncthreads();
            // residual r = z - sum_s w_s (b' kron a_y kron a_z)_s, w_s = A_s (pi mu + d y)_s.  Its
            // energy reaches ~1e4 noise units, so the steering values enter as (hi, lo) pairs
            // (~1e-10), the products of the high parts are summed exactly on a grid fixed for
            // this (p, j) (2^E > 4 (max_k |z_k| + sum_s |w_s|) bounds every partial sum), and
            // the remainders and the low-part cross terms are summed in FP32
            if (wid == 1) {
                float b = 0.f, zm = 0.f;
                for (int s = lane; s < S; s += 32) b += fabsf(cmS[s].x) + fabsf(cmS[s].y);
                for (int k = lane; k < Nz; k += 32) zm = fmaxf(zm, fabsf(zs[k].x) + fabsf(zs[k].y));
                b = warp_sum_f(b);
                #pragma unroll
                for (int o = 16; o > 0; o >>= 1) zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
                if (lane == 0) red[2] = (double)(b + zm);
            }
            __syncthreads();
            int gE;
            frexpf(4.0f * (float)red[2] + 1e-30f, &gE);
            const float GM = ldexpf(1.5f, gE);
            ff rr{0.f, 0.f};
            for (int k = tid; k < Nz; k += IB_T) {
                const int f = k / Nm, ym = k - f * Nm, y = ym / G.Mz, m = ym - y * G.Mz;
                const float2 zk = zs[k];
                float2 gr, rm;
                gr.x = __fsub_rn(__fadd_rn(zk.x, GM), GM);
                gr.y = __fsub_rn(__fadd_rn(zk.y, GM), GM);
                rm.x = __fsub_rn(zk.x, gr.x);
                rm.y = __fsub_rn(zk.y, gr.y);
                for (int s = 0; s < S; ++s) {
                    // w_s (FP32, exact) times psi'_sk = b'_f a_y a_z as a (hi, lo) pair
                    const float2* fs = fac + (size_t)s * nfac;
                    const float2* fl = flo + (size_t)s * nfac;
                    const float4 ay = cpair_mul(fs[Nf + y], fl[Nf + y], fs[Nf + G.My + m], fl[Nf + G.My + m]);
                    const float4 c = cpair_mul(fs[f], fl[f], make_float2(ay.x, ay.y), make_float2(ay.z, ay.w));
                    const float2 u = cmS[s];
                    float t;
                    t = __fsub_rn(fmaf(u.x, c.x, GM), GM); gr.x = __fsub_rn(gr.x, t); rm.x -= fmaf(u.x, c.x, -t);
                    t = __fsub_rn(fmaf(-u.y, c.y, GM), GM); gr.x = __fsub_rn(gr.x, t); rm.x -= fmaf(-u.y, c.y, -t);
                    t = __fsub_rn(fmaf(u.x, c.y, GM), GM); gr.y = __fsub_rn(gr.y, t); rm.y -= fmaf(u.x, c.y, -t);
                    t = __fsub_rn(fmaf(u.y, c.x, GM), GM); gr.y = __fsub_rn(gr.y, t); rm.y -= fmaf(u.y, c.x, -t);
                    rm.x -= fmaf(u.x, c.z, -u.y * c.w);
                    rm.y -= fmaf(u.x, c.w, u.y * c.z);
                }
                float hx, lx, hy, ly;
                two_sum(gr.x, rm.x, hx, lx);
                two_sum(gr.y, rm.y, hy, ly);
                ff_acc_sq(rr, make_float2(hx, hy));
                rr.lo = fmaf(2.0f * hx, lx, fmaf(2.0f * hy, ly, rr.lo));
            }
            rr = warp_sum_ff(rr);
            if (lane == 0) red[8 + wid] = ff_to_d(rr);
            __syncthreads();
            if (tid == 0) {
                double rrs = 0.0;
                for (int w2 = 0; w2 < IB_T / 32; ++w2) rrs += red[8 + w2];
                const double lg = lg_eb[j];
                total += -(rrs * inv_eb[j] + red[0]) - (red[1] - S * lg) - Nz * (LOG_PI + lg);
            }
        }
        if (tid == 0) D.lw_x[pp] = total;
    }
}

// ---------------------------------------------------------------- nu (thread per (j, p), FP64)
// 1/d of a positive normal number: the hardware's ~20-bit reciprocal and two Newton steps
__device__ __forceinline__ double nu_rcp(double d) {
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(d));
    r = fma(fma(-d, r, 1.0), r, r);
    return fma(fma(-d, r, 1.0), r, r);
}
// LDL^T of the tridiagonal eta I + T: bound by the FP64 pipe, so one reciprocal per row serves the
// quadratic form and the next row's multiplier (64 PFs x 4 PAs x 1e5: 0.91 ms, two divisions 1.44).
__global__ void k_nu(DevGeom G, DevParams Pm, DevState D, int S) {
    const int P = Pm.P, SM = Pm.S_max;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= G.J * P) return;
    const int j = idx / P, p = idx - j * P;
    const double eta = (double)D.eta[D.cur][(size_t)j * P + p];
    const double* T = D.nu_T + (size_t)j * 4 * SM;
    double rprev = 0.0, logdet = 0.0, quad = 0.0;
    double ur = 0.0, ui = 0.0;
    double scale = 1.0;
    for (int k = 0; k < S; ++k) {
        double dk = eta + T[k];
        double br = T[2 * SM + 2 * k], bi = T[2 * SM + 2 * k + 1];
        if (k > 0) {
            const double o = T[SM + k - 1];
            const double l = o * rprev;
            dk -= o * l;
            br -= l * ur; bi -= l * ui;
        }
        const double r = nu_rcp(dk);
        quad += (br * br + bi * bi) * r;
        scale *= dk;
        if (scale > 1e200 || scale < 1e-200) { logdet += log(scale); scale = 1.0; }
        rprev = r; ur = br; ui = bi;
    }
    logdet += log(scale);
    const double e2 = D.nu_c[2 * j];
    const double lnu = -(e2 - quad) / eta - (G.Nz - S) * log(eta) - logdet - G.Nz * log(M_PI);
    D.lw_eta[(size_t)j * P + p] = lnu;
}

// S below which every particle is evaluated in float-float (symmetric layouts), or in FP32 with only
// the ill-conditioned ones redone; from it on the FP32 bulk kernels and the selection by error bounds
constexpr int IOTA_FF_ALL_S = 24;

int launch_iota(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, cudaStream_t st) {
    if (S >= IOTA_FF_ALL_S) return launch_iota_bulk(G, Pm, D, S, z, st);
    if (iota_sym_ok(G, S)) {   // float-float for every particle; nothing is left to repair
        launch_iota_ff(G, Pm, D, S, z, true, st);
        return 1;
    }
    const int nfac = G.Nf + G.My + G.Mz;
    const size_t per_warp = iota32_warp_f2(S, nfac, G.Nf) * sizeof(float2);
    int wpb = 8;
    while (wpb > 1 && (size_t)G.Nz * sizeof(float2) + wpb * per_warp > 64 * 1024) wpb /= 2;
    const size_t smem = (size_t)G.Nz * sizeof(float2) + wpb * per_warp;
    cudaMemsetAsync(D.flags, 0, sizeof(int), st);
    smem_allow_max((const void*)k_iota);
    k_iota<<<(Pm.P + wpb - 1) / wpb, 32 * wpb, smem, st>>>(G, Pm, D, S, z);
    return 1;
}

int launch_iota_repair(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, cudaStream_t st) {
    if (iota_sym_ok(G, S)) {
        if (S < IOTA_FF_ALL_S) return 0;
        launch_iota_ff(G, Pm, D, S, z, false, st);
        return 1;
    }
    const int nfac = G.Nf + G.My + G.Mz;
    const size_t smem = iota_blk_smem(S, nfac, G.Nf, G.Nz);
    constexpr int NCG = IOTA_BLK_NCG;
    smem_allow_max((const void*)k_iota_blk<NCG>);
    int sms = 0, dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int wave = IOTA_BLK_PER_SM * std::max(sms, 1);
    k_iota_blk<NCG><<<wave, 32 * NCG, smem, st>>>(G, Pm, D, S, z, 0);
    return 1;
}

void launch_nu(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, cudaStream_t st) {
    const int n = G.J * Pm.P;
    k_nu<<<(n + 255) / 256, 256, 0, st>>>(G, Pm, D, S);
}

}  // namespace bp

namespace bp {
size_t iota_blk_smem_bytes(const DevGeom& G, int S) {
    return iota_blk_smem(S, G.Nf + G.My + G.Mz, G.Nf, G.Nz);
}
}  // namespace bp
