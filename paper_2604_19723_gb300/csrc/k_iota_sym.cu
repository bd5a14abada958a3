// MT likelihood iota~ (Supplementary Sec. S-V) on layouts whose frequencies and element positions
// are symmetric about 0 (DevGeom::sym): a real problem in half the elements.
//
// Without its carrier c_s = e^{-i 2 pi d_s / lambda} a unit-modulus steering vector satisfies
// u_{Nz-1-k} = conj(u_k).  Hence
//   * the Gram u_a^H u_b = sum_{k < Nz/2} 2 (x_a x_b + y_a y_b) (u = x + i y) is real, and by the
//     Kronecker structure the product of three short real sums;
//   * the covariance eta_bar I + sum_s d_s^2 psi_s psi_s^H does not see the carriers, so log det and
//     the solves take the real symmetric A = eta_bar I + (dA)_a (dA)_b u_a^H u_b;
//   * with P_k = z_k + z_k', Q_k = z_k - z_k' (k' = Nz - 1 - k) a sum of steering vectors with complex
//     coefficients w is P_k = sum_s 2 w_s x_sk, Q_k = sum_s 2 i w_s y_sk, and
//     u_s^H z = sum_{k < Nz/2} x_sk P_k - i y_sk Q_k  (the middle element of odd Nz counts once).
// The elimination, the Gram and the element work are 2 to 4 times smaller than in the general
// complex form (k_like.cu, k_iota_bulk.cu), which other layouts take.
#include "bp_internal.cuh"
#include "bp_kernels.cuh"

namespace bp {

constexpr double IS_LOG_PI = 1.14472988584940017414;

struct IsDims { int Nh, Fh, hy, hz, hf, Nmh; };   // half counts: elements, frequencies, a_y, a_z, factors, a_y a_z
__host__ __device__ inline IsDims is_dims(const DevGeom& G) {
    IsDims d;
    d.Nh = (G.Nz + 1) / 2;
    d.Fh = (G.Nf + 1) / 2;
    d.hy = (G.My + 1) / 2;
    d.hz = (G.Mz + 1) / 2;
    d.hf = d.Fh + d.hy + d.hz;
    d.Nmh = (G.My * G.Mz + 1) / 2;
    return d;
}
__device__ __forceinline__ int is_tri(int i, int j) { return i * (i + 1) / 2 + j; }
__device__ __forceinline__ void is_tri_ab(int t, int& a, int& b) {
    a = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((a + 1) * (a + 2) / 2 <= t) ++a;
    while (a * (a + 1) / 2 > t) --a;
    b = t - a * (a + 1) / 2;
}
__device__ __forceinline__ float4 conj_if(float4 a, bool c) { return c ? make_float4(a.x, -a.y, a.z, -a.w) : a; }
// element (y, m) of the half table of a_y a_z: index ym below the middle, else the mirrored one's conjugate
__device__ __forceinline__ int is_half(int i, int n, int h, bool& c) { c = i >= h; return c ? n - 1 - i : i; }

// ---------------------------------------------------------------- float-float evaluation
// A team of TW warps per (particle, PA), the PAs of a particle in one block.  log det from a Cholesky
// factorisation of A in float-float (pivots of nearly coinciding columns keep ~1e-13), the quadratic
// form in its variational form |r|^2/eta_bar + |y|^2 at an FP32 minimiser y, the residual r from
// steering elements as (hi, lo) pairs (~1e-9) with the products of the high parts summed exactly on
// a grid fixed per (p, j).  Below 24 PFs every particle is evaluated (the FP32 warp kernel and the
// block-per-particle repair of the particles it flagged took 8.7 ms at 10 PFs x 30000 particles,
// Nz = 160; this takes 1.25 ms); from 24 PFs on the particles k_iota_select queues, with four warps
// per team, since few working sets of that size fit an SM.
// Bound: FP32 issue, the residual's ~50 instructions per (s, half element).
constexpr int IF_WMAX = 16;
constexpr float IF_RATIO_MAX = 100.0f;   // reported as ill-conditioned: sqrt(sum (A_kk / piv_k)^2) above this
struct IfPlan { size_t fac, ct, K, L, vec, z, warp; };
__host__ __device__ inline IfPlan if_plan(const DevGeom& G, int S) {
    const IsDims d = is_dims(G);
    IfPlan p{};
    size_t o = 0;
    p.fac = o; o += (size_t)S * d.hf * sizeof(float4);
    p.ct = o; o += (size_t)S * d.Nmh * sizeof(float4);
    p.z = o; o += (size_t)d.Nh * 2 * sizeof(float4);            // P (hi, lo), Q (hi, lo)
    p.K = o; o += (size_t)S * (S + 1) / 2 * sizeof(ff);
    p.vec = o; o += (size_t)S * (2 * sizeof(float2) + sizeof(ff) + 2 * sizeof(float));   // w, g | pivots | dA, 1/L_kk
    p.L = o; o += (size_t)S * (S + 1) / 2 * sizeof(float);
    p.warp = (o + 15) & ~(size_t)15;
    return p;
}
constexpr int IF_TEAM_MAX = 4;           // warps of a team
constexpr size_t IF_FIXED = 256 * sizeof(float4) + IF_WMAX * (3 * sizeof(double) + sizeof(float)) +
                            IF_WMAX * IF_TEAM_MAX * sizeof(ff) + IF_WMAX * sizeof(float);

// sum_i x_i.x y_i.x + x_i.y y_i.y of unit-modulus pairs: the high parts' products split on a grid of
// 2^-16 (their sums below 256 exact), remainders and cross terms in FP32
__device__ __forceinline__ ff if_dot(const float4* x, const float4* y, int n) {
    const float M = 192.0f;
    float h = 0.f, l = 0.f;
    for (int i = 0; i < n; ++i) {
        const float4 a = x[i], b = y[i];
        float t = __fsub_rn(fmaf(a.x, b.x, M), M);
        h = __fadd_rn(h, t);
        l += fmaf(a.x, b.z, fmaf(a.z, b.x, fmaf(a.x, b.x, -t)));
        t = __fsub_rn(fmaf(a.y, b.y, M), M);
        h = __fadd_rn(h, t);
        l += fmaf(a.y, b.w, fmaf(a.w, b.y, fmaf(a.y, b.y, -t)));
    }
    ff r;
    two_sum(h, l, r.hi, r.lo);
    return r;
}
// 2 sum over the proper half plus the middle (exactly 1) of an odd count
__device__ __forceinline__ ff if_sum(const float4* x, const float4* y, int n) {
    ff r = if_dot(x, y, n / 2);
    r = ff{2.0f * r.hi, 2.0f * r.lo};
    return (n & 1) ? ff_add(r, ff{1.0f, 0.f}) : r;
}

template <int TW>
__global__ void __launch_bounds__(TW == 1 ? 256 : 512, TW == 1 ? 3 : 1) k_iota_ff(DevGeom G, DevParams Pm, DevState D, int S, const float* __restrict__ z, int all, int W) {
    extern __shared__ float4 smf[];
    const int P = Pm.P, J = G.J, Nz = G.Nz, Nf = G.Nf, My = G.My, Mz = G.Mz, Nm = My * Mz;
    const IsDims dm = is_dims(G);
    constexpr int TT = 32 * TW;
    const int lane = threadIdx.x & 31, wid = threadIdx.x / TT, tt = threadIdx.x - wid * TT, wt = tt >> 5;   // team, place in it
    auto team_sync = [&]() {
        if constexpr (TW == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" :: "r"(1 + wid), "n"(TT) : "memory");
    };
    float4* ctab = smf;                                         // [256]
    double* part = reinterpret_cast<double*>(ctab + 256);       // [J] log iota per PA
    double* lgs = part + IF_WMAX;                               // [J] log eta_bar
    double* ies = lgs + IF_WMAX;                                // [J] 1 / eta_bar
    float* rat = reinterpret_cast<float*>(ies + IF_WMAX);       // [J] sum of squared pivot ratios
    ff* red = reinterpret_cast<ff*>(rat + IF_WMAX) + wid * TW;  // [TW] |r|^2 of the team's warps
    float* gmS = reinterpret_cast<float*>(reinterpret_cast<ff*>(rat + IF_WMAX) + IF_WMAX * IF_TEAM_MAX) + wid;   // residual grid
    const IfPlan pl = if_plan(G, S);
    char* base = reinterpret_cast<char*>(smf) + ((IF_FIXED + 15) & ~(size_t)15) + (size_t)wid * pl.warp;
    float4* fac = reinterpret_cast<float4*>(base + pl.fac);     // [S][hf] b_f, a_y, a_z (half of each)
    float4* ct = reinterpret_cast<float4*>(base + pl.ct);       // [S][Nmh] a_y a_z
    float4* zp = reinterpret_cast<float4*>(base + pl.z);        // [Nh] P, then [Nh] Q, as (hi, lo)
    float4* zq = zp + dm.Nh;
    ff* K = reinterpret_cast<ff*>(base + pl.K);                 // packed lower: A, then its elimination
    float2* ws = reinterpret_cast<float2*>(base + pl.vec);      // [S] A c pi mu, then w
    float2* gs = ws + S;                                        // [S] u^H z
    ff* piv = reinterpret_cast<ff*>(gs + S);                    // [S]
    float* dA = reinterpret_cast<float*>(piv + S);              // [S] d_s A_s
    float* ild = dA + S;                                        // [S] 1 / L_kk
    float* L = reinterpret_cast<float*>(base + pl.L);           // packed lower: the FP32 Gram, then the FP32 factor
    for (int i = threadIdx.x; i < 256; i += blockDim.x) ctab[i] = D.ctab[i];
    if (threadIdx.x < J) {
        lgs[threadIdx.x] = log(D.eta_bar[threadIdx.x]);
        ies[threadIdx.x] = 1.0 / D.eta_bar[threadIdx.x];
    }
    __syncthreads();
    const float* phi = D.phi[D.cur];
    const int count = all ? P : D.flags[0], npair = S * (S + 1) / 2;
    const bool odd = Nz & 1;
    int zj = -1;
    float zmax = 0.f;
    for (int w = blockIdx.x; w < count; w += gridDim.x) {
        const int p = all ? w : D.flags[1 + w];
        for (int j = wid; j < J; j += W) {
            team_sync();
            if (zj != j) {   // the observation's sums and differences, exactly
                for (int k = tt; k < dm.Nh; k += TT) {
                    const float* a = z + 2 * ((size_t)j * Nz + k);
                    const float* b = z + 2 * ((size_t)j * Nz + Nz - 1 - k);
                    float4 pv = make_float4(a[0], a[1], 0.f, 0.f), qv = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (k != Nz - 1 - k) {
                        two_sum(a[0], b[0], pv.x, pv.z);
                        two_sum(a[1], b[1], pv.y, pv.w);
                        two_sum(a[0], -b[0], qv.x, qv.z);
                        two_sum(a[1], -b[1], qv.y, qv.w);
                    }
                    zp[k] = pv;
                    zq[k] = qv;
                }
                team_sync();
                zmax = 0.f;
                for (int k = lane; k < dm.Nh; k += 32)
                    zmax = fmaxf(zmax, fmaxf(fabsf(zp[k].x) + fabsf(zp[k].y), fabsf(zq[k].x) + fabsf(zq[k].y)));
                #pragma unroll
                for (int o = 16; o > 0; o >>= 1) zmax = fmaxf(zmax, __shfl_xor_sync(0xffffffffu, zmax, o));
                zj = j;
            }
            const double eb = D.eta_bar[j];
            // per-PF scalars, then the factors as pairs
            for (int s = tt; s < S; s += TT) {
                const float* ph = phi + (size_t)s * 6 * P + p;
                const float4 g = D.geo[((size_t)s * J + j) * P + p];
                const float A = G.amp_c / (g.x + g.y);
                float h0, l0;
                ff_frac_mul2(g.x, g.y, G.inv_lam_hi, G.inv_lam_lo, h0, l0);
                float2 c, cl;
                cis_pair(ctab, -h0, -l0, c, cl);
                const float pi = (float)(D.zeta[s * J + j] * D.W[s]);
                const float gm = ph[3 * (size_t)P], mr = ph[4 * (size_t)P], mi = ph[5 * (size_t)P];
                dA[s] = A * sqrtf(fmaxf(pi * (gm + (mr * mr + mi * mi) * (1.0f - pi)), 0.0f));
                ws[s] = cmul(make_float2(A * pi * mr, A * pi * mi), c);
            }
            for (int i = tt; i < S * dm.hf; i += TT) {
                const int s = i / dm.hf, q = i - s * dm.hf;
                const size_t gi = ((size_t)s * J + j) * P + p;
                const float4 g = D.geo[gi];
                float th, tl;
                if (q < dm.Fh) {
                    ff_frac_mul2(g.x, g.y, G.fc_hi[q], G.fc_lo[q], th, tl);
                    th = -th; tl = -tl;
                } else {
                    const float2 gl = D.geo_lo[gi];
                    const bool y = q < dm.Fh + dm.hy;
                    const int e = q - dm.Fh - (y ? 0 : dm.hy);
                    const float c = y ? G.py_l[e] : G.pz_l[e], cl = y ? G.py_lo[e] : G.pz_lo[e];
                    const float u = y ? g.z : g.w, ul = y ? gl.x : gl.y;
                    th = __fmul_rn(c, u);
                    tl = fmaf(c, ul, fmaf(cl, u, fmaf(c, u, -th)));
                }
                float2 hi, lo;
                cis_pair(ctab, th, tl, hi, lo);
                fac[i] = make_float4(hi.x, hi.y, lo.x, lo.y);
            }
            team_sync();
            for (int i = tt; i < S * dm.Nmh; i += TT) {
                const int s = i / dm.Nmh, ym = i - s * dm.Nmh, y = ym / Mz, m = ym - y * Mz;
                const float4* fs = fac + s * dm.hf + dm.Fh;
                bool cy, cz;
                const int iy = is_half(y, My, dm.hy, cy), iz = is_half(m, Mz, dm.hz, cz);
                ct[i] = pair_mul_fx(conj_if(fs[iy], cy), conj_if(fs[dm.hy + iz], cz));
            }
            // Gram and A = eta_bar I + D G D, packed
            for (int t = tt; t < npair; t += TT) {
                int a, b;
                is_tri_ab(t, a, b);
                const float4 *fa = fac + a * dm.hf, *fb = fac + b * dm.hf;
                const ff g = ff_mul(if_sum(fa, fb, Nf), ff_mul(if_sum(fa + dm.Fh, fb + dm.Fh, My),
                                                               if_sum(fa + dm.Fh + dm.hy, fb + dm.Fh + dm.hy, Mz)));
                ff v = ff_mul(g, ff_prod(dA[a], dA[b]));
                if (a == b) v = ff_add(v, ff{(float)eb, (float)(eb - (double)(float)eb)});
                K[t] = v;
                L[t] = g.hi;
            }
            team_sync();
            // g_s = u_s^H z (FP32: the minimiser's rounding enters at second order)
            for (int s = wt; s < S; s += TW) {
                const float4 *fs = fac + s * dm.hf, *cs = ct + s * dm.Nmh;
                float gr = 0.f, gi = 0.f;
                for (int k = lane; k < dm.Nh; k += 32) {
                    const int f = k / Nm, ym = k - f * Nm;
                    bool cj;
                    const int ih = is_half(ym, Nm, dm.Nmh, cj);
                    const float4 b = fs[f], c = conj_if(cs[ih], cj);
                    const float x = fmaf(b.x, c.x, -b.y * c.y), y = fmaf(b.x, c.y, b.y * c.x);
                    const float4 pv = zp[k], qv = zq[k];
                    gr = fmaf(x, pv.x, fmaf(y, qv.y, gr));
                    gi = fmaf(x, pv.y, fmaf(-y, qv.x, gi));
                }
                gr = warp_sum_f(gr);
                gi = warp_sum_f(gi);
                if (lane == 0) gs[s] = make_float2(gr, gi);
            }
            team_sync();
            // right-hand side t_a = (dA)_a (g_a - sum_b G_ab w0_b): rows lane and lane + 32
            float2 r0 = make_float2(0.f, 0.f), r1 = r0;
            for (int half = 0; half < (wt != 0 ? 0 : S > 32 ? 2 : 1); ++half) {   // the team's first warp
                const int a = lane + 32 * half;
                if (a >= S) continue;
                float2 acc = gs[a];
                for (int b = 0; b < S; ++b) {
                    const float g = L[b <= a ? is_tri(a, b) : is_tri(b, a)];
                    acc.x = fmaf(-g, ws[b].x, acc.x);
                    acc.y = fmaf(-g, ws[b].y, acc.y);
                }
                acc = make_float2(dA[a] * acc.x, dA[a] * acc.y);
                if (half) r1 = acc; else r0 = acc;
            }
            team_sync();
            // elimination in float-float, right-looking
            float ratio2 = 0.f;
            for (int k = 0; k < S; ++k) {
                ff pk = K[is_tri(k, k)];
                if (!(pk.hi > 0.f)) pk = ff{1e-30f, 0.f};
                ff inv;
                {
                    const float r = __frcp_rn(pk.hi);
                    const float e = __fsub_rn(fmaf(-pk.hi, r, 1.0f), __fmul_rn(pk.lo, r));
                    fast_two_sum(r, __fmul_rn(r, e), inv.hi, inv.lo);
                }
                const float il = rsqrtf(pk.hi);
                if (tt == 0) {
                    piv[k] = pk;
                    ild[k] = il;
                    const float akk = fmaf(dA[k] * dA[k], L[is_tri(k, k)], (float)eb);   // before the elimination
                    ratio2 = fmaf(akk * inv.hi, akk * inv.hi, ratio2);
                }
                const int n = S - k - 1;
                for (int t = tt; t < n * (n + 1) / 2; t += TT) {
                    int a, c;
                    is_tri_ab(t, a, c);
                    const int i = k + 1 + a, cc = k + 1 + c;
                    const ff x = ff_mul(K[is_tri(i, k)], inv), y = K[is_tri(cc, k)];
                    ff& v = K[is_tri(i, cc)];
                    const float pr = __fmul_rn(x.hi, y.hi);
                    const float e = fmaf(x.hi, y.lo, fmaf(x.lo, y.hi, fmaf(x.hi, y.hi, -pr)));
                    float sh, sl;
                    two_sum(v.hi, -pr, sh, sl);
                    sl = __fadd_rn(sl, __fsub_rn(v.lo, e));
                    fast_two_sum(sh, sl, v.hi, v.lo);
                }
                team_sync();
                // column k of the FP32 factor (the Gram's column k has been used)
                for (int i = k + 1 + tt; i < S; i += TT) L[is_tri(i, k)] = K[is_tri(i, k)].hi * il;
            }
            team_sync();
            ffexp det{ff{1.f, 0.f}, 0};
            ff yy{0.f, 0.f};
            if (wt == 0) {
                // log det from the float-float product of the pivots (exponents apart)
                for (int k = lane; k < S; k += 32) ffexp_mul(det, piv[k]);
                #pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    const ff om{__shfl_xor_sync(0xffffffffu, det.m.hi, o), __shfl_xor_sync(0xffffffffu, det.m.lo, o)};
                    const int oe = __shfl_xor_sync(0xffffffffu, det.e, o);
                    ffexp_mul(det, om);
                    det.e += oe;
                }
                // L L^T y = t
                const float i0 = lane < S ? ild[lane] : 0.f, i1 = lane + 32 < S ? ild[lane + 32] : 0.f;
                auto solve_step = [&](int k, bool fwd) {
                    const bool hi_row = k >= 32;
                    const float2 own = hi_row ? r1 : r0;
                    const float io = hi_row ? i1 : i0;
                    const float2 yk = make_float2(__shfl_sync(0xffffffffu, own.x * io, k & 31),
                                                  __shfl_sync(0xffffffffu, own.y * io, k & 31));
                    if (lane == (k & 31)) { if (hi_row) r1 = yk; else r0 = yk; }
                    auto upd = [&](int i, float2& r) {
                        if (fwd ? (i > k && i < S) : (i < k)) {
                            const float l = fwd ? L[is_tri(i, k)] : L[is_tri(k, i)];
                            r.x = fmaf(-l, yk.x, r.x);
                            r.y = fmaf(-l, yk.y, r.y);
                        }
                    };
                    upd(lane, r0);
                    if (S > 32) upd(lane + 32, r1);
                };
                for (int k = 0; k < S; ++k) solve_step(k, true);
                for (int k = S - 1; k >= 0; --k) solve_step(k, false);
                // w = A c pi mu + (dA) y, |y|^2 and the grid of the residual's sums
                float wsum = 0.f;
                for (int half = 0; half < (S > 32 ? 2 : 1); ++half) {
                    const int a = lane + 32 * half;
                    if (a >= S) continue;
                    const float2 y = half ? r1 : r0;
                    ff_acc_sq(yy, y);
                    const float2 w0 = ws[a], wv = make_float2(fmaf(dA[a], y.x, w0.x), fmaf(dA[a], y.y, w0.y));
                    ws[a] = wv;
                    wsum += fabsf(wv.x) + fabsf(wv.y);
                }
                yy = warp_sum_ff(yy);
                wsum = warp_sum_f(wsum);
                int gE;
                frexpf(4.0f * (zmax + 2.0f * wsum) + 1e-30f, &gE);
                if (lane == 0) *gmS = ldexpf(1.5f, gE);
            }
            team_sync();
            const float GM = *gmS;
            ff rr{0.f, 0.f};
            for (int k = tt; k < dm.Nh; k += TT) {
                const int f = k / Nm, ym = k - f * Nm;
                bool cj;
                const int ih = is_half(ym, Nm, dm.Nmh, cj);
                const bool mid = odd && k == dm.Nh - 1;
                const float mul = mid ? 1.0f : 2.0f;
                const float4 pv = zp[k], qv = zq[k];
                // acc: grid sum + GM; rem: what the grid left
                float acc[4] = {__fadd_rn(pv.x, GM), __fadd_rn(pv.y, GM), __fadd_rn(qv.x, GM), __fadd_rn(qv.y, GM)};
                float rem[4] = {__fsub_rn(pv.x, __fsub_rn(acc[0], GM)) + pv.z, __fsub_rn(pv.y, __fsub_rn(acc[1], GM)) + pv.w,
                                __fsub_rn(qv.x, __fsub_rn(acc[2], GM)) + qv.z, __fsub_rn(qv.y, __fsub_rn(acc[3], GM)) + qv.w};
                const float4 *fb = fac + f, *cb = ct + ih;
                for (int s = 0; s < S; ++s) {
                    const float4 u = pair_mul_fx(fb[s * dm.hf], conj_if(cb[s * dm.Nmh], cj));
                    const float2 wv = ws[s];
                    const float wx = -mul * wv.x, wy = -mul * wv.y;
                    auto mac = [&](int i, float a, float b, float bl) {
                        const float t = fmaf(a, b, acc[i]);
                        const float d = __fsub_rn(acc[i], t);        // minus the grid part: exact
                        rem[i] += fmaf(a, bl, fmaf(a, b, d));
                        acc[i] = t;
                    };
                    mac(0, wx, u.x, u.z);
                    mac(1, wy, u.x, u.z);
                    mac(2, -wy, u.y, u.w);
                    mac(3, wx, u.y, u.w);
                }
                float e = 0.f;
                ff q{0.f, 0.f};
                #pragma unroll
                for (int i = 0; i < 4; i += 2) {
                    float hx, lx, hy, ly;
                    two_sum(__fsub_rn(acc[i], GM), rem[i], hx, lx);
                    two_sum(__fsub_rn(acc[i + 1], GM), rem[i + 1], hy, ly);
                    ff_acc_sq(q, make_float2(hx, hy));
                    e = fmaf(2.0f * hx, lx, fmaf(2.0f * hy, ly, e));
                }
                q.lo += e;
                const float sc = mid ? 1.0f : 0.5f;
                rr = ff_add(rr, ff{sc * q.hi, sc * q.lo});
            }
            rr = warp_sum_ff(rr);
            if constexpr (TW > 1) {
                if (lane == 0) red[wt] = rr;
                team_sync();
                rr = red[0];
                for (int q = 1; q < TW; ++q) rr = ff_add(rr, red[q]);
            }
            if (tt == 0) {
                const double lg = lgs[j];
                part[j] = -(ff_to_d(rr) * ies[j] + ff_to_d(yy)) - (ffexp_log(det) - S * lg) - Nz * (IS_LOG_PI + lg);
                rat[j] = ratio2;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double t = 0.0;
            float r2 = 0.f;
            for (int j = 0; j < J; ++j) { t += part[j]; r2 += rat[j]; }
            D.lw_x[p] = t;
            if (all && sqrtf(r2) > IF_RATIO_MAX) {
                const int slot = atomicAdd(&D.flags[0], 1);
                if (bp_in_range(slot, P, D.kerr)) D.flags[1 + slot] = p;
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- FP32 evaluation with an error bound
// Every particle from 24 PFs on (the quantities, the bound and the selection are those of
// k_iota_bulk.cu): log det A and rhs^H A^-1 rhs from one LDL^T elimination of the real A, e = z -
// sum_s w0_s u_s element by element, |e|^2 - rhs^H A^-1 rhs.  One warp per (particle, PA); the lower
// triangle lives in registers, lane (tr, tc) of 8 x 4 owning the entries (8 ia + tr, 4 ib + tc);
// column k travels through shared memory (published by its owners one step ahead, one warp
// barrier per step).
// Bound: FP32 issue (about half of it the FMAs of Gram, elimination, e and rhs).  A block of 64
// threads per particle on the complex matrix took 27.7 ms at 64 PFs x 1e5 particles (Nz = 160) and
// 69 ms at 32 x 262144 (Nz = 1024).
constexpr float IB_ERR_PER_RATIO = 4.0e-6f;    // as in k_iota_bulk.cu
constexpr float IB_ERR_PER_ENERGY = 1.0e-6f;
constexpr int IB_W = 4;                        // warps (PAs of a particle) per block
constexpr int IB_FC = 4;                       // frequencies per lane and pass of the residual
constexpr int IB_CR = 12, IB_CC = 20;          // strides of the published column (conflict-free 128-bit reads)
struct IbPlan { size_t fac, ct, pq, col, vec, warp; int fst, cst; };
template <int NB>
__host__ __device__ inline IbPlan ib_plan(const DevGeom& G, int S) {
    const IsDims d = is_dims(G);
    IbPlan p{};
    p.fst = d.hf | 1;                          // odd row strides
    p.cst = d.Nmh | 1;
    size_t o = 0;
    p.pq = o; o += (size_t)d.Fh * G.My * G.Mz * sizeof(float4);
    p.col = o; o += 2 * (8 * IB_CR + 4 * IB_CC) * sizeof(float);
    p.fac = o; o += (size_t)S * p.fst * sizeof(float2);
    p.ct = o; o += (size_t)S * p.cst * sizeof(float2);
    p.vec = o; o += (size_t)8 * NB * (sizeof(float2) + sizeof(float));
    p.warp = (o + 15) & ~(size_t)15;
    return p;
}
constexpr size_t IB_FIXED = 2 * 16 * (sizeof(double) + 2 * sizeof(float));

// registers: 168 (72 of them the triangle) up to 64 PFs, 3 blocks of four warps per SM; 80 up to 32 PFs
template <int NB>
__global__ void __launch_bounds__(32 * IB_W, NB > 4 ? 3 : 6) k_iota_bulk_sym(DevGeom G, DevParams Pm, DevState D, int S, const float* __restrict__ z,
                                                          int W) {
    constexpr int NSL = NB * (NB + 1);                          // register slots (ia, ib <= 2 ia + 1)
    static_assert(NB <= 8, "column buffer strides");
    extern __shared__ float4 smb[];
    const int P = Pm.P, J = G.J, Nz = G.Nz, Nf = G.Nf, My = G.My, Mz = G.Mz, Nm = My * Mz;
    const IsDims dm = is_dims(G);
    const IbPlan pl = ib_plan<NB>(G, S);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tr = lane & 7, tc = lane >> 3;
    double* part = reinterpret_cast<double*>(smb);              // [2][16] log iota per PA (particle parity)
    float* perr = reinterpret_cast<float*>(part + 32);          // [2][16] bound per PA
    float* pbad = perr + 32;                                    // [2][16] breakdown per PA
    char* base = reinterpret_cast<char*>(smb) + IB_FIXED + (size_t)wid * pl.warp;
    float4* pq = reinterpret_cast<float4*>(base + pl.pq);       // [Fh Nm] e: P, Q
    float* col = reinterpret_cast<float*>(base + pl.col);       // [2][by row residue 8 x IB_CR | by column residue 4 x IB_CC]
    float2* fac = reinterpret_cast<float2*>(base + pl.fac);     // [S][fst] b_f, a_y, a_z (half of each)
    float2* ct = reinterpret_cast<float2*>(base + pl.ct);       // [S][cst] a_y a_z (half)
    float2* ws = reinterpret_cast<float2*>(base + pl.vec);      // [8 NB] A c pi mu
    float* dA = reinterpret_cast<float*>(ws + 8 * NB);          // [8 NB] d_s A_s
    const float* phi = D.phi[D.cur];
    const bool odd = Nz & 1;
    // element blocks of the residual: NL lanes over (y, m), the groups of lanes over frequencies
    const int NL = min(Nm, 32), ngrp = 32 / NL, lg = lane / NL, ly = lane - lg * NL;
    const int npass = (dm.Fh + ngrp * IB_FC - 1) / (ngrp * IB_FC), fc = (dm.Fh + ngrp * npass - 1) / (ngrp * npass);
    int par = 0;
    for (int p = blockIdx.x; p < P; p += gridDim.x, par ^= 1) {
        for (int j = wid; j < J; j += W) {
            __syncwarp();
            const float ebf = (float)D.eta_bar[j];
            for (int s = lane; s < 8 * NB; s += 32) {
                float2 w = make_float2(0.f, 0.f);
                float d = 0.f;
                if (s < S) {
                    const float* ph = phi + (size_t)s * 6 * P + p;
                    const float4 g = D.geo[((size_t)s * J + j) * P + p];
                    const float A = G.amp_c / (g.x + g.y);
                    float h, l;
                    ff_frac_mul2(g.x, g.y, G.inv_lam_hi, G.inv_lam_lo, h, l);
                    const float2 c = cispi_ff(-2.0f * h, -2.0f * l);
                    const float pi = (float)(D.zeta[s * J + j] * D.W[s]);
                    const float gm = ph[3 * (size_t)P], mr = ph[4 * (size_t)P], mi = ph[5 * (size_t)P];
                    d = A * sqrtf(fmaxf(pi * (gm + (mr * mr + mi * mi) * (1.0f - pi)), 0.0f));
                    w = cmul(make_float2(A * pi * mr, A * pi * mi), c);
                }
                ws[s] = w;
                dA[s] = d;
            }
            for (int i = lane; i < S * dm.hf; i += 32) {
                const int s = i / dm.hf, q = i - s * dm.hf;
                const size_t gi = ((size_t)s * J + j) * P + p;
                const float4 g = D.geo[gi];
                float th, tl;
                if (q < dm.Fh) {
                    ff_frac_mul2(g.x, g.y, G.fc_hi[q], G.fc_lo[q], th, tl);
                    th = -th; tl = -tl;
                } else {
                    const float2 gl = D.geo_lo[gi];
                    const bool y = q < dm.Fh + dm.hy;
                    const int e = q - dm.Fh - (y ? 0 : dm.hy);
                    const float c = y ? G.py_l[e] : G.pz_l[e], cl = y ? G.py_lo[e] : G.pz_lo[e];
                    const float u = y ? g.z : g.w, ul = y ? gl.x : gl.y;
                    th = __fmul_rn(c, u);
                    tl = fmaf(c, ul, fmaf(cl, u, fmaf(c, u, -th)));
                }
                fac[s * pl.fst + q] = cispi_ff(2.0f * th, 2.0f * tl);
            }
            __syncwarp();
            for (int i = lane; i < S * dm.Nmh; i += 32) {
                const int s = i / dm.Nmh, ym = i - s * dm.Nmh, y = ym / Mz, m = ym - y * Mz;
                const float2* fs = fac + s * pl.fst + dm.Fh;
                bool cy, cz;
                const int iy = is_half(y, My, dm.hy, cy), iz = is_half(m, Mz, dm.hz, cz);
                float2 a = fs[iy], b = fs[dm.hy + iz];
                if (cy) a.y = -a.y;
                if (cz) b.y = -b.y;
                ct[s * pl.cst + ym] = cmul(a, b);
            }
            __syncwarp();
            // e = z - sum_s w0_s u_s as sums and differences of mirrored elements; |e|^2
            float ee = 0.f;
            for (int y0 = 0; y0 < Nm; y0 += NL) {
                const int ym = y0 + ly;
                bool cj = false;
                const int ih = ym < Nm ? is_half(ym, Nm, dm.Nmh, cj) : 0;
                const float sg = cj ? -1.0f : 1.0f;
                for (int ps = 0; ps < npass; ++ps) {
                    const int f0 = (ps * ngrp + lg) * fc;
                    const bool act = ym < Nm && lg < ngrp && f0 < dm.Fh;
                    float4 a[IB_FC];
                    #pragma unroll
                    for (int i = 0; i < IB_FC; ++i) {
                        const int k = (f0 + i) * Nm + ym;
                        a[i] = make_float4(0.f, 0.f, 0.f, 0.f);
                        if (act && i < fc && f0 + i < dm.Fh && k < dm.Nh) {
                            const float* za = z + 2 * ((size_t)j * Nz + k);
                            const float* zb = z + 2 * ((size_t)j * Nz + Nz - 1 - k);
                            a[i] = make_float4(za[0] + zb[0], za[1] + zb[1], za[0] - zb[0], za[1] - zb[1]);
                            if (odd && k == dm.Nh - 1) a[i] = make_float4(2.0f * za[0], 2.0f * za[1], 0.f, 0.f);
                        }
                    }
                    const int fl = act ? f0 : 0;
                    for (int s = 0; s < S; ++s) {
                        float2 c = ct[s * pl.cst + ih];
                        c.y *= sg;
                        const float2 w = ws[s];
                        const float2* b = fac + s * pl.fst + fl;
                        #pragma unroll
                        for (int i = 0; i < IB_FC; ++i) {
                            if (i < fc) {
                                const float2 bb = b[i];
                                const float x2 = 2.0f * fmaf(bb.x, c.x, -bb.y * c.y), y2 = 2.0f * fmaf(bb.x, c.y, bb.y * c.x);
                                a[i].x = fmaf(-w.x, x2, a[i].x);
                                a[i].y = fmaf(-w.y, x2, a[i].y);
                                a[i].z = fmaf(w.y, y2, a[i].z);
                                a[i].w = fmaf(-w.x, y2, a[i].w);
                            }
                        }
                    }
                    #pragma unroll
                    for (int i = 0; i < IB_FC; ++i) {
                        const int k = (f0 + i) * Nm + ym;
                        if (act && i < fc && f0 + i < dm.Fh) {
                            float4 v = a[i];
                            if (k >= dm.Nh) v = make_float4(0.f, 0.f, 0.f, 0.f);
                            const float q = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, v.w * v.w)));
                            if (odd && k == dm.Nh - 1) {         // carried doubled
                                v.x *= 0.5f; v.y *= 0.5f; v.z = 0.f; v.w = 0.f;
                                ee += fmaf(v.x, v.x, v.y * v.y);
                            } else {
                                ee = fmaf(0.5f, q, ee);
                            }
                            pq[k] = v;
                        }
                    }
                }
            }
            ee = warp_sum_f(ee);
            __syncwarp();
            // rhs_s = (dA)_s u_s^H e, rows lane and lane + 32: per frequency the sums over (y, m), the mirrored
            // element's factor being the conjugate
            float2 rhs[2];
            #pragma unroll
            for (int hr = 0; hr < (NB > 4 ? 2 : 1); ++hr) {
                const int s = lane + 32 * hr;
                float2 g = make_float2(0.f, 0.f);
                if (s < S) {
                    const float2 *fs = fac + s * pl.fst, *cs = ct + s * pl.cst;
                    for (int f = 0; f < dm.Fh; ++f) {
                        float2 al = make_float2(0.f, 0.f), be = al;
                        const float4* ef = pq + f * Nm;
                        auto add = [&](float2 c, float4 e) {
                            al.x = fmaf(c.x, e.x, fmaf(c.y, e.w, al.x));
                            al.y = fmaf(c.x, e.y, fmaf(-c.y, e.z, al.y));
                            be.x = fmaf(c.y, e.x, fmaf(-c.x, e.w, be.x));
                            be.y = fmaf(c.y, e.y, fmaf(c.x, e.z, be.y));
                        };
                        for (int ym = 0; ym < Nm / 2; ++ym) {
                            const float2 c = cs[ym];
                            add(c, ef[ym]);
                            add(make_float2(c.x, -c.y), ef[Nm - 1 - ym]);
                        }
                        if (Nm & 1) add(cs[Nm / 2], ef[Nm / 2]);
                        const float2 b = fs[f];
                        g.x = fmaf(b.x, al.x, fmaf(-b.y, be.x, g.x));
                        g.y = fmaf(b.x, al.y, fmaf(-b.y, be.y, g.y));
                    }
                    g = make_float2(dA[s] * g.x, dA[s] * g.y);
                }
                rhs[hr] = g;
            }
            // Gram of this lane's entries: frequencies, then the antenna factors row block by row block
            float A[NSL];
            #pragma unroll
            for (int q = 0; q < NSL; ++q) A[q] = 0.f;
            auto ld = [&](int s, int q) { return s < S ? fac[s * pl.fst + q] : make_float2(0.f, 0.f); };
            for (int f = 0; f < Nf / 2; ++f) {
                float2 ra[NB];
                #pragma unroll
                for (int ia = 0; ia < NB; ++ia) ra[ia] = ld(8 * ia + tr, f);
                #pragma unroll
                for (int ib = 0; ib < 2 * NB; ++ib) {
                    const float2 cb = ld(4 * ib + tc, f);
                    #pragma unroll
                    for (int ia = ib / 2; ia < NB; ++ia) {
                        float& v = A[ia * (ia + 1) + ib];
                        v = fmaf(ra[ia].x, cb.x, fmaf(ra[ia].y, cb.y, v));
                    }
                }
            }
            const float mf = (Nf & 1) ? 1.0f : 0.0f, my = (My & 1) ? 1.0f : 0.0f, mz = (Mz & 1) ? 1.0f : 0.0f;
            #pragma unroll
            for (int ia = 0; ia < NB; ++ia) {
                float sy[2 * NB], sz[2 * NB];
                #pragma unroll
                for (int ib = 0; ib <= 2 * ia + 1; ++ib) sy[ib] = sz[ib] = 0.f;
                const int a = 8 * ia + tr;
                for (int u = 0; u < My / 2; ++u) {
                    const float2 r = ld(a, dm.Fh + u);
                    #pragma unroll
                    for (int ib = 0; ib <= 2 * ia + 1; ++ib) {
                        const float2 cb = ld(4 * ib + tc, dm.Fh + u);
                        sy[ib] = fmaf(r.x, cb.x, fmaf(r.y, cb.y, sy[ib]));
                    }
                }
                for (int u = 0; u < Mz / 2; ++u) {
                    const float2 r = ld(a, dm.Fh + dm.hy + u);
                    #pragma unroll
                    for (int ib = 0; ib <= 2 * ia + 1; ++ib) {
                        const float2 cb = ld(4 * ib + tc, dm.Fh + dm.hy + u);
                        sz[ib] = fmaf(r.x, cb.x, fmaf(r.y, cb.y, sz[ib]));
                    }
                }
                const float da = dA[a];
                #pragma unroll
                for (int ib = 0; ib <= 2 * ia + 1; ++ib) {
                    const int b = 4 * ib + tc;
                    float& v = A[ia * (ia + 1) + ib];
                    // rows and columns beyond S have dA = 0: the identity
                    v = fmaf(2.0f, v, mf) * (fmaf(2.0f, sy[ib], my) * fmaf(2.0f, sz[ib], mz)) * (da * dA[b]);
                    if (a == b) v = a < S ? v + ebf : 1.0f;
                }
            }
            // LDL^T elimination with the forward substitution
            float yy = 0.f, pv0 = 1.f, pv1 = 1.f;
            auto publish = [&](int buf, int row, float v) {
                float* c = col + buf * (8 * IB_CR + 4 * IB_CC);
                c[(row & 7) * IB_CR + (row >> 3)] = v;
                c[8 * IB_CR + (row & 3) * IB_CC + (row >> 2)] = v;
            };
            if (tc == 0) {
                #pragma unroll
                for (int ia = 0; ia < NB; ++ia) publish(0, 8 * ia + tr, A[ia * (ia + 1)]);
            }
            __syncwarp();
            #pragma unroll
            for (int kb = 0; kb < 2 * NB; ++kb) {               // columns 4 kb .. 4 kb + 3: slots ib = kb
                #pragma unroll 1
                for (int r = 0; r < 4; ++r) {
                    const int k = 4 * kb + r;
                    if (k >= S) break;                          // uniform
                    const int K = kb / 2;
                    const float* cr = col + (k & 1) * (8 * IB_CR + 4 * IB_CC);
                    const float* cc = cr + 8 * IB_CR;
                    const float piv = cc[(k & 3) * IB_CC + (k >> 2)];
                    const float ipiv = 1.0f / piv;
                    // forward substitution: y_k = rhs_k / piv_k, rhs_i -= A_ik y_k
                    {
                        const float2 own = (NB > 4 && k >= 32) ? rhs[1] : rhs[0];
                        const float2 rk = make_float2(__shfl_sync(0xffffffffu, own.x, k & 31), __shfl_sync(0xffffffffu, own.y, k & 31));
                        const float2 y = make_float2(rk.x * ipiv, rk.y * ipiv);
                        if (lane == (k & 31)) {
                            yy = fmaf(fmaf(rk.x, rk.x, rk.y * rk.y), ipiv, yy);
                            if (NB > 4 && k >= 32) pv1 = piv; else pv0 = piv;
                        }
                        if (lane > k && lane < S) {
                            const float v = cr[(lane & 7) * IB_CR + (lane >> 3)];
                            rhs[0].x = fmaf(-v, y.x, rhs[0].x);
                            rhs[0].y = fmaf(-v, y.y, rhs[0].y);
                        }
                        if (NB > 4 && lane + 32 > k && lane + 32 < S) {
                            const float v = cr[(lane & 7) * IB_CR + (lane >> 3) + 4];
                            rhs[1].x = fmaf(-v, y.x, rhs[1].x);
                            rhs[1].y = fmaf(-v, y.y, rhs[1].y);
                        }
                    }
                    float xa[8], xc[16];
                    #pragma unroll
                    for (int q = 0; q < NB; q += 4) {
                        if (q + 3 >= K) {
                            const float4 v = *reinterpret_cast<const float4*>(cr + tr * IB_CR + q);
                            xa[q] = v.x * -ipiv; xa[q + 1] = v.y * -ipiv; xa[q + 2] = v.z * -ipiv; xa[q + 3] = v.w * -ipiv;
                        }
                    }
                    #pragma unroll
                    for (int q = 0; q < 2 * NB; q += 4) {
                        if (q + 3 >= kb) {
                            const float4 v = *reinterpret_cast<const float4*>(cc + tc * IB_CC + q);
                            xc[q] = v.x; xc[q + 1] = v.y; xc[q + 2] = v.z; xc[q + 3] = v.w;
                        }
                    }
                    // the trailing entries: columns beyond k (in the slot of column k only those of larger residue)
                    #pragma unroll
                    for (int ia = K; ia < NB; ++ia) {
                        #pragma unroll
                        for (int ib = kb; ib <= 2 * ia + 1; ++ib) {
                            float& v = A[ia * (ia + 1) + ib];
                            if (ib > kb || tc > r) v = fmaf(xa[ia], xc[ib], v);
                        }
                    }
                    // owners of column k + 1 publish it
                    if (r < 3) {
                        if (tc == r + 1) {
                            #pragma unroll
                            for (int ia = K; ia < NB; ++ia) publish((k + 1) & 1, 8 * ia + tr, A[ia * (ia + 1) + kb]);
                        }
                    } else if (kb + 1 < 2 * NB) {
                        if (tc == 0) {
                            #pragma unroll
                            for (int ia = (kb + 1) / 2; ia < NB; ++ia)
                                publish((k + 1) & 1, 8 * ia + tr, A[ia * (ia + 1) + (kb + 1 < 2 * NB ? kb + 1 : kb)]);
                        }
                    }
                    __syncwarp();
                }
            }
            // log det, sum A_kk / piv_k, the smallest pivot
            float dm0 = 1.f, rsum = 0.f, pmin = 3.0e38f;
            int de = 0;
            auto take = [&](int k, float pv) {
                if (k >= S) return;
                int e;
                dm0 = frexpf(dm0 * pv, &e);
                de += e;
                rsum += fmaf(dA[k] * dA[k], (float)Nz, ebf) / pv;
                pmin = fminf(pmin, pv);
            };
            take(lane, pv0);
            if (NB > 4) take(lane + 32, pv1);
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                int e;
                dm0 = frexpf(dm0 * __shfl_xor_sync(0xffffffffu, dm0, o), &e);
                de += __shfl_xor_sync(0xffffffffu, de, o) + e;
                rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
                pmin = fminf(pmin, __shfl_xor_sync(0xffffffffu, pmin, o));
            }
            yy = warp_sum_f(yy);
            if (lane == 0) {
                const double eb = D.eta_bar[j];
                const double q = (double)ee - (double)yy;       // eta_bar e^H C^-1 e
                const double logdet = log((double)dm0) + (double)de * 0.69314718055994530942;
                const double lgb = log(eb);
                const double v = -q / eb - logdet - (double)(Nz - S) * lgb - (double)Nz * IS_LOG_PI;
                const float eq = IB_ERR_PER_ENERGY * (float)(((double)ee + (double)yy) / eb);
                part[par * 16 + j] = v;
                perr[par * 16 + j] = IB_ERR_PER_RATIO * rsum + eq;
                // every pivot of eta_bar I + D G D is at least eta_bar, and q >= 0: anything else is a
                // breakdown of the FP32 elimination
                pbad[par * 16 + j] = (!(pmin > 0.5f * ebf) || !(q / eb > -(double)eq) || !isfinite(v)) ? 1.f : 0.f;
            }
        }
        __syncthreads();   // the buffers of the other parity are free again after the next one
        if (threadIdx.x == 0) {
            double t = 0.0;
            float e = 0.f, bad = 0.f;
            for (int j = 0; j < J; ++j) { t += part[par * 16 + j]; e += perr[par * 16 + j]; bad += pbad[par * 16 + j]; }
            D.lw_x[p] = t;
            D.iota_err[p] = bad != 0.f ? INFINITY : e;
        }
    }
}

template <int NB>
static bool launch_bulk_sym_nb(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, cudaStream_t st) {
    const size_t warp = ib_plan<NB>(G, S).warp, limit = 227 * 1024;
    int W = min(G.J, IB_W);
    while (W > 1 && IB_FIXED + W * warp > limit) --W;
    const size_t smem = IB_FIXED + W * warp;
    if (smem > limit) return false;
    smem_allow_max((const void*)k_iota_bulk_sym<NB>);
    const int per_sm = max(1, min(32 / W, (int)((limit + 1024) / (smem + 1024))));
    k_iota_bulk_sym<NB><<<min(Pm.P, sm_count() * per_sm * 4), 32 * W, smem, st>>>(G, Pm, D, S, z, W);
    return true;
}

// FP32 log iota~ with error bounds of every particle; false if the layout or the sizes do not allow it
bool launch_iota_bulk_sym(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, cudaStream_t st) {
    if (!G.sym) return false;
    if (S <= 32) return launch_bulk_sym_nb<4>(G, Pm, D, S, z, st);
    return launch_bulk_sym_nb<8>(G, Pm, D, S, z, st);
}

// whether the real form applies: a symmetric layout whose working set fits one warp
bool iota_sym_ok(const DevGeom& G, int S) {
    return G.sym && ((IF_FIXED + 15) & ~(size_t)15) + if_plan(G, S).warp <= 227 * 1024;
}

// float-float log iota~ of every particle (all), or of the queued ones
void launch_iota_ff(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, bool all, cudaStream_t st) {
    const size_t fixed = (IF_FIXED + 15) & ~(size_t)15, warp = if_plan(G, S).warp, limit = 227 * 1024;
    const int TW = all ? 1 : IF_TEAM_MAX;
    int W = min(G.J, (TW == 1 ? 8 : 16) / TW);
    while (W > 1 && fixed + W * warp > limit) --W;
    const size_t smem = fixed + W * warp;
    const int per_sm = max(1, min(64 / (W * TW), (int)((limit + 1024) / (smem + 1024))));
    if (all) cudaMemsetAsync(D.flags, 0, sizeof(int), st);
    auto go = [&](auto kernel) {
        smem_allow_max((const void*)kernel);
        kernel<<<min(Pm.P, sm_count() * per_sm), 32 * TW * W, smem, st>>>(G, Pm, D, S, z, all ? 1 : 0, W);
    };
    if (TW == 1) go(k_iota_ff<1>);
    else go(k_iota_ff<IF_TEAM_MAX>);
}

}  // namespace bp
