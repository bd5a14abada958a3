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
// steering elements as (hi, lo) pairs (~1e-10) with the products of the high parts summed exactly on
// a grid fixed per (p, j).  Below 24 PFs every particle is evaluated (the FP32 warp kernel and the
// block-per-particle repair of the particles it flagged took 8.7 ms at 10 PFs x 30000 particles,
// Nz = 160; this 1.32 ms with index divisions, a search per triangle entry and a reduction per PF, 0.99
// without); from 24 PFs on the particles k_iota_select queues, with four warps
// per team, since few working sets of that size fit an SM.
// Bound: FP32 issue, the residual's ~50 instructions per (s, half element).
constexpr int IF_WMAX = 16;
constexpr float IF_RATIO_MAX = 100.0f;   // reported as ill-conditioned: sqrt(sum (A_kk / piv_k)^2) above this
struct IfPlan { size_t fac, ct, K, L, vec, z, warp; };
__host__ __device__ inline IfPlan if_plan(const DevGeom& G, int S) {
    const IsDims d = is_dims(G);
    IfPlan p{};
    size_t o = 0;
    p.fac = o; o += (size_t)S * (d.hf | 1) * sizeof(float4);
    p.ct = o; o += (size_t)S * d.Nmh * sizeof(float4);
    p.z = o; o += (size_t)d.Nh * 2 * sizeof(float4);            // P (hi, lo), Q (hi, lo)
    p.vec = o; o += (size_t)S * (sizeof(float4) + sizeof(float2) + sizeof(ff) + 2 * sizeof(float));   // w, g | pivots | dA, 1/L_kk
    p.K = o; o += (size_t)S * (S + 1) / 2 * sizeof(ff);
    p.L = o; o += (size_t)S * (S + 1) / 2 * sizeof(float);
    p.warp = (o + 15) & ~(size_t)15;
    return p;
}
constexpr int IF_TEAM_MAX = 4;           // warps of a team
// n / d by a multiplication (n d < 2^32)
struct IsDiv { uint32_t m, d; };
__device__ __forceinline__ IsDiv is_div(int d) { return IsDiv{0xffffffffu / (uint32_t)d + 1u, (uint32_t)d}; }
__device__ __forceinline__ int operator/(int n, IsDiv v) { return v.d == 1 ? n : (int)__umulhi((uint32_t)n, v.m); }
constexpr size_t IF_FIXED = 256 * sizeof(float4) + IF_WMAX * (3 * sizeof(double) + sizeof(float)) +
                            IF_WMAX * IF_TEAM_MAX * sizeof(ff) + IF_WMAX * sizeof(float);
// shared by the block: IF_FIXED, the elements' places [Nh], the triangle's (row, column) [S (S + 1) / 2]
__host__ __device__ inline size_t if_fixed(const DevGeom& G, int S) {
    return (IF_FIXED + (size_t)is_dims(G).Nh * sizeof(uint32_t) + (size_t)S * (S + 1) / 2 * sizeof(ushort) + 15) & ~(size_t)15;
}

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
    const int fst = dm.hf | 1;                                  // odd: rows on distinct banks (an even
    // stride of 40 cost 40 PFs x 8192 of Nz = 300 0.87 ms of 3.3)
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
    uint32_t* kt = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(smf) + IF_FIXED);   // [Nh] f, index and conjugation of a_y a_z
    ushort* tri = reinterpret_cast<ushort*>(kt + dm.Nh);        // [S (S + 1) / 2] row, column
    const IfPlan pl = if_plan(G, S);
    char* base = reinterpret_cast<char*>(smf) + if_fixed(G, S) + (size_t)wid * pl.warp;
    float4* fac = reinterpret_cast<float4*>(base + pl.fac);     // [S][fst] b_f, a_y, a_z (half of each)
    float4* ct = reinterpret_cast<float4*>(base + pl.ct);       // [S][Nmh] a_y a_z
    float4* zp = reinterpret_cast<float4*>(base + pl.z);        // [Nh] P, then [Nh] Q, as (hi, lo)
    float4* zq = zp + dm.Nh;
    ff* K = reinterpret_cast<ff*>(base + pl.K);                 // packed lower: A, then its elimination
    float4* ws = reinterpret_cast<float4*>(base + pl.vec);      // [S] (A c pi mu), then -2 w, (2 Im w, -2 Re w)
    float2* gs = reinterpret_cast<float2*>(ws + S);             // [S] u^H z
    ff* piv = reinterpret_cast<ff*>(gs + S);                    // [S]
    float* dA = reinterpret_cast<float*>(piv + S);              // [S] d_s A_s
    float* ild = dA + S;                                        // [S] 1 / L_kk
    float* L = reinterpret_cast<float*>(base + pl.L);           // packed lower: the FP32 Gram, then the FP32 factor
    for (int i = threadIdx.x; i < 256; i += blockDim.x) ctab[i] = D.ctab[i];
    if (threadIdx.x < J) {
        lgs[threadIdx.x] = log(D.eta_bar[threadIdx.x]);
        ies[threadIdx.x] = 1.0 / D.eta_bar[threadIdx.x];
    }
    for (int k = threadIdx.x; k < dm.Nh; k += blockDim.x) {
        const int f = k / Nm;
        bool cj;
        const int ih = is_half(k - f * Nm, Nm, dm.Nmh, cj);
        kt[k] = (uint32_t)f | ((uint32_t)ih << 15) | (cj ? 0x80000000u : 0u);
    }
    for (int t = threadIdx.x; t < S * (S + 1) / 2; t += blockDim.x) {
        int a, b;
        is_tri_ab(t, a, b);
        tri[t] = (ushort)(a | (b << 8));
    }
    __syncthreads();
    const IsDiv by_hf = is_div(dm.hf), by_Nmh = is_div(dm.Nmh), by_Mz = is_div(Mz);
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
            const float ebh = (float)eb, ebl = (float)(eb - (double)ebh);
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
                const float2 w0 = cmul(make_float2(A * pi * mr, A * pi * mi), c);
                ws[s] = make_float4(w0.x, w0.y, 0.f, 0.f);
            }
            for (int i = tt; i < S * dm.hf; i += TT) {
                const int s = i / by_hf, q = i - s * dm.hf;
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
                fac[s * fst + q] = make_float4(hi.x, hi.y, lo.x, lo.y);
            }
            team_sync();
            for (int i = tt; i < S * dm.Nmh; i += TT) {
                const int s = i / by_Nmh, ym = i - s * dm.Nmh, y = ym / by_Mz, m = ym - y * Mz;
                const float4* fs = fac + s * fst + dm.Fh;
                bool cy, cz;
                const int iy = is_half(y, My, dm.hy, cy), iz = is_half(m, Mz, dm.hz, cz);
                ct[i] = pair_mul_fx(conj_if(fs[iy], cy), conj_if(fs[dm.hy + iz], cz));
            }
            // Gram and A = eta_bar I + D G D, packed
            for (int t = tt; t < npair; t += TT) {
                const int a = tri[t] & 255, b = tri[t] >> 8;
                const float4 *fa = fac + a * fst, *fb = fac + b * fst;
                const ff g = ff_mul(if_sum(fa, fb, Nf), ff_mul(if_sum(fa + dm.Fh, fb + dm.Fh, My),
                                                               if_sum(fa + dm.Fh + dm.hy, fb + dm.Fh + dm.hy, Mz)));
                ff v = ff_mul(g, ff_prod(dA[a], dA[b]));
                if (a == b) v = ff_add(v, ff{ebh, ebl});
                K[t] = v;
                L[t] = g.hi;
            }
            team_sync();
            // g_s = u_s^H z (FP32: the minimiser's rounding enters at second order)
            for (int s0 = 4 * wt; s0 < S; s0 += 4 * TW) {     // four PFs at a time
                float g[8];
                #pragma unroll
                for (int q = 0; q < 8; ++q) g[q] = 0.f;
                #pragma unroll 1
                for (int k = lane; k < dm.Nh; k += 32) {
                    const uint32_t at = kt[k];
                    const float4 pv = zp[k], qv = zq[k];
                    const float4 *fs = fac + (at & 0x7fff), *cs = ct + ((at >> 15) & 0xffff);
                    const float sg = (at >> 31) ? -1.0f : 1.0f;
                    #pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int s = min(s0 + q, S - 1);
                        const float2 b = *reinterpret_cast<const float2*>(fs + s * fst);
                        float2 c = *reinterpret_cast<const float2*>(cs + s * dm.Nmh);
                        c.y *= sg;
                        const float x = fmaf(b.x, c.x, -b.y * c.y), y = fmaf(b.x, c.y, b.y * c.x);
                        g[2 * q] = fmaf(x, pv.x, fmaf(y, qv.y, g[2 * q]));
                        g[2 * q + 1] = fmaf(x, pv.y, fmaf(-y, qv.x, g[2 * q + 1]));
                    }
                }
                // the eight sums over lanes at once: halving the values while lanes pair up
                #pragma unroll
                for (int o = 16, n = 4; o >= 4; o >>= 1, n >>= 1) {
                    const bool up = lane & o;
                    #pragma unroll
                    for (int q = 0; q < n; ++q) {
                        const float keep = up ? g[q + n] : g[q], give = up ? g[q] : g[q + n];
                        g[q] = keep + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                }
                g[0] += __shfl_xor_sync(0xffffffffu, g[0], 2);
                g[0] += __shfl_xor_sync(0xffffffffu, g[0], 1);
                // lane bits 4, 3, 2 select value 4 b4 + 2 b3 + b2
                const int s = s0 + (((lane >> 4) & 1) << 1) + ((lane >> 3) & 1);
                if ((lane & 3) == 0 && s < S) reinterpret_cast<float*>(gs + s)[(lane >> 2) & 1] = g[0];
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
                    const float2 w0 = *reinterpret_cast<const float2*>(ws + b);
                    acc.x = fmaf(-g, w0.x, acc.x);
                    acc.y = fmaf(-g, w0.y, acc.y);
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
                    const float akk = fmaf(dA[k] * dA[k], L[is_tri(k, k)], ebh);   // before the elimination
                    ratio2 = fmaf(akk * inv.hi, akk * inv.hi, ratio2);
                }
                const int n = S - k - 1;
                for (int t = tt; t < n * (n + 1) / 2; t += TT) {
                    const int i = k + 1 + (tri[t] & 255), cc = k + 1 + (tri[t] >> 8);
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
                    const float4 w0 = ws[a];
                    const float2 wv = make_float2(fmaf(dA[a], y.x, w0.x), fmaf(dA[a], y.y, w0.y));
                    ws[a] = make_float4(-2.0f * wv.x, -2.0f * wv.y, 2.0f * wv.y, -2.0f * wv.x);
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
            const f2x GM2 = f2_dup(GM);
            #pragma unroll 1
            for (int k = tt; k < dm.Nh; k += TT) {
                const uint32_t at = kt[k];
                const bool mid = odd && k == dm.Nh - 1;
                const float sg = (at >> 31) ? -1.0f : 1.0f, dbl = mid ? 2.0f : 1.0f;   // the middle element is carried doubled
                const float4 pv = zp[k], qv = zq[k];
                // (P re, P im), (Q re, Q im): grid sum + GM, and what the grid left
                const f2x p2 = f2_pack(dbl * pv.x, dbl * pv.y), q2 = f2_pack(qv.x, qv.y);
                f2x acc0 = f2_add(p2, GM2), acc1 = f2_add(q2, GM2);
                f2x rem0 = f2_add(f2_sub(p2, f2_sub(acc0, GM2)), f2_pack(dbl * pv.z, dbl * pv.w));
                f2x rem1 = f2_add(f2_sub(q2, f2_sub(acc1, GM2)), f2_pack(qv.z, qv.w));
                const float4 *fb = fac + (at & 0x7fff), *cb = ct + ((at >> 15) & 0xffff);
                #pragma unroll 2
                for (int s = 0; s < S; ++s) {
                    float4 c = cb[s * dm.Nmh];
                    c.y *= sg;
                    c.w *= sg;
                    const float4 u = pair_mul_fx(fb[s * fst], c);
                    const float4 wv = ws[s];
                    auto mac = [&](f2x& acc, f2x& rem, f2x a, f2x b, f2x bl) {
                        const f2x t = f2_fma(a, b, acc);
                        const f2x d = f2_sub(acc, t);                // minus the grid part: exact
                        rem = f2_add(rem, f2_fma(a, bl, f2_fma(a, b, d)));
                        acc = t;
                    };
                    mac(acc0, rem0, f2_pack(wv.x, wv.y), f2_dup(u.x), f2_dup(u.z));
                    mac(acc1, rem1, f2_pack(wv.z, wv.w), f2_dup(u.y), f2_dup(u.w));
                }
                float e = 0.f;
                ff q{0.f, 0.f};
                #pragma unroll
                for (int i = 0; i < 2; ++i) {
                    uint32_t g0, g1, m0, m1;
                    f2_unpack(f2_sub(i ? acc1 : acc0, GM2), g0, g1);
                    f2_unpack(i ? rem1 : rem0, m0, m1);
                    float hx, lx, hy, ly;
                    two_sum(__uint_as_float(g0), __uint_as_float(m0), hx, lx);
                    two_sum(__uint_as_float(g1), __uint_as_float(m1), hy, ly);
                    ff_acc_sq(q, make_float2(hx, hy));
                    e = fmaf(2.0f * hx, lx, fmaf(2.0f * hy, ly, e));
                }
                q.lo += e;
                const float sc = mid ? 0.25f : 0.5f;
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
            // nothing is left to repair, but the ill-conditioned ones are counted, and listed for the diagnostics
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
// sum_s w0_s u_s element by element, |e|^2 - rhs^H A^-1 rhs.  One warp per (particle, PA).
//   * e: a_y a_z = c of an element (y, m) is conj(c) at the mirrored (My - 1 - y, Mz - 1 - m), so sums and
//     differences over that pair (P+, P-, Q+, Q-) need the products b c only part by part: lanes over
//     the pairs (groups of lanes over PFs where the pairs leave lanes idle), two frequencies per
//     packed FP32 pair, eight packed FMAs per PF, pair and two frequencies.
//   * rhs: lanes over PFs; per frequency the sums over the pairs in the same eight FMAs, then the
//     frequencies' factors.
//   * A: the lower triangle in registers, lane (tr, tc) of 8 x 4 owning (8 ia + tr, 4 ib + tc).  Panels of
//     eight columns go through shared memory: lanes take rows, factor the panel with shuffles (the
//     forward substitution rides along), then every lane applies the rank-8 update to its entries.
// Bound: FP32 issue.  The whole stage at 64 PFs x 1e5 particles (Nz = 160) / 32 x 262144 (Nz = 1024):
// 27.7 / 69 ms with a block of 64 threads per particle on the complex matrix, 15.1 / 54.4 with this
// split but one column of the elimination at a time and unpacked e and rhs, 12.0 / 26.7 with both packed
// element by element and the panels unrolled, 9.4 / 22.1 over mirrored pairs with long loops rolled
// (instruction fetch was a fifth of the stalls), 8.9 / 19.8 as it is (panel in the residual's place, Re and
// Im of the factors in one row: 13.7 instead of 16 KB per warp, 16 instead of 12 warps per SM, at 32 PFs).
constexpr float IB_ERR_PER_RATIO = 4.0e-6f;    // as in k_iota_bulk.cu
constexpr float IB_ERR_PER_ENERGY = 1.0e-6f;
constexpr int IB_W = 4;                        // warps (PAs of a particle) per block
constexpr int IB_FP = 4;                       // frequency pairs per lane and pass
constexpr int IB_Q = 8;                        // Re P+, Im Q-, Im P+, -Re Q-, -Re P-, Im Q+, -Im P-, -Re Q+
constexpr int IB_PST = 12;                     // row stride of the panel (conflict-free 128-bit accesses)
struct IbPlan { size_t pq, pan, fx, fy, ant, vec, warp; int fp, f4, ast; };
template <int NB>
__host__ __device__ inline IbPlan ib_plan(const DevGeom& G, int S) {
    const IsDims d = is_dims(G);
    IbPlan p{};
    p.f4 = (d.Fh + 7) & ~7;                    // frequencies, padded to a lane's four pairs
    p.fp = 2 * p.f4 + 4;                       // stride of a row (Re b, Im b): 16-byte rows, 8 rows on distinct banks
    p.ast = (d.hy + d.hz) | 1;
    const size_t R = 8 * NB;                   // rows beyond S are zero
    size_t o = 0;
    // the panel takes the residual's place, which the elimination no longer needs
    const size_t pq = (size_t)d.Nmh * IB_Q * p.f4 * sizeof(float), pan = R * IB_PST * sizeof(float);
    p.pq = p.pan = o; o += pq > pan ? pq : pan;
    p.fx = o; p.fy = o + p.f4 * sizeof(float); o += R * p.fp * sizeof(float);
    p.vec = o; o += R * (sizeof(float4) + sizeof(float));
    p.ant = o; o += R * p.ast * sizeof(float2);
    p.warp = (o + 15) & ~(size_t)15;
    return p;
}
constexpr size_t IB_FIXED = 2 * 16 * (sizeof(double) + 2 * sizeof(float)) + 2 * 16 * sizeof(double);

// registers: 168 (72 of them the triangle) up to 64 PFs, 3 blocks of four warps per SM; 4 blocks up to 32 PFs
template <int NB>
__global__ void __launch_bounds__(32 * IB_W, NB > 4 ? 3 : 4) k_iota_bulk_sym(DevGeom G, DevParams Pm, DevState D, int S,
                                                                             const float* __restrict__ z, int W) {
    constexpr int NSL = NB * (NB + 1);                          // register slots (ia, ib <= 2 ia + 1)
    constexpr int NR = NB > 4 ? 2 : 1;                          // rows per lane: lane, lane + 32
    extern __shared__ float4 smb[];
    const int P = Pm.P, J = G.J, Nz = G.Nz, Nf = G.Nf, My = G.My, Mz = G.Mz, Nm = My * Mz;
    const IsDims dm = is_dims(G);
    const IbPlan pl = ib_plan<NB>(G, S);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tr = lane & 7, tc = lane >> 3;
    double* part = reinterpret_cast<double*>(smb);              // [2][16] log iota per PA (particle parity)
    double* lgs = part + 32;                                    // [16] log eta_bar
    double* ies = lgs + 16;                                     // [16] 1 / eta_bar
    float* perr = reinterpret_cast<float*>(ies + 16);           // [2][16] bound per PA
    float* pbad = perr + 32;                                    // [2][16] breakdown per PA
    char* base = reinterpret_cast<char*>(smb) + IB_FIXED + (size_t)wid * pl.warp;
    float* pq = reinterpret_cast<float*>(base + pl.pq);         // [Nmh][IB_Q][f4] e
    float* pan = reinterpret_cast<float*>(base + pl.pan);       // [8 NB][IB_PST] panel of eight columns
    float* fx = reinterpret_cast<float*>(base + pl.fx);         // [8 NB][fp] Re b_f
    float* fy = reinterpret_cast<float*>(base + pl.fy);         // [8 NB][fp] Im b_f (in the same rows)
    float2* ant = reinterpret_cast<float2*>(base + pl.ant);     // [8 NB][ast] a_y, a_z (half of each)
    float4* ws = reinterpret_cast<float4*>(base + pl.vec);      // [8 NB] -4 A c pi mu (two parts)
    float* dA = reinterpret_cast<float*>(ws + 8 * NB);          // [8 NB] d_s A_s
    const float* phi = D.phi[D.cur];
    if (threadIdx.x < J) {
        lgs[threadIdx.x] = log(D.eta_bar[threadIdx.x]);
        ies[threadIdx.x] = 1.0 / D.eta_bar[threadIdx.x];
    }
    for (int i = lane; i < 8 * NB * pl.fp; i += 32) fx[i] = 0.f;     // (fy with it) rows and columns beyond S and Fh stay zero
    for (int i = lane; i < 8 * NB * pl.ast; i += 32) ant[i] = make_float2(0.f, 0.f);
    __syncthreads();
    // residual: NL lanes over the element pairs, the groups of lanes over frequency pairs (gf groups of up to
    // IB_FP) and what is left of them over PFs (gs)
    const int np2 = (dm.Fh + 1) / 2;
    const int NL = min(dm.Nmh, 32), ngrp = 32 / NL, gf = min(ngrp, (np2 + IB_FP - 1) / IB_FP), gs = ngrp / gf;
    const int lg = lane / NL, ly = lane - lg * NL, fg = lg % gf, sg = min(lg / gf, gs - 1);
    const bool first = lg < gf;                                 // the lanes that collect
    // Gram over frequencies in pairs; the middle one of an odd count (exactly 1) may be among them
    const int gp = (Nf / 2 + 1) / 2;
    const float mf = (Nf & 1) ? ((Nf / 2) & 1 ? -1.0f : 1.0f) : 0.0f;
    const float my = (My & 1) ? 1.0f : 0.0f, mz = (Mz & 1) ? 1.0f : 0.0f;
    int par = 0;
    for (int p = blockIdx.x; p < P; p += gridDim.x, par ^= 1) {
        for (int j = wid; j < J; j += W) {
            __syncwarp();
            const float ebf = (float)D.eta_bar[j];
            #pragma unroll 1
            for (int hr = 0; hr < NR; ++hr) {   // factors and weights, lanes over PFs
                const int s = lane + 32 * hr;
                float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
                float d = 0.f;
                if (s < S) {
                    const float* ph = phi + (size_t)s * 6 * P + p;
                    const size_t gi = ((size_t)s * J + j) * P + p;
                    const float4 g = D.geo[gi];
                    const float2 gl = D.geo_lo[gi];
                    const float gm = ph[3 * (size_t)P], mr = ph[4 * (size_t)P], mi = ph[5 * (size_t)P];
                    const float pi = (float)(D.zeta[s * J + j] * D.W[s]);
                    const float A = G.amp_c / (g.x + g.y);
                    float h, l;
                    ff_frac_mul2(g.x, g.y, G.inv_lam_hi, G.inv_lam_lo, h, l);
                    const float2 c = cispi_ff(-2.0f * h, -2.0f * l);
                    d = A * sqrtf(fmaxf(pi * (gm + (mr * mr + mi * mi) * (1.0f - pi)), 0.0f));
                    const float2 w0 = cmul(make_float2(A * pi * mr, A * pi * mi), c);
                    w = make_float4(-4.0f * w0.x, -4.0f * w0.y, 0.f, 0.f);
                    #pragma unroll 1
                    for (int f = 0; f < dm.Fh; ++f) {
                        const float2 b = freq_factor(G, g, f);
                        fx[s * pl.fp + f] = b.x;
                        fy[s * pl.fp + f] = b.y;
                    }
                    #pragma unroll 1
                    for (int q = 0; q < dm.hy + dm.hz; ++q) {
                        const bool y = q < dm.hy;
                        const int e = y ? q : q - dm.hy;
                        const float cc = y ? G.py_l[e] : G.pz_l[e], cl = y ? G.py_lo[e] : G.pz_lo[e];
                        const float u = y ? g.z : g.w, ul = y ? gl.x : gl.y;
                        const float t = __fmul_rn(cc, u);
                        ant[s * pl.ast + q] = cispi_ff(2.0f * t, 2.0f * fmaf(cc, ul, fmaf(cl, u, fmaf(cc, u, -t))));
                    }
                }
                if (s < 8 * NB) { ws[s] = w; dA[s] = d; }
            }
            __syncwarp();
            // a_y a_z of element ym of row s
            auto antenna = [&](int s, int iy, float sy, int iz, float sz) {
                float2 a = ant[s * pl.ast + iy], b = ant[s * pl.ast + iz];
                a.y *= sy;
                b.y *= sz;
                return cmul(a, b);
            };
            // e = z - sum_s w0_s u_s and |e|^2
            float ee = 0.f;
            for (int q0 = 0; q0 < dm.Nmh; q0 += NL) {
                const int ym = q0 + ly, y = min(ym, dm.Nmh - 1) / Mz, m = min(ym, dm.Nmh - 1) - y * Mz, ym2 = Nm - 1 - ym;
                const bool self = ym2 == ym, act = ym < dm.Nmh && first;
                bool cy, cz;
                const int iy = is_half(y, My, dm.hy, cy), iz = dm.hy + is_half(m, Mz, dm.hz, cz);
                const float sy = cy ? -1.0f : 1.0f, sz = cz ? -1.0f : 1.0f, sw = self ? 0.5f : 1.0f;
                for (int b0 = 0; b0 < np2; b0 += gf * IB_FP) {   // frequency pairs
                    const int g0 = min(b0 + fg * IB_FP, np2), nf = min(IB_FP, np2 - g0), fl = nf > 0 ? 2 * g0 : 0;
                    f2x a[IB_FP][IB_Q];
                    #pragma unroll
                    for (int i = 0; i < IB_FP; ++i) {
                        float v[2][IB_Q];
                        #pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            const int f = 2 * (g0 + i) + h;
                            #pragma unroll
                            for (int q = 0; q < IB_Q; ++q) v[h][q] = 0.f;
                            if (act && f < dm.Fh) {
                                auto obs = [&](int k) { return make_float2(z[2 * ((size_t)j * Nz + k)], z[2 * ((size_t)j * Nz + k) + 1]); };
                                const float2 z0 = obs(f * Nm + ym), z1 = obs(Nz - 1 - (f * Nm + ym));
                                const float2 P = make_float2(z0.x + z1.x, z0.y + z1.y), Q = make_float2(z0.x - z1.x, z0.y - z1.y);
                                float2 P2 = make_float2(0.f, 0.f), Q2 = P2;
                                if (!self) {
                                    const float2 z2 = obs(f * Nm + ym2), z3 = obs(Nz - 1 - (f * Nm + ym2));
                                    P2 = make_float2(z2.x + z3.x, z2.y + z3.y);
                                    Q2 = make_float2(z2.x - z3.x, z2.y - z3.y);
                                }
                                v[h][0] = P.x + P2.x;
                                v[h][2] = P.y + P2.y;
                                v[h][5] = Q.y + Q2.y;
                                v[h][7] = -(Q.x + Q2.x);
                                if (!self) {
                                    v[h][1] = Q.y - Q2.y;
                                    v[h][3] = Q2.x - Q.x;
                                    v[h][4] = P2.x - P.x;
                                    v[h][6] = P2.y - P.y;
                                }
                            }
                        }
                        #pragma unroll
                        for (int q = 0; q < IB_Q; ++q) a[i][q] = f2_pack(v[0][q], v[1][q]);
                    }
                    #pragma unroll 1
                    for (int s = sg; s < S; s += gs) {
                        float2 c = antenna(s, iy, sy, iz, sz);
                        const float2 w = *reinterpret_cast<const float2*>(ws + s);
                        c.x *= sw;
                        c.y *= sw;
                        const f2x t0 = f2_dup(w.x * c.x), t1 = f2_dup(w.y * c.x), t2 = f2_dup(w.x * c.y), t3 = f2_dup(w.y * c.y);
                        const float2 *bx = reinterpret_cast<const float2*>(fx + s * pl.fp + fl),
                                     *by = reinterpret_cast<const float2*>(fy + s * pl.fp + fl);
                        #pragma unroll
                        for (int i = 0; i < IB_FP; ++i) {
                            if (i < nf) {
                                const float2 xv = bx[i], yv = by[i];
                                const f2x x2 = f2_pack(xv.x, xv.y), y2 = f2_pack(yv.x, yv.y);
                                a[i][0] = f2_fma(t0, x2, a[i][0]);
                                a[i][1] = f2_fma(t2, x2, a[i][1]);
                                a[i][2] = f2_fma(t1, x2, a[i][2]);
                                a[i][3] = f2_fma(t3, x2, a[i][3]);
                                a[i][4] = f2_fma(t2, y2, a[i][4]);
                                a[i][5] = f2_fma(t0, y2, a[i][5]);
                                a[i][6] = f2_fma(t3, y2, a[i][6]);
                                a[i][7] = f2_fma(t1, y2, a[i][7]);
                            }
                        }
                    }
                    #pragma unroll
                    for (int i = 0; i < IB_FP; ++i) {
                        if (b0 + i >= np2) break;                 // uniform
                        f2x t[IB_Q];                              // the groups' shares (for the first group's lanes)
                        #pragma unroll
                        for (int q = 0; q < IB_Q; ++q) t[q] = a[i][q];
                        #pragma unroll 1
                        for (int g = 1; g < gs; ++g) {
                            #pragma unroll
                            for (int q = 0; q < IB_Q; ++q) t[q] = f2_add(t[q], __shfl_sync(0xffffffffu, a[i][q], lane + g * gf * NL));
                        }
                        const int f0 = 2 * (g0 + i);
                        if (act && i < nf) {
                            #pragma unroll
                            for (int q = 0; q < IB_Q; ++q) {
                                uint32_t u0, u1;
                                f2_unpack(t[q], u0, u1);
                                float v0 = __uint_as_float(u0), v1 = __uint_as_float(u1);
                                // the middle frequency holds both elements of a pair as one: half of each sum
                                if ((Nf & 1) && f0 == dm.Fh - 1) v0 *= 0.5f;
                                if ((Nf & 1) && f0 + 1 == dm.Fh - 1) v1 *= 0.5f;
                                if (f0 + 1 >= dm.Fh) v1 = 0.f;
                                const float g1 = self ? 0.5f : 0.25f;
                                ee = fmaf(((Nf & 1) && f0 == dm.Fh - 1 ? 2.0f : 1.0f) * g1 * v0, v0, ee);
                                ee = fmaf(((Nf & 1) && f0 + 1 == dm.Fh - 1 ? 2.0f : 1.0f) * g1 * v1, v1, ee);
                                *reinterpret_cast<float2*>(pq + (ym * IB_Q + q) * pl.f4 + f0) = make_float2(v0, v1);
                            }
                        }
                    }
                }
            }
            // (read below where the last pair is the first of four frequencies)
            if (2 * np2 < pl.f4)
                for (int i = lane; i < dm.Nmh * IB_Q; i += 32) *reinterpret_cast<float2*>(pq + i * pl.f4 + 2 * np2) = make_float2(0.f, 0.f);
            ee = warp_sum_f(ee);
            __syncwarp();
            // rhs_s = (dA)_s u_s^H e
            float2 rhs[NR];
            {
                float gr[NR], gi[NR];
                #pragma unroll
                for (int hr = 0; hr < NR; ++hr) gr[hr] = gi[hr] = 0.f;
                for (int f0 = 0; f0 < dm.Fh; f0 += 8) {
                    f2x xr[NR][4], xi[NR][4], yr[NR][4], yi[NR][4];
                    #pragma unroll
                    for (int hr = 0; hr < NR; ++hr)
                        #pragma unroll
                        for (int i = 0; i < 4; ++i) xr[hr][i] = xi[hr][i] = yr[hr][i] = yi[hr][i] = f2_dup(0.f);
                    const bool wide = f0 + 4 < dm.Fh, full = f0 + 6 < dm.Fh;   // uniform: the later frequencies of the eight
                    int y = 0, m = 0;
                    #pragma unroll 1
                    for (int ym = 0; ym < dm.Nmh; ++ym) {
                        bool cy, cz;
                        const int iy = is_half(y, My, dm.hy, cy), iz = dm.hy + is_half(m, Mz, dm.hz, cz);
                        const float sy = cy ? -1.0f : 1.0f, sz = cz ? -1.0f : 1.0f;
                        const float* e = pq + (size_t)ym * IB_Q * pl.f4 + f0;
                        f2x cx[NR], cyy[NR];
                        #pragma unroll
                        for (int hr = 0; hr < NR; ++hr) {
                            const float2 c = antenna(min(lane + 32 * hr, 8 * NB - 1), iy, sy, iz, sz);
                            cx[hr] = f2_dup(c.x);
                            cyy[hr] = f2_dup(c.y);
                        }
                        auto acc = [&](int i, int q, f2x (&o)[NR][4], const f2x (&c)[NR]) {   // two frequency pairs of one sum
                            const float4 v = *reinterpret_cast<const float4*>(e + q * pl.f4 + 2 * i);
                            #pragma unroll
                            for (int hr = 0; hr < NR; ++hr) {
                                o[hr][i] = f2_fma(c[hr], f2_pack(v.x, v.y), o[hr][i]);
                                if (i == 0 || full) o[hr][i + 1] = f2_fma(c[hr], f2_pack(v.z, v.w), o[hr][i + 1]);
                            }
                        };
                        #pragma unroll
                        for (int i = 0; i < 4; i += 2) {
                            if (i == 0 || wide) {
                                acc(i, 0, xr, cx);
                                acc(i, 1, xr, cyy);
                                acc(i, 2, xi, cx);
                                acc(i, 3, xi, cyy);
                                acc(i, 4, yr, cyy);
                                acc(i, 5, yr, cx);
                                acc(i, 6, yi, cyy);
                                acc(i, 7, yi, cx);
                            }
                        }
                        if (++m == Mz) { m = 0; ++y; }
                    }
                    #pragma unroll
                    for (int hr = 0; hr < NR; ++hr) {
                        const int s = min(lane + 32 * hr, 8 * NB - 1);
                        f2x r2 = f2_dup(0.f), i2 = r2;
                        #pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const float2 xv = *reinterpret_cast<const float2*>(fx + s * pl.fp + f0 + 2 * i);
                            const float2 yv = *reinterpret_cast<const float2*>(fy + s * pl.fp + f0 + 2 * i);
                            const f2x bx = f2_pack(xv.x, xv.y), by = f2_pack(yv.x, yv.y);
                            r2 = f2_fma(bx, xr[hr][i], f2_fma(by, yr[hr][i], r2));
                            i2 = f2_fma(bx, xi[hr][i], f2_fma(by, yi[hr][i], i2));
                        }
                        uint32_t r0, r1, i0, i1;
                        f2_unpack(r2, r0, r1);
                        f2_unpack(i2, i0, i1);
                        gr[hr] += __uint_as_float(r0) + __uint_as_float(r1);
                        gi[hr] += __uint_as_float(i0) + __uint_as_float(i1);
                    }
                }
                #pragma unroll
                for (int hr = 0; hr < NR; ++hr) {
                    const float d = dA[min(lane + 32 * hr, 8 * NB - 1)];
                    rhs[hr] = make_float2(d * gr[hr], d * gi[hr]);
                }
            }
            // Gram of this lane's entries: frequencies two at a time, then the antenna factors row block by row block
            float A[NSL];
            #pragma unroll
            for (int q = 0; q < NSL; ++q) A[q] = 0.f;
            #pragma unroll 1
            for (int g = 0; g < gp; ++g) {
                float2 rx[NB], ry[NB];
                #pragma unroll
                for (int ia = 0; ia < NB; ++ia) {
                    rx[ia] = *reinterpret_cast<const float2*>(fx + (8 * ia + tr) * pl.fp + 2 * g);
                    ry[ia] = *reinterpret_cast<const float2*>(fy + (8 * ia + tr) * pl.fp + 2 * g);
                }
                #pragma unroll
                for (int ib = 0; ib < 2 * NB; ++ib) {
                    const float2 cx = *reinterpret_cast<const float2*>(fx + (4 * ib + tc) * pl.fp + 2 * g);
                    const float2 cy = *reinterpret_cast<const float2*>(fy + (4 * ib + tc) * pl.fp + 2 * g);
                    #pragma unroll
                    for (int ia = ib / 2; ia < NB; ++ia) {
                        float& v = A[ia * (ia + 1) + ib];
                        v = fmaf(rx[ia].x, cx.x, fmaf(ry[ia].x, cy.x, fmaf(rx[ia].y, cx.y, fmaf(ry[ia].y, cy.y, v))));
                    }
                }
            }
            #pragma unroll
            for (int ia = 0; ia < NB; ++ia) {
                float sy[2 * NB], sz[2 * NB];
                #pragma unroll
                for (int ib = 0; ib <= 2 * ia + 1; ++ib) sy[ib] = sz[ib] = 0.f;
                const int a = 8 * ia + tr;
                const float2* ra = ant + a * pl.ast;
                const float2* rc = ant + tc * pl.ast;
                #pragma unroll 1
                for (int u = 0; u < My / 2; ++u) {
                    const float2 r = ra[u];
                    #pragma unroll
                    for (int ib = 0; ib <= 2 * ia + 1; ++ib) {
                        const float2 cb = rc[4 * ib * pl.ast + u];
                        sy[ib] = fmaf(r.x, cb.x, fmaf(r.y, cb.y, sy[ib]));
                    }
                }
                #pragma unroll 1
                for (int u = dm.hy; u < dm.hy + Mz / 2; ++u) {
                    const float2 r = ra[u];
                    #pragma unroll
                    for (int ib = 0; ib <= 2 * ia + 1; ++ib) {
                        const float2 cb = rc[4 * ib * pl.ast + u];
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
            // LDL^T elimination by panels of eight columns, with the forward substitution
            float yy = 0.f, pv[NR];
            #pragma unroll
            for (int hr = 0; hr < NR; ++hr) pv[hr] = 1.f;
            // (one copy of the panel's code for every panel: unrolled, instruction fetch set the time)
            #pragma unroll 1
            for (int K = 0; 8 * K < S; ++K) {
                __syncwarp();
                #pragma unroll
                for (int q = 0; q < NB; ++q) {
                    if (q == K) {
                        #pragma unroll
                        for (int ia = q; ia < NB; ++ia) {
                            pan[(8 * ia + tr) * IB_PST + tc] = A[ia * (ia + 1) + 2 * q];
                            pan[(8 * ia + tr) * IB_PST + 4 + tc] = A[ia * (ia + 1) + 2 * q + 1];
                        }
                    }
                }
                __syncwarp();
                float x[NR][8], ip[8];
                #pragma unroll
                for (int hr = 0; hr < NR; ++hr) {
                    const float4* r = reinterpret_cast<const float4*>(pan + min(lane + 32 * hr, 8 * NB - 1) * IB_PST);
                    const float4 v0 = r[0], v1 = r[1];
                    x[hr][0] = v0.x; x[hr][1] = v0.y; x[hr][2] = v0.z; x[hr][3] = v0.w;
                    x[hr][4] = v1.x; x[hr][5] = v1.y; x[hr][6] = v1.z; x[hr][7] = v1.w;
                }
                const bool up = NR > 1 && K >= 4;                   // row k = 8 K + c belongs to lane k % 32 of half k / 32
                const int ow = (8 * K) & 31;
                #pragma unroll
                for (int c = 0; c < 8; ++c) {
                    // (rows above k hold nothing that is used again)
                    const float xc = up ? x[NR - 1][c] : x[0][c];
                    const float2 rc = up ? rhs[NR - 1] : rhs[0];
                    const float piv = __shfl_sync(0xffffffffu, xc, ow + c);
                    ip[c] = __frcp_rn(piv);
                    const float2 rk = make_float2(__shfl_sync(0xffffffffu, rc.x, ow + c), __shfl_sync(0xffffffffu, rc.y, ow + c));
                    const float2 y = make_float2(rk.x * ip[c], rk.y * ip[c]);
                    yy = fmaf(rk.x, y.x, fmaf(rk.y, y.y, yy));
                    if (lane == ow + c) {
                        if (up) pv[NR - 1] = piv; else pv[0] = piv;
                    }
                    #pragma unroll
                    for (int c2 = c + 1; c2 < 8; ++c2) {
                        const float l = -ip[c] * __shfl_sync(0xffffffffu, xc, ow + c2);
                        #pragma unroll
                        for (int hr = 0; hr < NR; ++hr) x[hr][c2] = fmaf(x[hr][c], l, x[hr][c2]);
                    }
                    #pragma unroll
                    for (int hr = 0; hr < NR; ++hr) {
                        rhs[hr].x = fmaf(-x[hr][c], y.x, rhs[hr].x);
                        rhs[hr].y = fmaf(-x[hr][c], y.y, rhs[hr].y);
                    }
                }
                #pragma unroll
                for (int hr = 0; hr < NR; ++hr) {
                    if (lane + 32 * hr < 8 * NB) {
                        float4* r = reinterpret_cast<float4*>(pan + (lane + 32 * hr) * IB_PST);
                        r[0] = make_float4(x[hr][0], x[hr][1], x[hr][2], x[hr][3]);
                        r[1] = make_float4(x[hr][4], x[hr][5], x[hr][6], x[hr][7]);
                    }
                }
                __syncwarp();
                #pragma unroll
                for (int KK = 0; KK + 1 < NB; ++KK) {               // the rank-8 update, four columns at a time
                    if (KK != K) continue;
                    #pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        float4 rv[NB];
                        #pragma unroll
                        for (int ia = KK + 1; ia < NB; ++ia) {
                            const float4 v = *reinterpret_cast<const float4*>(pan + (8 * ia + tr) * IB_PST + 4 * q);
                            rv[ia] = make_float4(v.x * -ip[4 * q], v.y * -ip[4 * q + 1], v.z * -ip[4 * q + 2], v.w * -ip[4 * q + 3]);
                        }
                        #pragma unroll
                        for (int ib = 2 * (KK + 1); ib < 2 * NB; ++ib) {
                            const float4 cv = *reinterpret_cast<const float4*>(pan + (4 * ib + tc) * IB_PST + 4 * q);
                            #pragma unroll
                            for (int ia = ib / 2; ia < NB; ++ia) {
                                float& v = A[ia * (ia + 1) + ib];
                                v = fmaf(rv[ia].x, cv.x, fmaf(rv[ia].y, cv.y, fmaf(rv[ia].z, cv.z, fmaf(rv[ia].w, cv.w, v))));
                            }
                        }
                    }
                }
            }
            // log det, sum A_kk / piv_k, the smallest pivot
            float dm0 = 1.f, rsum = 0.f, pmin = 3.0e38f;
            int de = 0;
            #pragma unroll
            for (int hr = 0; hr < NR; ++hr) {
                const int k = lane + 32 * hr;
                if (k < S) {
                    int e;
                    dm0 = frexpf(dm0 * pv[hr], &e);
                    de += e;
                    rsum += fmaf(dA[k] * dA[k], (float)Nz, ebf) / pv[hr];
                    pmin = fminf(pmin, pv[hr]);
                }
            }
            #pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                int e;
                dm0 = frexpf(dm0 * __shfl_xor_sync(0xffffffffu, dm0, o), &e);
                de += __shfl_xor_sync(0xffffffffu, de, o) + e;
                rsum += __shfl_xor_sync(0xffffffffu, rsum, o);
                pmin = fminf(pmin, __shfl_xor_sync(0xffffffffu, pmin, o));
            }
            if (lane == 0) {
                const double ieb = ies[j], lgb = lgs[j];
                const double q = ((double)ee - (double)yy) * ieb;   // e^H C^-1 e
                const double logdet = log((double)dm0) + (double)de * 0.69314718055994530942;
                const double v = -q - logdet - (double)(Nz - S) * lgb - (double)Nz * IS_LOG_PI;
                const float eq = IB_ERR_PER_ENERGY * (float)(((double)ee + (double)yy) * ieb);
                part[par * 16 + j] = v;
                perr[par * 16 + j] = IB_ERR_PER_RATIO * rsum + eq;
                // every pivot of eta_bar I + D G D is at least eta_bar, and q >= 0: anything else is a
                // breakdown of the FP32 elimination
                pbad[par * 16 + j] = (!(pmin > 0.5f * ebf) || !(q > -(double)eq) || !isfinite(v)) ? 1.f : 0.f;
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
    const int per_sm = max(1, min(16 / W, (int)((limit + 1024) / (smem + 1024))));
    k_iota_bulk_sym<NB><<<min(Pm.P, sm_count() * per_sm * 4), 32 * W, smem, st>>>(G, Pm, D, S, z, W);
    return true;
}

// FP32 log iota~ with error bounds of every particle; false if the layout or the sizes do not allow it
bool launch_iota_bulk_sym(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, cudaStream_t st) {
    if (!G.sym) return false;
    if (S <= 32) return launch_bulk_sym_nb<4>(G, Pm, D, S, z, st);
    if (S <= 48) return launch_bulk_sym_nb<6>(G, Pm, D, S, z, st);
    return launch_bulk_sym_nb<8>(G, Pm, D, S, z, st);
}

// whether the real form applies: a symmetric layout whose working set fits one warp
bool iota_sym_ok(const DevGeom& G, int S) {
    return G.sym && if_fixed(G, S) + if_plan(G, S).warp <= 227 * 1024;
}

// float-float log iota~ of every particle (all), or of the queued ones
void launch_iota_ff(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const float* z, bool all, cudaStream_t st) {
    const size_t fixed = if_fixed(G, S), warp = if_plan(G, S).warp, limit = 227 * 1024;
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
