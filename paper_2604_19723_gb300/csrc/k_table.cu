// Message table and the particle-independent stage of the update.
//
// Table (Supplementary Sec. S-V; Proposition 1 terms mu^(3), mu^(4)), for
// every (s, j), with W = sum_p w_alpha, pi = zeta W:
//   m    = c_m sum_p w_beta sqrt(gamma + |mu|^2 (1 - pi)) psi_s^(j,p)
//   m^w  = c_w sum_p w_beta sqrt(gamma + |mu|^2 (1 - W))  psi_s^(j,p)
//   mu4  = W sum_p w_beta mu psi_s^(j,p),  mu3 = zeta mu4
// (c_m, c_w) = (W zeta, W) as printed in S-V, or their square roots.
// FP32 accumulation over runs of particles, float-float across them, FP64 across blocks.
//
// Stage per (s, j), FP64 (S-V "PF state update message", "PR state update
// message", S-VI): A_s = eta_bar I + M_{-s} M_{-s}^H is represented by a
// Cholesky-whitened basis V of M_{-s} (the inversion lemma of S-V with the small
// inverse factored), which with the null residual r0 = eta_bar A_s^-1 e0
// (e0 = z - sum_{s'!=s} mu3_s') is all the PF likelihood needs; the same forms give
// the PR existence test omega~(1)/omega~(0) -> p_s^(j) (eq. PR-normalization).
//
// nu (S-V "Noise variance update message"): G = M^H M is reduced once per j
// to a real symmetric tridiagonal T = Q^H G Q (Householder), with b = Q^H M^H e;
// each particle then needs O(S) work (k_like.cu).
#include "bp_internal.cuh"
#include "bp_kernels.cuh"
#include "per_device.cuh"

namespace bp {

// ---------------------------------------------------------------- table reduction
// grid (nsplit, S, J x element blocks).  A chunk of particles is staged in shared memory (thread per
// particle: frequency and antenna factors, the three weighted amplitudes with the carrier), then
// every thread accumulates two elements over its group's share of the chunk.  With u_k = x + i y the
// unit-modulus element and c the complex weight, the four real sums of c_r and c_i with x and y
// give both sum_p c u_k and, on a layout symmetric about 0 (u_{Nz-1-k} = conj(u_k)), the
// mirrored element's sum_p c conj(u_k): half the elements are formed.  (x, y) travel as packed FP32
// pairs; FP32 accumulation over runs of TABLE_FLUSH particles, float-float across.
// Bound: FP32 issue and shared-memory reads (16 instructions per element pair and particle).
// Measured (message-table stage, with k_geom): 32 PFs x 262144, Nz = 1024: 92.9 -> 18.4 ms; 64 x 1e5,
// Nz = 160: 8.3 -> 3.4; 40 x 8192, Nz = 300: 2.3 -> 0.44; 10 x 30000: 0.49 -> 0.21 (against a thread
// per element with three complex products and FP64 sums every 64 particles).
constexpr int TABLE_FLUSH = 64;
struct TablePlan { int nel, nb, na, nt, ntb, nblk, threads, chunk; size_t smem; };
static __host__ __device__ inline TablePlan table_plan(const DevGeom& G, int chunk_req) {
    TablePlan t;
    t.nel = G.sym ? (G.Nz + 1) / 2 : G.Nz;
    t.na = G.My * G.Mz;
    t.nb = (t.nel - 1) / t.na + 1;                    // frequencies of the formed elements
    t.nt = (t.nel + 1) / 2;                           // element pairs
    t.threads = t.nt <= 128 ? 128 : 256;
    t.nblk = (t.nt + t.threads - 1) / t.threads;
    t.ntb = (t.nt + t.nblk - 1) / t.nblk;             // pairs per block
    const size_t row = (size_t)((t.nb + t.na) | 1) * sizeof(float2) + 3 * sizeof(float4);
    t.chunk = (chunk_req == 16 || chunk_req == 32 || chunk_req == 64) ? chunk_req : 128;
    while (t.chunk > 16 && t.chunk * row > 100 * 1024) t.chunk /= 2;
    const size_t stage = t.chunk * row, out = (size_t)t.threads * 24 * sizeof(double);
    t.smem = (stage > out ? stage : out) + 16;
    return t;
}

__global__ void __launch_bounds__(256, 2) k_table(DevGeom G, DevParams Pm, DevState D, int S, int nsplit, int chunk_req) {
    extern __shared__ float4 sm[];
    const TablePlan tp = table_plan(G, chunk_req);
    const int split = blockIdx.x, s = blockIdx.y, j = blockIdx.z / tp.nblk, eb = blockIdx.z - j * tp.nblk;
    const int P = Pm.P, J = G.J, My = G.My, Mz = G.Mz, Nm = My * Mz, Nz = G.Nz;
    const int per = (P + nsplit - 1) / nsplit;
    const int p0 = split * per, p1 = min(P, p0 + per);
    const int tid = threadIdx.x, stride = (tp.nb + tp.na) | 1;   // odd row stride (bank spread)
    float4* cf = sm;                                             // [chunk][3] weights (c_r, c_r, c_i, c_i)
    float2* rows = reinterpret_cast<float2*>(sm + 3 * (size_t)tp.chunk);   // [chunk][stride] b_f, a_y a_z
    // this thread's elements tile and tile + ntb of the block's 2 ntb, and its group of particles
    const int ngrp = tp.threads / tp.ntb, grp = tid / tp.ntb, tile = tid - grp * tp.ntb;
    int ob[2], oa[2];
    #pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int k = min(eb * 2 * tp.ntb + tile + e * tp.ntb, tp.nel - 1), f = k / Nm;
        ob[e] = f;
        oa[e] = tp.nb + (k - f * Nm);
    }
    const float pi = (float)(D.zeta[s * J + j] * D.W[s]);
    const float pd = (float)(1.0 - D.W[s]);
    const float* ph = D.phi[D.cur] + (size_t)s * 6 * P;
    const float4* geo = D.geo + ((size_t)s * J + j) * P;
    const float2* geol = D.geo_lo + ((size_t)s * J + j) * P;
    f2x acc[2][6], hi[2][6], lo[2][6];
    #pragma unroll
    for (int e = 0; e < 2; ++e)
        #pragma unroll
        for (int i = 0; i < 6; ++i) acc[e][i] = hi[e][i] = lo[e][i] = f2_dup(0.f);
    int held = 0;                                                // particles in acc
    auto flush = [&]() {
        #pragma unroll
        for (int e = 0; e < 2; ++e)
            #pragma unroll
            for (int i = 0; i < 6; ++i) {                        // two_sum
                const f2x a = hi[e][i], b = acc[e][i], t = f2_add(a, b), bb = f2_sub(t, a);
                lo[e][i] = f2_add(lo[e][i], f2_add(f2_sub(a, f2_sub(t, bb)), f2_sub(b, bb)));
                hi[e][i] = t;
                acc[e][i] = f2_dup(0.f);
            }
        held = 0;
    };
    for (int c0 = p0; c0 < p1; c0 += tp.chunk) {
        const int cn = min(tp.chunk, p1 - c0);
        __syncthreads();
        for (int t = tid; t < cn; t += tp.threads) {
            const int p = c0 + t;
            const float4 g = geo[p];
            const float2 gl = geol[p], c = carrier_factor(G, g);
            float2* b = rows + (size_t)t * stride;
            float2* a = b + tp.nb;
            for (int f = 0; f < tp.nb; ++f) b[f] = freq_factor(G, g, f);
            auto factor = [&](float c, float cl, float u, float ul) {
                const float h = __fmul_rn(c, u);
                return cispi_ff(2.0f * h, 2.0f * fmaf(c, ul, fmaf(cl, u, fmaf(c, u, -h))));
            };
            // a_z into the row's first Mz places, then the products of each a_y from the last y down
            for (int m = 0; m < Mz; ++m) a[m] = factor(G.pz_l[m], G.pz_lo[m], g.w, gl.y);
            for (int y = My - 1; y >= 0; --y) {
                const float2 ay = factor(G.py_l[y], G.py_lo[y], g.z, gl.x);
                for (int m = 0; m < Mz; ++m) a[y * Mz + m] = cmul(ay, a[m]);
            }
            const float gm = ph[3 * (size_t)P + p], mr = ph[4 * (size_t)P + p], mi = ph[5 * (size_t)P + p];
            const float m2 = mr * mr + mi * mi;
            const float wb = (float)D.w_x[p];
            const float ca = wb * sqrtf(fmaxf(gm + m2 * (1.0f - pi), 0.0f));
            const float cb = wb * sqrtf(fmaxf(gm + m2 * pd, 0.0f));
            const float2 c3 = cmul(make_float2(wb * mr, wb * mi), c);
            cf[3 * t] = make_float4(ca * c.x, ca * c.x, ca * c.y, ca * c.y);
            cf[3 * t + 1] = make_float4(cb * c.x, cb * c.x, cb * c.y, cb * c.y);
            cf[3 * t + 2] = make_float4(c3.x, c3.x, c3.y, c3.y);
        }
        __syncthreads();
        if (grp < ngrp) {
            for (int t = grp; t < cn; t += ngrp) {
                const float2* row = rows + (size_t)t * stride;
                f2x w[6];
                #pragma unroll
                for (int i = 0; i < 3; ++i) {
                    const float4 c = cf[3 * t + i];
                    w[2 * i] = f2_pack(c.x, c.y);
                    w[2 * i + 1] = f2_pack(c.z, c.w);
                }
                #pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float2 b = row[ob[e]], a = row[oa[e]];
                    const f2x u = f2_pack(fmaf(b.x, a.x, -b.y * a.y), fmaf(b.x, a.y, b.y * a.x));
                    #pragma unroll
                    for (int i = 0; i < 6; ++i) acc[e][i] = f2_fma(w[i], u, acc[e][i]);
                }
                if (++held == TABLE_FLUSH) flush();
            }
        }
    }
    flush();
    __syncthreads();
    // the groups' sums in a fixed order; per element and weight (sum c_r x, sum c_r y), (sum c_i x, sum c_i y)
    double* out = reinterpret_cast<double*>(sm);                 // [ngrp][2 ntb][12]
    if (grp < ngrp) {
        #pragma unroll
        for (int e = 0; e < 2; ++e)
            #pragma unroll
            for (int i = 0; i < 6; ++i) {
                uint32_t h0, h1, l0, l1;
                f2_unpack(hi[e][i], h0, h1);
                f2_unpack(lo[e][i], l0, l1);
                double* o = out + ((size_t)grp * 2 * tp.ntb + tile + e * tp.ntb) * 12 + 2 * i;
                o[0] = (double)__uint_as_float(h0) + (double)__uint_as_float(l0);
                o[1] = (double)__uint_as_float(h1) + (double)__uint_as_float(l1);
            }
    }
    __syncthreads();
    const int SJ = Pm.S_max * J;
    for (int t = tid; t < 2 * tp.ntb * 3; t += tp.threads) {
        const int i = t / (2 * tp.ntb), el = t - i * 2 * tp.ntb, k = eb * 2 * tp.ntb + el;
        if (k >= tp.nel) continue;
        double r[4] = {0.0, 0.0, 0.0, 0.0};
        for (int g = 0; g < ngrp; ++g)
            #pragma unroll
            for (int q = 0; q < 4; ++q) r[q] += out[((size_t)g * 2 * tp.ntb + el) * 12 + 4 * i + q];
        double2* o = reinterpret_cast<double2*>(D.tab_part) + (((size_t)split * 3 + i) * SJ + (size_t)s * J + j) * Nz;
        o[k] = make_double2(r[0] - r[3], r[1] + r[2]);
        if (G.sym && k != Nz - 1 - k) o[Nz - 1 - k] = make_double2(r[0] + r[3], r[2] - r[1]);
    }
}

// sums the partials in fixed order and applies the existence scale factors (thread per element and weight)
__global__ void k_table_final(DevGeom G, DevParams Pm, DevState D, int S, int nsplit) {
    const int J = G.J, Nz = G.Nz;
    const int SJ = Pm.S_max * J, n = S * J * Nz;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= 3 * n) return;
    const int i = idx / n, el = idx - i * n;
    const int k = el % Nz, sj = el / Nz;
    const int s = sj / J, j = sj - s * J;
    const double W = D.W[s], zeta = D.zeta[s * J + j];
    const double2* part = reinterpret_cast<const double2*>(D.tab_part) + ((size_t)i * SJ + (size_t)s * J + j) * Nz + k;
    const size_t step = (size_t)3 * SJ * Nz;
    double2 a = make_double2(0.0, 0.0);
    #pragma unroll 8
    for (int sp = 0; sp < nsplit; ++sp) {
        const double2 t = part[sp * step];
        a.x += t.x; a.y += t.y;
    }
    double2* tab = reinterpret_cast<double2*>(D.tab);
    const size_t o = ((size_t)s * J + j) * Nz + k;
    const size_t plane = (size_t)SJ * Nz;
    if (i == 2) {
        const double2 m4 = make_double2(W * a.x, W * a.y);
        tab[3 * plane + o] = m4;
        tab[2 * plane + o] = make_double2(zeta * m4.x, zeta * m4.y);
    } else {
        double c = i == 0 ? W * zeta : W;
        if (Pm.mvec_scaling != 0) c = sqrt(c);
        tab[i * plane + o] = make_double2(c * a.x, c * a.y);
    }
}

// ---------------------------------------------------------------- Gram matrix per j (FP64)
// G_j[a][b] = m_a^H m_b, a warp per pair.
__global__ void k_gram(DevGeom G, DevParams Pm, DevState D, int S, double* gram) {
    const int j = blockIdx.y;
    const int J = G.J, Nz = G.Nz, SM = Pm.S_max;
    const double2* tab = reinterpret_cast<const double2*>(D.tab);
    const int npair = S * (S + 1) / 2;            // pairs (a >= b)
    const int warps = blockDim.x / 32, lane = threadIdx.x & 31;
    for (int task = blockIdx.x * warps + (threadIdx.x >> 5); task < npair; task += gridDim.x * warps) {
        double2 acc = make_double2(0.0, 0.0);
        int a = (int)((sqrtf(8.0f * task + 1.0f) - 1.0f) * 0.5f);
        while ((a + 1) * (a + 2) / 2 <= task) ++a;
        while (a * (a + 1) / 2 > task) --a;
        const int b = task - a * (a + 1) / 2;
        const double2* ma = tab + ((size_t)a * J + j) * Nz;
        const double2* mb = tab + ((size_t)b * J + j) * Nz;
        #pragma unroll 4
        for (int k = lane; k < Nz; k += 32) {
            acc = zfmac(ma[k], mb[k], acc);
        }
        acc.x = warp_sum_d(acc.x); acc.y = warp_sum_d(acc.y);
        if (lane == 0) {
            double2* Gm = reinterpret_cast<double2*>(gram) + (size_t)j * SM * SM;
            Gm[a * SM + b] = acc;
            Gm[b * SM + a] = make_double2(acc.x, -acc.y);
        }
    }
}

// ---------------------------------------------------------------- kappa / omega stage per (s, j), FP64
// With B = I + M_{-s}^H M_{-s}/eta_bar = L L^H (Cholesky) the whitened basis V = M_{-s} L^{-H} satisfies
// V V^H = M_{-s} B^{-1} M_{-s}^H, so the inversion lemma gives
// a^H A_s^{-1} b = (a^H b - (V^H a)^H (V^H b)/eta_bar)/eta_bar for every form of S-V, and
// r0 = eta_bar A_s^{-1} e0 = e0 - V V^H e0/eta_bar.  V and r0 leave as columns of V64
// [S][J][SCA][Nz] (r0 in column SCA - 1) for k_kappa_digits.
// One factorisation per PA serves every PF: with all S columns B = L L^H and V_f = M L^{-H}.  Without row s
// L is a triangle with one superdiagonal from row s on, which the unitary Q of K - s plane rotations
// of neighbouring columns removes: (L without row s) Q = [L_s 0], and V_s = V_f Q without its last
// column (the same basis that a factorisation of its own would give, at 12 operations per element
// and rotation instead of K^2/2 products).  x^H V_s is x^H V_f under the same rotations.
// Bound: the FP64 pipe (2 FMA per clock and SM) and the serial chains of pivots and rotations.
// Measured, 4 PAs: 64 PFs x Nz = 160 1.74 -> 0.46 ms (with the Gram), 40 x 300 1.50 -> 0.34, 32 x 1024
// 1.54 -> 0.40, 8 x 160 0.070 -> 0.066 (against a factorisation and a solve for every (s, j)).
constexpr int STAGE_THREADS = 256;
constexpr int STAGE_WRED = 12;  // per-warp partial sums: the omega test's nine scalars, m^H e_all and |e_all|^2
__host__ __device__ inline int stage_row(int K, int r) {   // start of row r of [L; carried rows of K]
    return r < K ? r * (r + 1) / 2 : K * (K + 1) / 2 + (r - K) * K;
}
// behind the Gram matrices [J][S_max][S_max]: V_f [J][S_max][Nz], e_all [J][Nz], L [J][S_max (S_max + 1)/2]
struct StageWs { double2 *Vf, *e, *L; };
__host__ __device__ inline StageWs stage_ws(double* gram, int J, int SM, int Nz) {
    StageWs w;
    w.Vf = reinterpret_cast<double2*>(gram) + (size_t)J * SM * SM;
    w.e = w.Vf + (size_t)J * SM * Nz;
    w.L = w.e + (size_t)J * Nz;
    return w;
}
size_t stage_ws_bytes(int J, int SM, int Nz) {
    return ((size_t)J * SM * SM + (size_t)J * SM * Nz + (size_t)J * Nz + (size_t)J * SM * (SM + 1) / 2) * sizeof(double2);
}

// Block (j, EC elements): B, and the EC rows of M as rows S .. S + EC - 1 of a right-looking Cholesky that
// carries them along: they leave as rows of V_f.  Every block repeats the factorisation (S^3/6 products: 46
// us of FP64 at 64 PFs, in parallel on as many SMs); e_all = z - sum_t mu3_t of its elements on the way.
__global__ void __launch_bounds__(STAGE_THREADS) k_stage_basis(DevGeom G, DevParams Pm, DevState D, int S, int EC, const float* z,
                                                               double* gram) {
    const int j = blockIdx.x, k0 = blockIdx.y * EC;
    const int J = G.J, Nz = G.Nz, SM = Pm.S_max, ne = min(EC, Nz - k0);
    const double eb = D.eta_bar[j];
    const size_t plane = (size_t)SM * J * Nz;
    const double2* tab = reinterpret_cast<const double2*>(D.tab);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = STAGE_THREADS / 32;
    extern __shared__ double2 sh[];
    double2* Lp = sh;                             // packed lower triangle, then ne rows of S
    double* il = reinterpret_cast<double*>(Lp + stage_row(S, S + EC));   // 1 / L_cc
    const double2* Gm = reinterpret_cast<const double2*>(gram) + (size_t)j * SM * SM;
    const StageWs ws = stage_ws(gram, J, SM, Nz);
    for (int r = wid; r < S; r += nw)
        for (int c = lane; c <= r; c += 32) {
            double2 g = Gm[r * SM + c];
            g.x /= eb; g.y /= eb;
            if (r == c) { g.x += 1.0; g.y = 0.0; }
            Lp[stage_row(S, r) + c] = g;
        }
    for (int i = tid; i < S * ne; i += STAGE_THREADS) {
        const int c = i / ne, e = i - c * ne;
        Lp[stage_row(S, S + e) + c] = tab[((size_t)c * J + j) * Nz + k0 + e];
    }
    for (int e = tid; e < ne; e += STAGE_THREADS) {
        const int k = k0 + e;
        double2 v = make_double2((double)z[2 * (j * Nz + k)], (double)z[2 * (j * Nz + k) + 1]);
        for (int t = 0; t < S; ++t) {
            const double2 m3 = tab[2 * plane + ((size_t)t * J + j) * Nz + k];
            v.x -= m3.x; v.y -= m3.y;
        }
        ws.e[(size_t)j * Nz + k] = v;
    }
    __syncthreads();
    // Columns stay unscaled (x_rk = l_rk l_kk), so a step is one pass and one barrier: v_rc -= x_rk conj(x_ck) / p_k;
    // whoever updates the next pivot inverts it.  Every pivot of B is at least 1.
    if (tid == 0) il[0] = 1.0 / fmax(Lp[0].x, 1.0);
    __syncthreads();
    for (int k = 0; k + 1 < S; ++k) {
        const double ip = il[k];
        for (int r = k + 1 + (tid >> 4); r < S + ne; r += STAGE_THREADS / 16) {
            const int row = stage_row(S, r), end = min(r, S - 1);
            double2 x = Lp[row + k];
            x.x *= -ip; x.y *= -ip;
            for (int c = k + 1 + (tid & 15); c <= end; c += 16) {
                double2& v = Lp[row + c];
                v = zfmac(Lp[stage_row(S, c) + k], x, v);
                if (r == k + 1 && c == r) il[r] = 1.0 / fmax(v.x, 1.0);
            }
        }
        __syncthreads();
    }
    for (int c = tid; c < S; c += STAGE_THREADS) il[c] = rsqrt(fmax(Lp[stage_row(S, c) + c].x, 1.0));
    __syncthreads();
    for (int i = tid; i < S * ne; i += STAGE_THREADS) {
        const int c = i / ne, e = i - c * ne;
        const double2 v = Lp[stage_row(S, S + e) + c];
        ws.Vf[((size_t)j * SM + c) * Nz + k0 + e] = make_double2(v.x * il[c], v.y * il[c]);
    }
    if (blockIdx.y == 0) {
        double2* Lg = ws.L + (size_t)j * (SM * (SM + 1) / 2);
        for (int r = wid; r < S; r += nw)
            for (int c = lane; c <= r; c += 32) {
                const double2 v = Lp[stage_row(S, r) + c];
                Lg[stage_row(S, r) + c] = r == c ? make_double2(fmax(v.x, 1.0) * il[r], 0.0) : make_double2(v.x * il[c], v.y * il[c]);
            }
    }
}

__host__ __device__ inline size_t stage_kappa_smem(int S, int Nz) {
    return ((size_t)S * (S + 1) / 2 + 4 * (size_t)S + (size_t)Nz) * sizeof(double2) +
           ((size_t)S + STAGE_WRED * (STAGE_THREADS / 32)) * sizeof(double);
}
__global__ void __launch_bounds__(STAGE_THREADS) k_stage_kappa(DevGeom G, DevParams Pm, DevState D, int S, int SCA,
                                                                  double* gram, double* nu_b, double* V64) {
    const int s = blockIdx.x, j = blockIdx.y;
    const int J = G.J, Nz = G.Nz, SM = Pm.S_max;
    const int K = S - 1;                          // columns of M_{-s}
    const double eb = D.eta_bar[j];
    const size_t plane = (size_t)SM * J * Nz;
    const double2* tab = reinterpret_cast<const double2*>(D.tab);
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, nw = STAGE_THREADS / 32;
    extern __shared__ double2 sh[];
    double2* Lp = sh;                             // packed lower triangle of all PFs
    double2* cr = Lp + stage_row(S, S);           // [3][S] x^H V_f, then x^H V_s, of x = e0, m^w, mu4
    double2* qa = cr + 3 * S;                     // rotation of columns (i, i + 1), i = s .. K - 1: (a, b)
    double2* E0 = qa + S;                         // e0 = z - sum_{t != s} mu3_t (Nz)
    double* qb = reinterpret_cast<double*>(E0 + Nz);
    double* wred = qb + S;                        // [STAGE_WRED][nw]
    const StageWs ws = stage_ws(gram, J, SM, Nz);
    const double2* Vf = ws.Vf + (size_t)j * SM * Nz;
    const double2* mp = tab + ((size_t)s * J + j) * Nz;
    const double2* mwp = tab + 1 * plane + ((size_t)s * J + j) * Nz;
    const double2* m3p = tab + 2 * plane + ((size_t)s * J + j) * Nz;
    const double2* m4p = tab + 3 * plane + ((size_t)s * J + j) * Nz;
    {
        const double2* Lg = ws.L + (size_t)j * (SM * (SM + 1) / 2);
        for (int i = stage_row(S, s) + tid; i < S * (S + 1) / 2; i += STAGE_THREADS) Lp[i] = Lg[i];
    }
    // e0 and the block sums of |e0|^2, m^H e0, |m|^2, mu4^H e0, |mu4|^2, m^H mu4 (m = m^w_s)
    {
        double acc[STAGE_WRED] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
        for (int k = tid; k < Nz; k += STAGE_THREADS) {
            const double2 ea = ws.e[(size_t)j * Nz + k], m3 = m3p[k];
            const double2 e0 = make_double2(ea.x + m3.x, ea.y + m3.y);
            E0[k] = e0;
            const double2 mw = mwp[k], m4 = m4p[k];
            const double2 me = zmulc(mw, e0), ue = zmulc(m4, e0), mu = zmulc(mw, m4);
            acc[0] += e0.x * e0.x + e0.y * e0.y;
            acc[1] += me.x; acc[2] += me.y;
            acc[3] += mw.x * mw.x + mw.y * mw.y;
            acc[4] += ue.x; acc[5] += ue.y;
            acc[6] += m4.x * m4.x + m4.y * m4.y;
            acc[7] += mu.x; acc[8] += mu.y;
            const double2 be = zmulc(mp[k], ea);
            acc[9] += be.x; acc[10] += be.y;
            acc[11] += ea.x * ea.x + ea.y * ea.y;
        }
        #pragma unroll
        for (int q = 0; q < STAGE_WRED; ++q) {
            const double v = warp_sum_d(acc[q]);
            if (lane == 0) wred[q * nw + wid] = v;
        }
    }
    __syncthreads();
    if (wid == 0) {
        // the rotations: lanes over the rows i >= s of L without row s (row i was i + 1), t the entry of the
        // column that travels.  [t_i, L_{i+1,i+1}] -> [rho, 0] with (a, b) = (t_i, L_{i+1,i+1}) / rho:
        // (x_i, x_{i+1}) -> (x_i conj(a) + x_{i+1} b, x_{i+1} a - x_i b)
        double2 t[2];
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = s + lane + 32 * h;
            t[h] = i < K ? Lp[stage_row(S, i + 1) + s] : make_double2(0.0, 0.0);
        }
        for (int c = s; c < K; ++c) {
            const int o = c - s;
            const double2 own = o < 32 ? t[0] : t[1];
            double2 a = make_double2(__shfl_sync(0xffffffffu, own.x, o & 31), __shfl_sync(0xffffffffu, own.y, o & 31));
            double b = Lp[stage_row(S, c + 1) + c + 1].x;
            const double ir = rsqrt(fma(a.x, a.x, fma(a.y, a.y, b * b)));
            a.x *= ir; a.y *= ir; b *= ir;
            if (lane == 0) { qa[c] = a; qb[c] = b; }
            #pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = s + lane + 32 * h;
                if (i > c && i < K) {
                    const double2 x = Lp[stage_row(S, i + 1) + c + 1], u = zmul(x, a);
                    t[h] = make_double2(fma(-b, t[h].x, u.x), fma(-b, t[h].y, u.y));
                }
            }
        }
    } else {
        for (int t = wid - 1; t < S; t += nw - 1) {   // one warp per column of V_f
            const double2* vt = Vf + (size_t)t * Nz;
            double2 x0 = make_double2(0.0, 0.0), x1 = x0, x2 = x0;
            #pragma unroll 4
            for (int k = lane; k < Nz; k += 32) {
                const double2 v = vt[k];
                x0 = zfmac(v, E0[k], x0);
                x1 = zfmac(v, mwp[k], x1);
                x2 = zfmac(v, m4p[k], x2);
            }
            x0 = make_double2(warp_sum_d(x0.x), warp_sum_d(x0.y));
            x1 = make_double2(warp_sum_d(x1.x), warp_sum_d(x1.y));
            x2 = make_double2(warp_sum_d(x2.x), warp_sum_d(x2.y));
            if (lane == 0) {
                cr[t] = make_double2(x0.x, -x0.y);
                cr[S + t] = make_double2(x1.x, -x1.y);
                cr[2 * S + t] = make_double2(x2.x, -x2.y);
            }
        }
    }
    __syncthreads();
    if (tid < 3) {
        double2* c = cr + tid * S;
        double2 t = c[s];
        for (int i = s; i < K; ++i) {
            const double2 x = c[i + 1], a = qa[i], u = zmulc(a, t), w = zmul(x, a);
            const double b = qb[i];
            c[i] = make_double2(fma(b, x.x, u.x), fma(b, x.y, u.y));
            t = make_double2(fma(-b, t.x, w.x), fma(-b, t.y, w.y));
        }
    }
    if (tid >= 32 && tid < 32 + STAGE_WRED) {
        double v = 0.0;
        for (int w = 0; w < nw; ++w) v += wred[(tid - 32) * nw + w];
        wred[(tid - 32) * nw] = v;   // the block sum in slot 0
        // the noise likelihood's b = M^H e_all, |e_all|^2
        double* nb = nu_b + 2 * (size_t)j * (SM + 1);
        if (tid - 32 == 9 || tid - 32 == 10) nb[2 * s + tid - 41] = v;
        if (s == 0 && tid - 32 == 11) { nb[2 * SM] = v; nb[2 * SM + 1] = 0.0; }
    }
    __syncthreads();
    const double2* ye = cr;                       // conj of V^H e0, V^H m^w, V^H mu4
    const double2* vm = cr + S;
    const double2* v4 = cr + 2 * S;
    if (wid == 0) {
        double a[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
        for (int c = lane; c < K; c += 32) {
            const double2 e = make_double2(ye[c].x, -ye[c].y), b = make_double2(vm[c].x, -vm[c].y),
                          u = make_double2(v4[c].x, -v4[c].y);
            const double2 t1 = zmulc(b, e), t2 = zmulc(u, e), t3 = zmulc(b, u);
            a[0] += e.x * e.x + e.y * e.y;
            a[1] += t1.x; a[2] += t1.y;
            a[3] += b.x * b.x + b.y * b.y;
            a[4] += t2.x;
            a[6] += u.x * u.x + u.y * u.y;
            a[7] += t3.x; a[8] += t3.y;
        }
        #pragma unroll
        for (int q = 0; q < 9; ++q) a[q] = (wred[q * nw] - warp_sum_d(a[q]) / eb) / eb;   // forms x^H A^-1 y
        if (lane == 0) {
            // e0^H A^-1 e0, and with e1 = e0 - mu4: e1^H A^-1 e1
            const double Q00 = a[0], Q11 = a[0] - 2.0 * a[4] + a[6];
            // m^H A^-1 m >= 0 (A positive definite); a negative value is cancellation
            // rounding of a PF whose m-vector lies in the span of the others: clamp it
            const double mAm = fmax(a[3], 0.0);
            // m^H A^-1 e1 = m^H A^-1 e0 - m^H A^-1 mu4
            const double2 mAe1 = make_double2(a[1] - a[7], a[2] - a[8]);
            const double llr = (mAe1.x * mAe1.x + mAe1.y * mAe1.y) / (1.0 + mAm) - Q11 + Q00 - log1p(mAm);
            D.llr_w[s * J + j] = llr;
            const double zeta = D.zeta[s * J + j];
            double pr;
            if (zeta >= 1.0) pr = 1.0;
            else if (zeta <= 0.0) pr = 0.0;
            else {
                const double u = log(zeta) - log1p(-zeta) + llr;
                pr = (u >= 0) ? 1.0 / (1.0 + exp(-u)) : exp(u) / (1.0 + exp(u));
            }
            D.bel[BEL_PPR + s * J + j] = pr;
        }
    }
    // columns of V_s: those before s are V_f's, the others rotated; r0 on the way
    double2* Vs = reinterpret_cast<double2*>(V64) + ((size_t)s * J + j) * SCA * Nz;
    const double ieb = 1.0 / eb;
    for (int k = tid; k < Nz; k += STAGE_THREADS) {
        double2 r0 = make_double2(0.0, 0.0);
        auto put = [&](int c, double2 v) {
            Vs[(size_t)c * Nz + k] = v;
            r0 = zfmac(ye[c], v, r0);             // v (V^H e0)_c
        };
        #pragma unroll 4
        for (int c = 0; c < s; ++c) put(c, Vf[(size_t)c * Nz + k]);
        double2 t = Vf[(size_t)s * Nz + k];
        #pragma unroll 4
        for (int c = s; c < K; ++c) {
            const double2 x = Vf[(size_t)(c + 1) * Nz + k], a = qa[c], u = zmulc(a, t), w = zmul(x, a);
            const double b = qb[c];
            put(c, make_double2(fma(b, x.x, u.x), fma(b, x.y, u.y)));
            t = make_double2(fma(-b, t.x, w.x), fma(-b, t.y, w.y));
        }
        const double2 e0 = E0[k];
        Vs[(size_t)(SCA - 1) * Nz + k] = make_double2(fma(-ieb, r0.x, e0.x), fma(-ieb, r0.y, e0.y));
    }
}

// ---------------------------------------------------------------- nu: Householder tridiagonalisation per j (FP64)
// T = Q^H G Q real symmetric tridiagonal, b' = Q^H b with b = M^H e_all; the
// off-diagonal phases are moved into b' so that T has non-negative off-diagonals.
// Block of 128 threads per j.  A step has one chain of square roots and divisions (the Householder vector v
// stays unnormalised: H = I - beta v v^H, beta = 1 / (|x| (|x| + |x_0|))); its two rounds of sums over the column
// are taken by every warp for itself (lane i the rows i and i + 32 of the trailing block), so a step
// has four barriers.  Only the lower triangle is kept.  Bound: latency (J blocks).
// Measured: 64 PFs 1269 -> 805 us, 8 PFs 58 -> 37 us (against block-wide sums, normalised vectors and the
// whole matrix).
constexpr int NU_THREADS = 128;
__global__ void __launch_bounds__(NU_THREADS) k_nu_tridiag(DevParams Pm, DevState D, int S, const double* gram, const double* nu_b) {
    const int j = blockIdx.x;
    const int SM = Pm.S_max;
    extern __shared__ double2 sh[];
    double2* A = sh;                 // S x S, rows of S, lower triangle
    double2* v = A + (size_t)S * S;  // S
    double2* pv = v + S;             // S: p = beta A v, then w
    double2* b = pv + S;             // S
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const double2* Gm = reinterpret_cast<const double2*>(gram) + (size_t)j * SM * SM;
    const double2* bv = reinterpret_cast<const double2*>(nu_b) + (size_t)j * (SM + 1);
    for (int t = tid; t < S * S; t += NU_THREADS) A[t] = Gm[(t / S) * SM + (t % S)];
    for (int t = tid; t < S; t += NU_THREADS) b[t] = bv[t];
    __syncthreads();
    for (int k = 0; k + 2 < S; ++k) {
        const int n = S - k - 1, f = k + 1;       // trailing rows f .. S - 1
        // x = A[f:, k], scaled by a power of two to a largest part in [1, 2) so that its squares stay in range
        // (products of small existence weights do not); alpha = -ph |x| with ph the phase of x_0; v = x - alpha e1
        double2 x[2];
        uint32_t top = 0;                         // upper words of the magnitudes
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            x[h] = i < n ? A[(f + i) * S + k] : make_double2(0.0, 0.0);
            top = max(top, max((uint32_t)__double2hiint(x[h].x) & 0x7fffffffu, (uint32_t)__double2hiint(x[h].y) & 0x7fffffffu));
        }
        top = __reduce_max_sync(0xffffffffu, top);
        if (top < 0x00100000u) continue;          // the column is zero already (uniform across the block)
        const int ex = min((int)(top >> 20), 2045);
        const double up = __hiloint2double((2046 - ex) << 20, 0), down = __hiloint2double(ex << 20, 0);
        double nx2 = 0.0;
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            x[h].x *= up; x[h].y *= up;
            nx2 += x[h].x * x[h].x + x[h].y * x[h].y;
        }
        nx2 = warp_sum_d(nx2);
        const double2 x0 = make_double2(up * A[f * S + k].x, up * A[f * S + k].y);
        const double a2 = x0.x * x0.x + x0.y * x0.y;
        const bool ph = a2 > 1e-200;              // below, x_0 is nothing beside |x| >= 1: any phase will do
        const double nx = sqrt(nx2), ax0 = ph ? sqrt(a2) : 0.0;
        const double beta = 1.0 / (nx * (nx + ax0)), q = ph ? nx / ax0 : 0.0;
        const double2 al = ph ? make_double2(-x0.x * q, -x0.y * q) : make_double2(-nx, 0.0);   // alpha
        if (lane == 0) { x[0].x -= al.x; x[0].y -= al.y; }
        if (wid == 0) {
            #pragma unroll
            for (int h = 0; h < 2; ++h)
                if (lane + 32 * h < n) v[f + lane + 32 * h] = x[h];
        }
        __syncthreads();
        // p = beta A v on the trailing block: two threads per row
        {
            const int i = tid >> 1;
            double2 acc = make_double2(0.0, 0.0);
            if (i < n) {
                const int r = f + i;
                for (int c = f + (tid & 1); c < S; c += 2) {
                    const double2 a = c <= r ? A[r * S + c] : A[c * S + r], vc = v[c];
                    const double ai = c <= r ? a.y : -a.y;
                    acc.x += a.x * vc.x - ai * vc.y;
                    acc.y += a.x * vc.y + ai * vc.x;
                }
            }
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
            if (i < n && !(tid & 1)) pv[f + i] = make_double2(beta * acc.x, beta * acc.y);
        }
        __syncthreads();
        // K = beta/2 v^H p (real), v^H b
        double kr = 0.0, vbx = 0.0, vby = 0.0;
        double2 pr[2];
        #pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = lane + 32 * h;
            pr[h] = make_double2(0.0, 0.0);
            if (i < n) {
                pr[h] = pv[f + i];
                kr += zmulc(x[h], pr[h]).x;
                const double2 u = zmulc(x[h], b[f + i]);
                vbx += u.x; vby += u.y;
            }
        }
        kr = 0.5 * beta * warp_sum_d(kr);
        vbx = beta * warp_sum_d(vbx);
        vby = beta * warp_sum_d(vby);
        __syncthreads();                          // p and b have been read
        // w = p - K v; b <- H b = b - beta v (v^H b)
        if (wid == 0) {
            #pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = lane + 32 * h;
                if (i < n) {
                    pv[f + i] = make_double2(pr[h].x - kr * x[h].x, pr[h].y - kr * x[h].y);
                    const double2 u = zmul(x[h], make_double2(vbx, vby));
                    b[f + i].x -= u.x; b[f + i].y -= u.y;
                }
            }
        }
        __syncthreads();
        // A <- A - v w^H - w v^H on the trailing block; below the diagonal of column k only alpha is left
        for (int i = tid >> 4; i < n; i += NU_THREADS / 16) {
            const int r = f + i;
            const double2 vr = v[r], wr = pv[r];
            for (int c = f + (tid & 15); c <= r; c += 16) {
                const double2 a1 = zmulc(pv[c], vr), a2 = zmulc(v[c], wr);
                double2& a = A[r * S + c];
                a.x -= a1.x + a2.x;
                a.y -= a1.y + a2.y;
            }
        }
        if (tid == 0) A[f * S + k] = make_double2(down * al.x, down * al.y);
        __syncthreads();
    }
    // make off-diagonals real non-negative: D = diag(e^{i th}), th_{k+1} = th_k + arg(e_k)
    double* out = D.nu_T + (size_t)j * 4 * SM;    // [a(SM) | o(SM) | b'(2 SM)]
    for (int k = tid; k + 1 < S; k += NU_THREADS) {
        // (off-diagonals near the end of the range, whose phases are lost, are nothing beside eta)
        const double2 e = A[(k + 1) * S + k];
        const double ae = hypot(e.x, e.y);
        const bool on = !(ae <= 1e-290);
        out[SM + k] = on ? ae : 0.0;
        v[k] = on ? make_double2(e.x / ae, e.y / ae) : make_double2(1.0, 0.0);
    }
    __syncthreads();
    if (tid == 0) {
        double2 ph = make_double2(1.0, 0.0);
        for (int k = 0; k < S; ++k) {
            pv[k] = ph;
            if (k + 1 < S) ph = zmul(ph, v[k]);
        }
        D.nu_c[2 * j] = bv[SM].x;   // |e_all|^2
    }
    __syncthreads();
    for (int k = tid; k < S; k += NU_THREADS) {
        out[k] = A[k * S + k].x;
        const double2 bb = zmulc(pv[k], b[k]);    // b'' = D^H b
        out[2 * SM + 2 * k] = bb.x;
        out[2 * SM + 2 * k + 1] = bb.y;
    }
}
void launch_table(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, int nsplit, int chunk_req,
                  cudaStream_t st) {
    const TablePlan t = table_plan(G, chunk_req);
    smem_allow_max((const void*)k_table);
    k_table<<<dim3(nsplit, S, G.J * t.nblk), t.threads, t.smem, st>>>(G, Pm, D, S, nsplit, chunk_req);
    const int tot = 3 * S * G.J * G.Nz;
    k_table_final<<<(tot + 255) / 256, 256, 0, st>>>(G, Pm, D, S, nsplit);
}

void launch_stage(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, int SCA, const float* z,
                  double* gram, double* nu_b, double* V64, cudaStream_t st) {
    const int gx = min(128, (S * (S + 1) / 2 + 7) / 8);
    k_gram<<<dim3(gx, G.J), 256, 0, st>>>(G, Pm, D, S, gram);
    // element blocks of the basis: about one per SM, 8 to 64 elements
    const int EC = min(64, max(8, (G.Nz * G.J + sm_count() - 1) / sm_count()));
    const size_t smb = (size_t)stage_row(S, S + EC) * sizeof(double2) + S * sizeof(double);
    smem_allow_max((const void*)k_stage_basis);
    k_stage_basis<<<dim3(G.J, (G.Nz + EC - 1) / EC), STAGE_THREADS, smb, st>>>(G, Pm, D, S, EC, z, gram);
    const size_t sm = stage_kappa_smem(S, G.Nz);
    smem_allow_max((const void*)k_stage_kappa);
    k_stage_kappa<<<dim3(S, G.J), STAGE_THREADS, sm, st>>>(G, Pm, D, S, SCA, gram, nu_b, V64);
}

void launch_nu_tridiag(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, const double* gram,
                       const double* nu_b, cudaStream_t st, cudaStream_t side, cudaEvent_t ev_fork, cudaEvent_t ev_join) {
    // on the side stream the J blocks run beside the MT likelihood (whose blocks are short; the
    // persistent PF likelihood before it would wait for the SMs they hold)
    const bool fork = side && ev_fork && ev_join;
    if (fork) {
        cudaEventRecord(ev_fork, st);
        cudaStreamWaitEvent(side, ev_fork, 0);
    }
    const size_t sm = ((size_t)S * S + 3 * (size_t)S) * sizeof(double2);
    smem_allow_max((const void*)k_nu_tridiag);
    k_nu_tridiag<<<G.J, NU_THREADS, sm, fork ? side : st>>>(Pm, D, S, gram, nu_b);
    if (fork) cudaEventRecord(ev_join, side);
}

static int current_device() {
    int dev = 0;
    cudaGetDevice(&dev);
    return dev;
}
static int device_attribute(int dev, cudaDeviceAttr attr, int fallback) {
    int a = 0;
    cudaDeviceGetAttribute(&a, attr, dev);
    return a > 0 ? a : fallback;
}

void smem_allow_max(const void* kernel) {
    static OncePerDevice done;
    done.run(current_device(), kernel, [&] {
        cudaFuncAttributes a{};
        cudaFuncGetAttributes(&a, kernel);
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin() - (int)a.sharedSizeBytes);
    });
}

int sm_count() {
    static NumberPerDevice v;
    const int dev = current_device();
    return v.get(dev, [&] { return device_attribute(dev, cudaDevAttrMultiProcessorCount, 1); });
}

int smem_optin() {
    static NumberPerDevice v;
    const int dev = current_device();
    return v.get(dev, [&] { return device_attribute(dev, cudaDevAttrMaxSharedMemoryPerBlockOptin, 48 * 1024); });
}

}  // namespace bp
