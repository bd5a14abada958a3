// PF likelihood kappa~ (Supplementary Sec. S-V, "PF state update message") of every
// (PF s, particle p), relative to the null hypothesis and summed over the PAs j.
//
// With A = eta_bar I + M M^H (M the other PFs' m-vectors), e0 = z - sum_{t != s} mu3_t,
// a = zeta mu and q = (gamma + |mu|^2 (1 - zeta)) zeta of the particle, and its steering vector
// psi, the matrix inversion and determinant lemmas give the log-ratio in closed form:
//     b = psi^H A^-1 e0,   alpha = psi^H A^-1 psi,   d = b - alpha a,
//     Delta = Re(conj(a) (b + d)) + q |d|^2 / (1 + q alpha) - log(1 + q alpha).
// The table stage supplies V with V V^H = M (I + M^H M / eta_bar)^-1 M^H and r0 = eta_bar A^-1 e0,
// so both scalars come from one contraction of psi with the columns of V~ = V / sqrt(eta_bar)
// and r0.  With psi = A u, |u_k| = 1, and h = u^H V~:
//     alpha = (A^2 / eta_bar) (|u|^2 - |h|^2),   b = A u^H r0 / eta_bar.
// alpha is a small difference where the others' span holds most of psi (PFs that nearly
// coincide), and Delta reaches ~1e3 nats, so h is needed to ~1e-10 of |u||V_c|, far beyond FP32.
//
// Precision on the tensor cores.  u (as a (hi, lo) FP32 pair, ~1e-9) and the columns of V~ and
// r0 (scaled by a power of two to just below 1) are written in fixed point as four signed
// base-256 digits of units 2^-7, 2^-15, 2^-23, 2^-31.  A digit has at most 8 bits, so it is exact
// in BF16, and a product of two digits is an integer multiple of its unit; the sums of the
// products of one total weight stay below 2^24 of that unit, so the FP32 accumulator of
// tcgen05.mma kind::f16 holds them exactly.  The digit products (i, k) with i + k <= 5 (ten of
// sixteen; the rest is below 2^-35 of |u||V_c|) go to four accumulators g_{i+k-2}, which the
// epilogue adds as an FP32 pair.  The earlier kernel (3xTF32, FP32 accumulation) needed a second
// contraction V conj(h) and an element-wise float-float residual to make the error of h
// second order; here there is one contraction, at twice the TF32 rate, and nothing per element
// after it.
//
// Half the elements.  The frequencies and the element positions are symmetric about 0, so without
// the carrier u_{Nz-1-k} = conj(u_k), and
//     u^H v = sum_{k < Nz/2} Re u_k (v_k + v_k') - i Im u_k (v_k - v_k'),   k' = Nz - 1 - k:
// the operand columns hold the sums and differences, the producers form one half of the elements,
// and K halves.  (A layout that is not symmetric takes all elements; the carrier phase turns
// u^H r0 once per particle.)
//
// Shape of the kernel.  M tile = 128 particles (TMEM lane = particle), N = 2 SW columns (Re h,
// Im h; SW = S rounded up to 8), K = 2 Nh (Re, Im interleaved; Nh elements) in chunks of 32.  The
// four digit slices of B lie side by side along N, and so do the accumulators, so the products
// of A's digit i with B's digits 1 .. 5 - i are one run of 2 SW (5 - i) columns (N <= 256 per
// instruction) onto g_{i-1} .. g_3.  One persistent block per SM: four producer groups of 128
// threads build the A chunks (group g forms elements 4 g .. 4 g + 3 of each chunk, in registers,
// two elements per packed FP32 instruction), one thread issues the MMAs and the bulk copies of
// the prebuilt B chunks, and the producers read the accumulators of a finished (s, p tile, j)
// after they have refilled the ring with the next one's first chunks, so the tensor cores wait
// only for that read (not at all where two accumulator sets fit in TMEM, SW <= 32).
// Bound: the producers' FP32 issue (about 45 instructions per element with its share of the factors
// and the epilogue); the tensor pipe is next (ten products of 128 x 2 SW x 2 Nh).
// Measured (PF likelihood stage, J = 4): 64 PFs x 1e5 particles, Nz = 160: 56.7 -> 15.6 ms; 32 PFs x
// 262144, Nz = 1024: 401 -> 87 ms; 10 PFs x 30000, Nz = 160: 3.66 -> 0.58 ms (against the 3xTF32
// kernel, below 33 PFs a CUDA-core kernel, with a second pass each).
#include "bp_internal.cuh"
#include "bp_kernels.cuh"
#include "tc_sm100.cuh"

namespace bp {

constexpr int KX_WAIT = 1 << 20;       // polls of a bounded wait
constexpr int KX_NG = 4;               // producer groups (128 threads each)
constexpr int KX_PT = 128 * KX_NG;     // producer threads
constexpr int KX_T = KX_PT + 32;       // + the issuing warp
constexpr int KX_KC = 32;              // real K per chunk (16 elements)
constexpr int KX_A = 4 * 128 * KX_KC * 2;   // bytes of A per chunk: 4 digits x 128 rows x KX_KC BF16
constexpr int KX_NST_MAX = 4;

__host__ __device__ inline int kx_sw(int S) { return (S + 7) & ~7; }
__host__ __device__ inline int kx_chunks(int Nh) { return (Nh + 15) / 16; }
__host__ __device__ inline uint32_t kx_bbytes(int SW) { return (uint32_t)(2 * SW) * KX_KC * 2 * 4; }   // 4 digits
// elements a particle forms: half of them where the layout is symmetric
__host__ __device__ inline int kx_elements(const DevGeom& G) { return G.sym ? (G.Nz + 1) / 2 : G.Nz; }
__host__ __device__ inline int kx_freqs(const DevGeom& G) { return (kx_elements(G) - 1) / (G.My * G.Mz) + 1; }
// shared memory after the ring: steering factors [nfac][128] as (hi, lo) pairs, cis table [256],
// partial sums [KX_NG][128], u^H r0 [128] (float4 each), column scales [3][64], barriers and flags
__host__ __device__ inline size_t kx_smem_fixed(int nfac) {
    return ((size_t)nfac * 128 + 256 + KX_NG * 128 + 128) * sizeof(float4) + 3 * 64 * sizeof(float) + 256;
}

// a b for unit-modulus pairs, two elements at a time, in fixed point: hi a multiple of 2^-22
// (adding 3 rounds each product onto that grid, where the sums are exact), lo the remainders and
// the low-order cross terms (|lo| < 2^-20)
struct KxW { f2x x, y, ny, xl, yl, nyl; };     // the outer factor of each of the two elements
struct KxU { f2x xh, yh, xl, yl; };
__device__ __forceinline__ KxW kx_w(float4 a, float4 b) {
    return KxW{f2_pack(a.x, b.x), f2_pack(a.y, b.y), f2_pack(-a.y, -b.y), f2_pack(a.z, b.z), f2_pack(a.w, b.w),
               f2_pack(-a.w, -b.w)};
}
__device__ __forceinline__ void kx_dot2(f2x a, f2x b, f2x c, f2x d, f2x al, f2x bl, f2x cl, f2x dl, f2x& hi, f2x& lo) {
    const f2x m = f2_dup(3.0f);                 // (a + al)(b + bl) + (c + cl)(d + dl)
    const f2x t = f2_fma(a, b, m), t2 = f2_fma(c, d, t);
    const f2x p = f2_fma(a, b, f2_sub(m, t)), q = f2_fma(c, d, f2_sub(t, t2));
    hi = f2_sub(t2, m);
    lo = f2_add(f2_fma(a, bl, f2_fma(al, b, p)), f2_fma(c, dl, f2_fma(cl, d, q)));
}
__device__ __forceinline__ KxU kx_mul(const KxW& w, const KxU& a) {
    KxU u;
    kx_dot2(w.x, a.xh, w.ny, a.yh, w.xl, a.xl, w.nyl, a.yl, u.xh, u.xl);
    kx_dot2(w.x, a.yh, w.y, a.xh, w.xl, a.yl, w.yl, a.xl, u.yh, u.yl);
    return u;
}
// the four digits of two elements: adding 1.5 x 2^23 units rounds to a multiple of the unit, the
// remainder is exact; digit i of element e in w[i][e] as the BF16 pair (Re, Im)
__device__ __forceinline__ void kx_digits(const KxU& u, uint32_t (&w)[4][2]) {
    const float M[4] = {98304.0f, 384.0f, 1.5f, 0.005859375f};   // 1.5 x 2^16, 2^8, 2^0, 2^-8
    f2x rx = u.xh, ry = u.yh;
    #pragma unroll
    for (int i = 0; i < 4; ++i) {
        const f2x m = f2_dup(M[i]), mn = f2_dup(-M[i]);
        const f2x sx = f2_add(f2_add(rx, m), mn), sy = f2_add(f2_add(ry, m), mn);
        uint32_t x0, x1, y0, y1;
        f2_unpack(sx, x0, x1);
        f2_unpack(sy, y0, y1);
        w[i][0] = __byte_perm(x0, y0, 0x7632);     // upper halves: the digits are exact in BF16
        w[i][1] = __byte_perm(x1, y1, 0x7632);
        if (i < 3) { rx = f2_sub(rx, sx); ry = f2_sub(ry, sy); }
        if (i == 1) { rx = f2_add(rx, u.xl); ry = f2_add(ry, u.yl); }
    }
}
// Delta of one (p, s, j): consts (1/eta_bar, zeta as pairs), amplitude A, gamma, mu, alpha_u =
// |u|^2 - |h|^2 and pr = u^H r0
__device__ inline ff kx_delta(float4 kc, float A, float gm, float mr, float mi, ff alpha_u, cff pr) {
    const ff ieb{kc.x, kc.y}, zeta{kc.z, kc.w};
    const ff Aeb = ff_mulf(ieb, A);                      // A / eta_bar
    const ff alpha = ff_mul(ff_mulf(Aeb, A), alpha_u);
    const cff b{ff_mul(Aeb, pr.re), ff_mul(Aeb, pr.im)};
    const cff a{ff_mulf(zeta, mr), ff_mulf(zeta, mi)};
    const cff d{ff_add(b.re, ff_neg(ff_mul(alpha, a.re))), ff_add(b.im, ff_neg(ff_mul(alpha, a.im)))};
    ff out = ff_add(ff_mul(a.re, ff_add(b.re, d.re)), ff_mul(a.im, ff_add(b.im, d.im)));
    const float zf = kc.z;
    const float q = (gm + (mr * mr + mi * mi) * (1.0f - zf)) * zf;
    if (q > 0.f) {
        const ff qa = ff_mulf(alpha, q);
        const ff g = ff_div(ff{q, 0.f}, ff_add(ff{1.0f, 0.f}, qa));
        const ff d2 = ff_add(ff_mul(d.re, d.re), ff_mul(d.im, d.im));
        out = ff_add(out, ff_mul(g, d2));
        out = ff_add(out, ff{-log1pf(qa.hi), 0.f});
    }
    return out;
}

// steering factors of one (particle, s, j) as (hi, lo) pairs (cis_pair, ~1e-9)
struct KxPath {
    float dh, dl, h0, l0;   // distance, carrier cycles (float-float)
    float uy, uz, uyl, uzl; // direction cosines
};
__device__ __forceinline__ KxPath kx_path(const DevGeom& G, float4 g, float2 gl) {
    KxPath t{g.x, g.y, 0.f, 0.f, g.z, g.w, gl.x, gl.y};
    ff_frac_mul2(g.x, g.y, G.inv_lam_hi, G.inv_lam_lo, t.h0, t.l0);
    return t;
}
// antenna factor i < My: a_y, else a_z of element i - My
__device__ __forceinline__ float4 kx_antenna(const DevGeom& G, const float4* tab, const KxPath& t, int i) {
    const bool y = i < G.My;
    const float c = y ? G.py_l[i] : G.pz_l[i - G.My], cl = y ? G.py_lo[i] : G.pz_lo[i - G.My];
    const float u = y ? t.uy : t.uz, ul = y ? t.uyl : t.uzl;
    const float p = __fmul_rn(c, u);
    const float e = fmaf(c, ul, fmaf(cl, u, fmaf(c, u, -p)));
    float2 hi, lo;
    cis_pair(tab, p, e, hi, lo);
    return make_float4(hi.x, hi.y, lo.x, lo.y);
}
__device__ __forceinline__ float4 kx_pair_mul(float4 a, float4 b) {
    return cpair_mul(make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y), make_float2(b.z, b.w));
}

// ---------------------------------------------------------------- operand digits of V~ and r0
// Block (s, j, part of the chunks): the columns' power-of-two scales (largest part in [1/2, 1)
// after scaling), then the four digit slices of its chunks of 16 elements as rows n < SW (Re h_n)
// and n >= SW (Im h_{n - SW}) against k = 2 e + part, K-major core matrices:
// [Re(v + v'), Im(v - v')] and [Im(v + v'), -Re(v - v')] for a symmetric layout (v' the mirrored
// element's, the middle element counted once), else [Re v, Im v] and [Im v, -Re v].  Column SW - 1
// is r0, unused columns are zero.  Bound: the FP64 conversions (82 us at 64 PFs x 4 PAs x Nz = 160).
constexpr int KX_DSPLIT = 4;   // blocks per (s, j)
__global__ void __launch_bounds__(256) k_kappa_digits(DevGeom G, DevState D, int S, int SCA, int SW,
                                                      const double2* __restrict__ V64) {
    const int s = blockIdx.x, j = blockIdx.y, J = G.J, Nz = G.Nz, K = S - 1, Nh = kx_elements(G);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const bool sym = G.sym != 0;
    const double eb = D.eta_bar[j];
    const double isq = 1.0 / sqrt(eb);
    const double2* V = V64 + ((size_t)s * J + j) * SCA * Nz;      // [SCA][Nz]
    // (Re(v + v'), Im(v - v'), Im(v + v'), Re(v - v')) of element k
    auto combo = [&](const double2* v, int k, double (&o)[4]) {
        const double2 a = v[k];
        o[0] = o[3] = a.x; o[1] = o[2] = a.y;
        if (sym) {
            const int k2 = Nz - 1 - k;
            const double2 b = v[k2];
            if (k2 != k) { o[0] += b.x; o[1] -= b.y; o[2] += b.y; o[3] -= b.x; }
            else { o[1] = o[3] = 0.0; }
        }
    };
    __shared__ double sc[64];                                      // scale of column c (incl. 1/sqrt(eta_bar))
    for (int c = wid; c < SW; c += nw) {
        const bool r0 = c == SW - 1;
        double f = 0.0;
        float inv = 0.f;
        if (r0 || c < K) {
            const double2* v = V + (size_t)(r0 ? SCA - 1 : c) * Nz;
            double m = 0.0;
            for (int k = lane; k < Nh; k += 32) {
                double o[4];
                combo(v, k, o);
                m = fmax(m, fmax(fmax(fabs(o[0]), fabs(o[1])), fmax(fabs(o[2]), fabs(o[3]))));
            }
            m = warp_max_d(m) * (r0 ? 1.0 : isq);
            if (m > 0.0 && isfinite(m)) {
                int e;
                frexp(m, &e);
                f = ldexp(r0 ? 1.0 : isq, -e);
                inv = ldexpf(1.0f, e);
            }
        }
        if (lane == 0) {
            sc[c] = f;
            if (blockIdx.z == 0) D.kSc[((size_t)s * J + j) * 64 + c] = inv;
        }
    }
    if (threadIdx.x == 0 && blockIdx.z == 0) {
        const double ieb = 1.0 / eb, zeta = D.zeta[s * J + j];
        const float ih = (float)ieb, zh = (float)zeta;
        D.kC[s * J + j] = make_float4(ih, (float)(ieb - (double)ih), zh, (float)(zeta - (double)zh));
    }
    __syncthreads();
    const int N1 = 2 * SW, NCk = kx_chunks(Nh);
    const uint32_t slice = (uint32_t)N1 * KX_KC * 2;   // bytes of one digit slice
    unsigned char* out = D.kB + ((size_t)s * J + j) * NCk * 4 * slice;
    // one item: column c of element 16 kc + e; consecutive threads walk the words of a core
    // matrix (4 elements x 8 rows)
    const int per = SW * 16;
    for (int t = blockIdx.z * blockDim.x + threadIdx.x; t < NCk * per; t += gridDim.z * blockDim.x) {
        const int kc = t / per, r = t - kc * per;
        const int e = (r & 3) + 4 * ((r >> 5) & 3), c = ((r >> 2) & 7) + 8 * (r >> 7);
        const int k = 16 * kc + e;
        long long q[4] = {0, 0, 0, 0};
        if (k < Nh && sc[c] != 0.0) {
            double o[4];
            combo(V + (size_t)(c == SW - 1 ? SCA - 1 : c) * Nz, k, o);
            const double f = sc[c] * 2147483648.0;
            #pragma unroll
            for (int i = 0; i < 4; ++i) q[i] = __double2ll_rn(o[i] * f);
            q[3] = -q[3];
        }
        unsigned char* o = out + (size_t)kc * 4 * slice;
        const uint32_t o1 = (uint32_t)tc::core_off16(c, 2 * e, KX_KC), o2 = (uint32_t)tc::core_off16(SW + c, 2 * e, KX_KC);
        float unit = 4.656612873077393e-10f;   // 2^-31
        #pragma unroll
        for (int i = 3; i >= 0; --i) {
            uint32_t w[4];
            #pragma unroll
            for (int v = 0; v < 4; ++v) {
                int d = (int)q[v];
                if (i > 0) {
                    d = (int)(signed char)(q[v] & 255);
                    q[v] = (q[v] - d) >> 8;
                }
                w[v] = __float_as_uint((float)d * unit) >> 16;   // at most 8 significant bits
            }
            *reinterpret_cast<uint32_t*>(o + (size_t)i * slice + o1) = w[0] | (w[1] << 16);
            *reinterpret_cast<uint32_t*>(o + (size_t)i * slice + o2) = w[2] | (w[3] << 16);
            unit *= 256.0f;
        }
    }
}

// ---------------------------------------------------------------- the tensor-core kernel
__device__ __forceinline__ void kx_bar() { asm volatile("bar.sync 1, %0;" :: "n"(KX_PT) : "memory"); }
__device__ __forceinline__ void kx_arrive(uint32_t mbar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mbar) : "memory");
}
__device__ __forceinline__ void kx_sts(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" :: "r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// VEC: largest of 4, 2, 1 that divides Mz (elements between possible row changes).  btab: the
// frequency factors stay in shared memory (else they are formed when a row of elements begins).
template <int VEC>
__global__ void __launch_bounds__(KX_T, 1) k_kappa_x(DevGeom G, DevParams Pm, DevState D, int S, int SW, int nst, int btab) {
    extern __shared__ __align__(1024) unsigned char smx[];
    const int P = Pm.P, J = G.J, Nz = G.Nz, My = G.My, Mz = G.Mz, Nm = My * Mz, Nf = G.Nf;
    const int Nh = kx_elements(G), Fh = btab ? kx_freqs(G) : 0;
    const int N1 = 2 * SW, NCk = kx_chunks(Nh);
    const int nfac = My + ((Mz + 1) & ~1) + Fh;
    const uint32_t bbytes = kx_bbytes(SW), stage = KX_A + bbytes;
    // steering factors of the 128 particles: a_y [My], a_z (pairs of elements for VEC > 1), b [Fh]
    float4* fy = reinterpret_cast<float4*>(smx + (size_t)nst * stage);
    float4* fz = fy + (size_t)My * 128;
    float4* fb = fz + (size_t)((Mz + 1) & ~1) * 128;
    float4* ctab = fy + (size_t)nfac * 128;                              // [256]
    float4* exs = ctab + 256;                                            // [KX_NG][128] |h|^2 (grid, rest), dev
    float4* exr = exs + KX_NG * 128;                                     // [128] u^H r0
    float* ssc = reinterpret_cast<float*>(exr + 128);                    // [3][64] column scales (unit mod 3: fetched one unit ahead, read one behind)
    uint64_t* mb = reinterpret_cast<uint64_t*>(ssc + 3 * 64);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mb + 2 * KX_NST_MAX + 4);
    volatile int* sbad = reinterpret_cast<volatile int*>(tslot + 1);
    const uint32_t mfull = tc::smem_u32(mb), mempty = mfull + 8 * KX_NST_MAX;   // slot filled; its MMAs done
    const uint32_t maccf = mempty + 8 * KX_NST_MAX, macce = maccf + 16;         // accumulator set complete; read
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int nacc = 8 * N1 <= 512 ? 2 : 1;                              // accumulator sets of 4 N1 columns
    uint32_t ncols = 32;
    while (ncols < (uint32_t)(nacc * 4 * N1)) ncols *= 2;
    if (warp == 0) tc::tmem_alloc(tslot, ncols);
    if (tid == 0) {
        for (int i = 0; i < nst; ++i) {
            tc::mbar_init(mfull + 8 * i, KX_PT / 32 + 1);    // every producer warp and the B copy
            tc::mbar_init(mempty + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(maccf + 8 * i, 1);
            tc::mbar_init(macce + 8 * i, KX_PT / 32);
        }
        tc::mbar_init_fence();
        *sbad = 0;
    }
    for (int i = tid; i < 256; i += KX_T) ctab[i] = D.ctab[i];
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    const uint32_t tmem = *tslot;
    // a wait that gives up marks the block bad: nobody waits any more, every loop runs out
    auto wait = [&](uint32_t mbar, uint32_t parity) {
        if (*sbad) return;
        if (!tc::mbar_wait(mbar, parity & 1u, KX_WAIT)) *sbad = 1;
    };
    const int ptiles = (P + 127) / 128, items = S * ptiles;
    const int nit = (int)blockIdx.x < items ? (items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int units = nit * J;                   // (item, j) in order
    const uint32_t ring = tc::smem_u32(smx);
    if (warp == KX_PT / 32) {
        // ---- issuing thread: B copies and MMAs
        if (lane == 0) {
            const int total = units * NCk;
            int li = 0, lj = 0, lk = 0, ls = 0;  // load cursor: item, j, chunk, slot
            auto load = [&]() {
                const int s = (blockIdx.x + li * gridDim.x) / ptiles;
                const unsigned char* src = D.kB + (((size_t)s * J + lj) * NCk + lk) * bbytes;
                tc::mbar_expect_tx(mfull + 8 * ls, bbytes);
                tc::bulk_g2s(ring + ls * stage + KX_A, src, bbytes, mfull + 8 * ls);
                if (++ls == nst) ls = 0;
                if (++lk == NCk) { lk = 0; if (++lj == J) { lj = 0; ++li; } }
            };
            int loaded = 0;
            for (; loaded < min(nst, total); ++loaded) load();
            int n = 0;
            for (int u = 0; u < units && !*sbad; ++u) {
                const int set = nacc == 2 ? (u & 1) : 0, use = nacc == 2 ? (u >> 1) : u;
                if (use > 0) wait(macce + 8 * set, use - 1);
                const uint32_t acc0 = tmem + (uint32_t)(set * 4 * N1);
                for (int kc = 0; kc < NCk && !*sbad; ++kc, ++n) {
                    const int st = n % nst;
                    wait(mfull + 8 * st, n / nst);
                    if (*sbad) break;
                    tc::fence_after_sync();
                    const uint32_t aB = ring + st * stage, bB = aB + KX_A;
                    #pragma unroll
                    for (int ks = 0; ks < KX_KC / 16; ++ks) {
                        #pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            const uint64_t da = tc::smem_desc(aB + i * (128 * KX_KC * 2) + ks * 256, 128, KX_KC * 16);
                            const int cols = (4 - i) * N1;
                            for (int c0 = 0; c0 < cols; c0 += 256) {
                                const int nn = min(256, cols - c0);
                                const uint64_t db = tc::smem_desc(bB + c0 * KX_KC * 2 + ks * 256, 128, KX_KC * 16);
                                tc::mma_bf16(acc0 + (uint32_t)(i * N1 + c0), da, db, tc::idesc_bf16_f32(128, nn),
                                             kc > 0 || ks > 0 || i > 0);
                            }
                        }
                    }
                    tc::mma_commit(mempty + 8 * st);
                    if (kc == NCk - 1) tc::mma_commit(maccf + 8 * set);
                    // the slot of chunk n - 1 takes chunk n - 1 + nst once its MMAs are done
                    if (n >= 1 && n - 1 + nst < total) {
                        wait(mempty + 8 * ((n - 1) % nst), (n - 1) / nst);
                        if (*sbad) break;
                        load();
                        ++loaded;
                    }
                }
            }
            // after a wait that gave up: let the copies and MMAs in flight land (bounded)
            if (*sbad) {
                for (int m = max(0, loaded - nst); m < loaded; ++m) tc::mbar_wait(mfull + 8 * (m % nst), (m / nst) & 1, KX_WAIT);
                for (int m = max(0, n - nst); m < n; ++m) tc::mbar_wait(mempty + 8 * (m % nst), (m / nst) & 1, KX_WAIT);
            }
        }
        __syncwarp();
    } else {
        // ---- producers and epilogue
        const int grp = warp >> 2, row = tid & 127;
        const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const uint32_t arow = (uint32_t)((row >> 3) * (KX_KC * 16) + (row & 7) * 16 + grp * 128);
        float GM = 1.5f;                          // grid of the |h|^2 sum: |h|^2 <= Nz
        for (int v = 1; v < 4 * Nz; v *= 2) GM *= 2.0f;
        // first element of this group's four in chunk 0, and the step of 16 elements, in (f, y, m)
        const int f_0 = 4 * grp / Nm, y_0 = (4 * grp - f_0 * Nm) / Mz, m_0 = 4 * grp - f_0 * Nm - y_0 * Mz;
        const int f_s = 16 / Nm, y_s = (16 - f_s * Nm) / Mz, m_s = 16 - f_s * Nm - y_s * Mz;
        float pA = 0.f, pDev = 0.f, pH0 = 0.f, pL0 = 0.f;   // previous unit: amplitude, |u|^2 - Nz (this group's part), carrier
        ff delta{0.f, 0.f};
        // reads the accumulators of unit u, and one group per item evaluates Delta
        auto epilogue = [&](int u) {
            const int it = u / J, j = u - it * J;
            const int item = blockIdx.x + it * gridDim.x, s = item / ptiles, p = (item - s * ptiles) * 128 + row;
            const int set = nacc == 2 ? (u & 1) : 0, use = nacc == 2 ? (u >> 1) : u;
            const float* scl = ssc + (u % 3) * 64;
            const bool fin = it % KX_NG == grp;
            float gm = 0.f, mr = 0.f, mi = 0.f;
            float4 kc = make_float4(0.f, 0.f, 0.f, 0.f);
            if (fin) {
                const float* ph = D.phi[D.cur] + (size_t)s * 6 * P + min(p, P - 1);
                gm = ph[3 * (size_t)P]; mr = ph[4 * (size_t)P]; mi = ph[5 * (size_t)P];
                kc = D.kC[s * J + j];
            }
            wait(maccf + 8 * set, use);
            __syncwarp();
            tc::fence_after_sync();
            const uint32_t acc0 = tlane + (uint32_t)(set * 4 * N1);
            const f2x gm2 = f2_dup(GM);
            f2x hg = f2_dup(0.f), hr = hg;
            for (int c0 = 8 * grp; c0 < SW; c0 += 8 * KX_NG) {
                #pragma unroll
                for (int part = 0; part < 2; ++part) {
                    uint32_t g[4][8];
                    #pragma unroll
                    for (int i = 0; i < 4; ++i) tc::tmem_ld8(acc0 + (uint32_t)(i * N1 + part * SW + c0), g[i]);
                    tc::tmem_ld_wait();
                    auto col2 = [&](int i, int q) { return f2_pack(__uint_as_float(g[i][q]), __uint_as_float(g[i][q + 1])); };
                    #pragma unroll
                    for (int q = 0; q < 8; q += 2) {     // two columns at a time
                        // g_0 + g_1 exactly, the rest onto its error
                        const f2x a = col2(0, q), b = col2(1, q), t = f2_add(a, b), bb = f2_sub(t, a);
                        const f2x e = f2_add(f2_add(f2_sub(a, f2_sub(t, bb)), f2_sub(b, bb)), f2_add(col2(2, q), col2(3, q)));
                        if (q == 6 && c0 + 8 == SW) {    // u^H r0 (its scale in the table is zero)
                            uint32_t lo, th, eh;
                            f2_unpack(t, lo, th);
                            f2_unpack(e, lo, eh);
                            float* r = reinterpret_cast<float*>(exr + row) + 2 * part;
                            r[0] = __uint_as_float(th);
                            r[1] = __uint_as_float(eh);
                        }
                        const f2x sc = f2_pack(scl[c0 + q], scl[c0 + q + 1]);   // powers of two: exact
                        const f2x hi = f2_mul(t, sc), lo = f2_mul(e, sc);
                        const f2x nt = f2_sub(gm2, f2_fma(hi, hi, gm2));        // - |.|^2 on the grid
                        hg = f2_sub(hg, nt);
                        hr = f2_fma(f2_add(hi, hi), lo, f2_add(hr, f2_fma(hi, hi, nt)));
                    }
                }
            }
            tc::fence_before_sync();
            __syncwarp();
            if (lane == 0) kx_arrive(macce + 8 * set);
            uint32_t g0, g1, r0, r1;
            f2_unpack(hg, g0, g1);
            f2_unpack(hr, r0, r1);
            exs[grp * 128 + row] = make_float4(__fadd_rn(__uint_as_float(g0), __uint_as_float(g1)),
                                               __uint_as_float(r0) + __uint_as_float(r1), pDev, 0.f);
            kx_bar();
            if (fin) {
                float sg = 0.f, sr = 0.f, dev = 0.f;
                #pragma unroll
                for (int g = 0; g < KX_NG; ++g) {
                    const float4 v = exs[g * 128 + row];
                    sg = __fadd_rn(sg, v.x);      // multiples of the grid: exact
                    sr += v.y;
                    dev += v.z;
                }
                ff au;
                two_sum(__fsub_rn((float)Nz, sg), dev - sr, au.hi, au.lo);
                if (!(au.hi > 0.f)) au = ff{0.f, 0.f};
                const float4 r = exr[row];
                const float rs = D.kSc[((size_t)s * J + j) * 64 + SW - 1];
                cff pr;
                fast_two_sum(r.x * rs, r.y * rs, pr.re.hi, pr.re.lo);
                fast_two_sum(r.z * rs, r.w * rs, pr.im.hi, pr.im.lo);
                float2 ch, cl;                    // the carrier: conj(e^{-i 2 pi d / lambda})
                cis_pair(ctab, pH0, pL0, ch, cl);
                pr = cff_mul(pr, cff{ff{ch.x, cl.x}, ff{ch.y, cl.y}});
                const ff dl = kx_delta(kc, pA, gm, mr, mi, au, pr);
                delta = j == 0 ? dl : ff_add(delta, dl);
                if (j == J - 1 && p < P) D.lw_y[(size_t)s * P + p] = ff_to_d(delta);
            }
        };
        float4 ngeo = make_float4(1.f, 0.f, 0.f, 0.f);
        float2 ngl = make_float2(0.f, 0.f);
        auto fetch = [&](int u) {                 // geometry record of unit u
            const int it = u / J, j = u - it * J;
            const int item = blockIdx.x + it * gridDim.x, s = item / ptiles, p = (item - s * ptiles) * 128 + row;
            const size_t gi = ((size_t)s * J + j) * P + min(p, P - 1);
            ngeo = D.geo[gi];
            ngl = D.geo_lo[gi];
            if (tid < 64) ssc[(u % 3) * 64 + tid] = tid < SW - 1 ? D.kSc[((size_t)s * J + j) * 64 + tid] : 0.f;
        };
        if (units > 0) fetch(0);
        int st = 0, use = 0;                      // ring slot and its turn
        for (int u = 0; u < units; ++u) {
            const float4 grec = ngeo;
            const float2 grl = ngl;
            const float A = G.amp_c / (grec.x + grec.y);
            float dev = 0.f;
            // the antenna factors of a symmetric layout come in conjugate pairs
            auto antenna = [&](int i, bool isz) {
                const float c = isz ? G.pz_l[i] : G.py_l[i], cl = isz ? G.pz_lo[i] : G.py_lo[i];
                const float uu = isz ? grec.w : grec.z, ul = isz ? grl.y : grl.x;
                const float t = __fmul_rn(c, uu);
                float2 hi, lo;
                cis_pair(ctab, t, fmaf(c, ul, fmaf(cl, uu, fmaf(c, uu, -t))), hi, lo);
                return make_float4(hi.x, hi.y, lo.x, lo.y);
            };
            auto put_z = [&](int m, float4 a) {
                if (VEC == 1) { fz[m * 128 + row] = a; return; }
                float* o = reinterpret_cast<float*>(fz + (m & ~1) * 128 + row) + (m & 1);   // (hx, hx', hy, hy'), then lo
                o[0] = a.x; o[2] = a.y;
                o[512] = a.z; o[514] = a.w;
            };
            auto freq = [&](int f) {              // b_f, without the carrier
                float h, l;
                ff_frac_mul2(grec.x, grec.y, G.fc_hi[f], G.fc_lo[f], h, l);
                float2 hi, lo;
                cis_pair(ctab, -h, -l, hi, lo);
                return make_float4(hi.x, hi.y, lo.x, lo.y);
            };
            auto unit_dev = [&](float4 a) { return pair_unit_dev(make_float2(a.x, a.y), make_float2(a.z, a.w)); };
            const float fdup = G.sym ? 2.0f : 1.0f;
            kx_bar();                             // every group is done with the previous unit's factors
            const int hy = G.sym ? (My + 1) / 2 : My, hz = G.sym ? (Mz + 1) / 2 : Mz;
            for (int i = grp; i < hy + hz + Fh; i += KX_NG) {
                if (i < hy) {
                    const float4 a = antenna(i, false);
                    const int i2 = My - 1 - i;
                    const bool two = G.sym && i2 != i;
                    fy[i * 128 + row] = a;
                    if (two) fy[i2 * 128 + row] = make_float4(a.x, -a.y, a.z, -a.w);
                    dev = fmaf((float)(Nf * Mz) * (two ? 2.0f : 1.0f), unit_dev(a), dev);
                } else if (i < hy + hz) {
                    const int m = i - hy, m2 = Mz - 1 - m;
                    const float4 a = antenna(m, true);
                    const bool two = G.sym && m2 != m;
                    put_z(m, a);
                    if (two) put_z(m2, make_float4(a.x, -a.y, a.z, -a.w));
                    dev = fmaf((float)(Nf * My) * (two ? 2.0f : 1.0f), unit_dev(a), dev);
                } else {
                    // (the middle frequency is 0: no deviation)
                    const int f = i - hy - hz;
                    const float4 a = freq(f);
                    fb[f * 128 + row] = a;
                    dev = fmaf((float)Nm * fdup, unit_dev(a), dev);
                }
            }
            kx_bar();
            if (u + 1 < units) fetch(u + 1);
            bool drained = u == 0;
            int f = f_0, y = y_0, m = m_0;
            for (int kc = 0; kc < NCk; ++kc) {
                // a slot of this unit's own ring turn frees only once the previous unit's
                // accumulators are read
                if (!drained && kc >= nst) { epilogue(u - 1); drained = true; }
                if (use > 0) wait(mempty + 8 * st, use - 1);
                const int k = 16 * kc + 4 * grp;
                uint32_t d[4][4];                 // [digit][element]
                #pragma unroll
                for (int i = 0; i < 4; ++i) d[i][0] = d[i][1] = d[i][2] = d[i][3] = 0u;
                if (k < Nh) {
                    int yy = y, mm = m, ff_ = f;
                    float4 b;
                    auto set_b = [&](int e) {
                        if (btab) { b = fb[ff_ * 128 + row]; return; }
                        b = freq(ff_);
                        const int cnt = min(min((ff_ + 1) * Nm, 16 * kc + 4 * grp + 4), Nh) - (k + e);
                        dev = fmaf((float)cnt * fdup, unit_dev(b), dev);
                    };
                    auto step = [&](int e, int by) {   // to element e (by elements on); true if the row changed
                        mm += by;
                        if (mm < Mz) return false;
                        mm = 0;
                        if (++yy == My) {
                            yy = 0;
                            ++ff_;
                            if (k + e < Nh) set_b(e);
                        }
                        return true;
                    };
                    set_b(0);
                    float4 w = pair_mul_fx(b, fy[yy * 128 + row]);
                    KxW w2;
                    if (VEC > 1) w2 = kx_w(w, w);
                    #pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        KxU a;
                        if (VEC > 1) {
                            if (VEC == 2 && q == 1 && step(2, 2) && k + 2 < Nh) {
                                w = pair_mul_fx(b, fy[yy * 128 + row]);
                                w2 = kx_w(w, w);
                            }
                            const int m2 = VEC == 4 ? mm + 2 * q : mm;
                            const float4 h = fz[m2 * 128 + row], l = fz[(m2 + 1) * 128 + row];
                            a = KxU{f2_pack(h.x, h.y), f2_pack(h.z, h.w), f2_pack(l.x, l.y), f2_pack(l.z, l.w)};
                        } else {
                            if (q == 1 && step(2, 1) && k + 2 < Nh) w = pair_mul_fx(b, fy[yy * 128 + row]);
                            const float4 a0 = fz[mm * 128 + row], w0 = w;
                            if (step(2 * q + 1, 1) && k + 2 * q + 1 < Nh) w = pair_mul_fx(b, fy[yy * 128 + row]);
                            const float4 a1 = fz[mm * 128 + row];
                            w2 = kx_w(w0, w);
                            a = KxU{f2_pack(a0.x, a1.x), f2_pack(a0.y, a1.y), f2_pack(a0.z, a1.z), f2_pack(a0.w, a1.w)};
                        }
                        uint32_t dd[4][2];
                        kx_digits(kx_mul(w2, a), dd);
                        #pragma unroll
                        for (int i = 0; i < 4; ++i) {
                            d[i][2 * q] = dd[i][0];
                            d[i][2 * q + 1] = dd[i][1];
                        }
                    }
                    if (k + 4 > Nh) {             // elements past the last one
                        #pragma unroll
                        for (int e = 1; e < 4; ++e)
                            if (k + e >= Nh) d[0][e] = d[1][e] = d[2][e] = d[3][e] = 0u;
                    }
                }
                const uint32_t dst = ring + st * stage + arow;
                #pragma unroll
                for (int i = 0; i < 4; ++i) kx_sts(dst + i * (128 * KX_KC * 2), d[i][0], d[i][1], d[i][2], d[i][3]);
                tc::fence_async_smem();
                __syncwarp();
                if (lane == 0) kx_arrive(mfull + 8 * st);
                if (++st == nst) { st = 0; ++use; }
                // 16 elements on
                m += m_s;
                y += y_s;
                f += f_s;
                if (m >= Mz) { m -= Mz; ++y; }
                if (y >= My) { y -= My; ++f; }
            }
            if (!drained) epilogue(u - 1);
            pA = A;
            pDev = dev;
            ff_frac_mul2(grec.x, grec.y, G.inv_lam_hi, G.inv_lam_lo, pH0, pL0);
        }
        if (units > 0) {
            kx_bar();                             // the exchange of the last epilogue has been read
            epilogue(units - 1);
        }
        if (*sbad && lane == 0) atomicOr(D.kerr, KERR_TIMEOUT);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (warp == 0) tc::tmem_dealloc(tmem, ncols);
}

// ---------------------------------------------------------------- CUDA-core kernel
// The same closed form without the tensor cores (a tile request can ask for it): thread per
// particle, the columns eight at a time, each product split on a grid fixed per (s, j) so that
// the grid parts add exactly (2^E > 4 Nz bounds every partial sum of the scaled columns) and the
// remainders and low-part cross terms in FP32.  Issue bound: 24 instructions per complex product.
constexpr int KCC_T = 128, KCC_C = 8, KCC_E = 32;   // threads, columns per pass, staged elements

__global__ void __launch_bounds__(KCC_T) k_kappa_cc(DevGeom G, DevParams Pm, DevState D, int S, int SCA, int SW,
                                                    const double2* __restrict__ V64) {
    extern __shared__ float4 smc[];
    const int P = Pm.P, J = G.J, Nz = G.Nz, My = G.My, Mz = G.Mz, Nm = My * Mz, nant = My + Mz, K = S - 1;
    float4* fa = smc;                              // [nant][KCC_T]
    float4* ctab = fa + (size_t)nant * KCC_T;      // [256]
    float4* vs = ctab + 256;                       // [KCC_E][KCC_C] scaled columns (re, im hi; re, im lo)
    const int s = blockIdx.y, tid = threadIdx.x, p = blockIdx.x * KCC_T + tid, pp = min(p, P - 1);
    for (int i = tid; i < 256; i += KCC_T) ctab[i] = D.ctab[i];
    const float* ph = D.phi[D.cur] + (size_t)s * 6 * P;
    float GM = 1.5f;
    for (int v = 1; v < 4 * Nz; v *= 2) GM *= 2.0f;
    ff delta{0.f, 0.f};
    for (int j = 0; j < J; ++j) {
        const size_t sj = (size_t)s * J + j;
        const double2* V = V64 + sj * SCA * Nz;
        const float* scl = D.kSc + sj * 64;
        const double isq = 1.0 / sqrt(D.eta_bar[j]);
        const float4 grec = D.geo[sj * P + pp];
        const KxPath path = kx_path(G, grec, D.geo_lo[sj * P + pp]);
        __syncthreads();
        float dev = 0.f, sg = 0.f, sr = 0.f;
        for (int i = 0; i < nant; ++i) {
            const float4 a = kx_antenna(G, ctab, path, i);
            dev = fmaf((float)(i < My ? G.Nf * Mz : G.Nf * My), pair_unit_dev(make_float2(a.x, a.y), make_float2(a.z, a.w)), dev);
            fa[i * KCC_T + tid] = a;
        }
        cff pr{ff{0.f, 0.f}, ff{0.f, 0.f}};
        for (int c0 = 0; c0 < SW; c0 += KCC_C) {
            float ar[KCC_C], ai[KCC_C], lr[KCC_C], li[KCC_C];
            #pragma unroll
            for (int q = 0; q < KCC_C; ++q) ar[q] = ai[q] = lr[q] = li[q] = 0.f;
            float4 b = make_float4(0.f, 0.f, 0.f, 0.f), w = b;
            for (int k0 = 0; k0 < Nz; k0 += KCC_E) {
                const int nk = min(KCC_E, Nz - k0);
                __syncthreads();
                for (int t = tid; t < KCC_C * KCC_E; t += KCC_T) {
                    const int e = t % KCC_E, q = t / KCC_E, c = c0 + q;
                    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
                    const bool r0 = c == SW - 1;
                    if (e < nk && (r0 || c < K) && scl[c] != 0.f) {
                        const double f = (r0 ? 1.0 : isq) / (double)scl[c];
                        const double2 x = V[(size_t)(r0 ? SCA - 1 : c) * Nz + k0 + e];
                        v.x = (float)(x.x * f);
                        v.y = (float)(x.y * f);
                        v.z = (float)(x.x * f - (double)v.x);
                        v.w = (float)(x.y * f - (double)v.y);
                    }
                    vs[e * KCC_C + q] = v;
                }
                __syncthreads();
                for (int e = 0; e < nk; ++e) {
                    const int k = k0 + e, f = k / Nm, ym = k - f * Nm, y = ym / Mz, m = ym - y * Mz;
                    if (ym == 0 || e == 0) {
                        float2 hi, lo;
                        bprime_pair(G, ctab, path.dh, path.dl, path.h0, path.l0, f, hi, lo);
                        b = make_float4(hi.x, hi.y, lo.x, lo.y);
                        if (c0 == 0 && ym == 0) dev = fmaf((float)Nm, pair_unit_dev(hi, lo), dev);
                    }
                    if (m == 0 || e == 0) w = kx_pair_mul(b, fa[y * KCC_T + tid]);
                    const float4 u = kx_pair_mul(w, fa[(My + m) * KCC_T + tid]);
                    #pragma unroll
                    for (int q = 0; q < KCC_C; ++q) {
                        const float4 v = vs[e * KCC_C + q];
                        auto mac = [&](float& g, float& l, float x, float xl, float c, float cl) {
                            const float t = __fsub_rn(fmaf(x, c, GM), GM);
                            g = __fadd_rn(g, t);
                            l += fmaf(x, cl, fmaf(xl, c, fmaf(x, c, -t)));
                        };
                        mac(ar[q], lr[q], u.x, u.z, v.x, v.z);
                        mac(ar[q], lr[q], u.y, u.w, v.y, v.w);
                        mac(ai[q], li[q], u.x, u.z, v.y, v.w);
                        mac(ai[q], li[q], -u.y, -u.w, v.x, v.z);
                    }
                }
            }
            #pragma unroll
            for (int q = 0; q < KCC_C; ++q) {
                const int c = c0 + q;
                const float sc = scl[c];
                    cff h;
            two_sum(ar[q], lr[q], h.re.hi, h.re.lo);
            two_sum(ai[q], li[q], h.im.hi, h.im.lo);
            h = cff{ff_mulf(h.re, sc), ff_mulf(h.im, sc)};
                if (c == SW - 1) { pr = h; continue; }
                const float v[2] = {h.re.hi, h.im.hi}, vl[2] = {h.re.lo, h.im.lo};
                #pragma unroll
                for (int part = 0; part < 2; ++part) {
                    const float t = __fsub_rn(fmaf(v[part], v[part], GM), GM);
                    sg = __fadd_rn(sg, t);
                    sr += fmaf(2.0f * v[part], vl[part], fmaf(v[part], v[part], -t));
                }
            }
        }
        ff au;
        two_sum(__fsub_rn((float)Nz, sg), dev - sr, au.hi, au.lo);
        if (!(au.hi > 0.f)) au = ff{0.f, 0.f};
        delta = ff_add(delta, kx_delta(D.kC[sj], G.amp_c / (grec.x + grec.y), ph[3 * (size_t)P + pp],
                                       ph[4 * (size_t)P + pp], ph[5 * (size_t)P + pp], au, pr));
    }
    if (p < P) D.lw_y[(size_t)s * P + p] = ff_to_d(delta);
}

// the (hi, lo) cis table of the steering factors, once per handle
__global__ void k_cis_table(float4* tab) { cis_table_fill(tab, threadIdx.x, blockDim.x); }
void launch_cis_table(const DevState& D, cudaStream_t st) { k_cis_table<<<1, 256, 0, st>>>(D.ctab); }

size_t kappa_operand_bytes(const DevGeom& G, int S_max) {
    return (size_t)S_max * G.J * kx_chunks(kx_elements(G)) * kx_bbytes(kx_sw(S_max));
}

int launch_kappa(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, int SCA, bool tensor,
                 const double* V64, cudaStream_t st) {
    const int SW = kx_sw(S), nant = G.My + G.Mz;
    const double2* V = reinterpret_cast<const double2*>(V64);
    k_kappa_digits<<<dim3(S, G.J, KX_DSPLIT), 256, 0, st>>>(G, D, S, SCA, SW, V);
    if (!tensor) {
        const size_t smem = ((size_t)nant * KCC_T + 256 + KCC_E * KCC_C) * sizeof(float4);
        smem_allow_max((const void*)k_kappa_cc);
        k_kappa_cc<<<dim3((Pm.P + KCC_T - 1) / KCC_T, S), KCC_T, smem, st>>>(G, Pm, D, S, SCA, SW, V);
        return 2;
    }
    // Frequency factors in shared memory where several rows of four elements share one and a ring of
    // three slots still fits; else as many slots as fit, up to four (two always do: 128 KB of
    // ring and 80 KB of factors for the largest array and SW = 64)
    const size_t stage = KX_A + kx_bbytes(SW), limit = 227 * 1024;
    const int nant2 = G.My + ((G.Mz + 1) & ~1), Fh = kx_freqs(G);
    const int btab = G.My * G.Mz > 4 && kx_smem_fixed(nant2 + Fh) + 3 * stage <= limit;
    const size_t fixed = kx_smem_fixed(nant2 + (btab ? Fh : 0));
    int nst = KX_NST_MAX;
    while (nst > 2 && fixed + nst * stage > limit) --nst;
    const size_t smem = fixed + nst * stage;
    const int items = S * ((Pm.P + 127) / 128), grid = items < sm_count() ? items : sm_count();
    auto go = [&](auto kernel) {
        smem_allow_max((const void*)kernel);
        kernel<<<grid, KX_T, smem, st>>>(G, Pm, D, S, SW, nst, btab);
    };
    if (G.Mz % 4 == 0) go(k_kappa_x<4>);
    else if (G.Mz % 2 == 0) go(k_kappa_x<2>);
    else go(k_kappa_x<1>);
    return 2;
}

}  // namespace bp
