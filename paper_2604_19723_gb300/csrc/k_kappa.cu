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
// Precision on the tensor cores.  u (as a (hi, lo) FP32 pair, ~1e-10) and the columns of V~ and
// r0 (scaled by a power of two to just below 1) are written in fixed point as four signed
// base-256 digits of units 2^-7, 2^-15, 2^-23, 2^-31.  A digit has at most 8 bits, so it is exact
// in BF16, and a product of two digits is an integer multiple of its unit.  The FP32 accumulator of
// tcgen05.mma kind::f16 holds sums up to 2^24 of that unit exactly.  The products of the first digits
// reach 1.43 x 2^14 units per element where u and a column are aligned (nearly coinciding PFs, r0 of a strong
// one), that is 717 elements; beyond, the columns are scaled one or two powers of two lower
// (kx_headroom; without, 2048 elements left 0.3 nats on log ratios of 1e5 and 10 on those of PFs
// millimetres apart).  The second digits change sign along the array, and their sums stay lower.  The digit products (i, k) with i + k <= 5 (ten of
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
// instruction) onto g_{i-1} .. g_3.  One persistent block per SM: two teams of 256 producer threads fill
// every other A chunk (eight elements per thread, in registers, two per packed FP32 instruction), one
// warp copies the prebuilt B chunks, one issues the MMAs, and the producers read the accumulators of
// a finished (s, p tile, j) after they have refilled the ring with the next one's first chunks,
// so the tensor cores wait only for that read (not at all where two accumulator sets fit, SW <= 16).
// Up to SW = 32 A goes through the half of tensor memory that the accumulators leave free.
// Bound: the producers' issue slots (28 instructions per element for its digits; the factors, the loop and
// the epilogue add as much at few elements); the tensor pipe is next (ten products of 128 x 2 SW x 2 Nh:
// 44 % busy at 32 PFs, Nz = 1024).
// Measured (PF likelihood stage, J = 4) with the 3xTF32 kernel (below 33 PFs a CUDA-core kernel), which
// takes a second pass / with one thread issuing, A in shared memory and exact products by two-term
// splits of full FP32 factors / as it is: 64 PFs x 1e5 particles, Nz = 160: 56.7 / 15.6 / 10.3 ms; 32 PFs x
// 262144, Nz = 1024: 401 / 87 / 41 ms; 10 PFs x 30000, Nz = 160: 3.66 / 0.58 / 0.42 ms.
#include "bp_internal.cuh"
#include "bp_kernels.cuh"
#include "tc_sm100.cuh"

namespace bp {

constexpr int KX_WAIT = 1 << 20;       // polls of a bounded wait
constexpr int KX_NG = 4;               // producer groups (128 threads each), two to a team
constexpr int KX_PT = 128 * KX_NG;     // producer threads
constexpr int KX_T = KX_PT + 64;       // + the issuing and the copying warp
constexpr int KX_KC = 32;              // real K per chunk (16 elements)
constexpr int KX_A = 4 * 128 * KX_KC * 2;   // bytes of A per chunk: 4 digits x 128 rows x KX_KC BF16
constexpr int KX_NS_MAX = 4;           // slots of a ring
constexpr int KX_ACOL = 256;           // first TMEM column of A (TA): slots of 4 digits x KX_KC / 2 columns

__host__ __device__ inline int kx_sw(int S) { return (S + 7) & ~7; }
__host__ __device__ inline int kx_chunks(int Nh) { return (Nh + 15) / 16; }
__host__ __device__ inline uint32_t kx_bbytes(int SW) { return (uint32_t)(2 * SW) * KX_KC * 2 * 4; }   // 4 digits
// elements a particle forms: half of them where the layout is symmetric
__host__ __device__ inline int kx_elements(const DevGeom& G) { return G.sym ? (G.Nz + 1) / 2 : G.Nz; }
// Powers of two r between the largest part of a scaled column and 1.  For the first digits |u_1| <= 1 + sqrt(2)/256
// and |v_1| <= sqrt(2) (2^-r + 1/256), and Nh |u_1| |v_1| 2^14 is to stay below 2^24.  (The columns are
// rounded at 2^-32; beside the steering elements' 2^-31 the lost bits do not show: log ratios of 2048
// elements agree with the CUDA-core kernel's to 1e-4, as at r = 0.)
__host__ __device__ inline int kx_headroom(int Nh) { return Nh <= 717 ? 0 : Nh <= 1429 ? 1 : 2; }
__host__ __device__ inline int kx_factors(const DevGeom& G, int yz) {
    return yz ? (G.My * G.Mz + 1) & ~1 : G.My + ((G.Mz + 1) & ~1);
}
__host__ __device__ inline int kx_freqs(const DevGeom& G) { return (kx_elements(G) - 1) / (G.My * G.Mz) + 1; }
// shared memory after the ring: steering factors [nfac][128] as (hi, lo) pairs, cis table [256],
// partial sums [KX_NG][128], u^H r0 [128] (float4 each), column scales [3][64], barriers and flags
__host__ __device__ inline size_t kx_smem_fixed(int nfac) {
    return ((size_t)nfac * 128 + 256 + KX_NG * 128 + 128) * sizeof(float4) + 3 * 64 * sizeof(float) + 256;
}

// Steering factors as (h, l) with h a multiple of 2^-11 (12 bits) and |l| <= 2^-12 or so: the products of
// the h parts and their sums are exact in FP32 (multiples of 2^-22), the cross terms are small.
__device__ __forceinline__ void kx_grid(float hi, float lo, float& h, float& l) {
    const float M = 6144.0f;                    // 1.5 x 2^12
    h = __fsub_rn(__fadd_rn(__fadd_rn(hi, lo), M), M);
    l = __fadd_rn(__fsub_rn(hi, h), lo);
}
__device__ __forceinline__ float4 kx_split(float4 a) {
    float4 r;
    kx_grid(a.x, a.z, r.x, r.z);
    kx_grid(a.y, a.w, r.y, r.w);
    return r;
}
// (a + al)(b + bl) + (c + cl)(d + dl) of split factors: hi exact, |lo| below 2^-9
__device__ __forceinline__ void kx_dot(float a, float b, float c, float d, float al, float bl, float cl, float dl, float& hi, float& lo) {
    hi = fmaf(c, d, __fmul_rn(a, b));
    lo = fmaf(c, dl, fmaf(cl, d, fmaf(a, bl, fmaf(al, b, fmaf(cl, dl, __fmul_rn(al, bl))))));
}
__device__ __forceinline__ float4 kx_mul_split(float4 a, float4 b) {
    float4 u;
    kx_dot(a.x, b.x, -a.y, b.y, a.z, b.z, -a.w, b.w, u.x, u.z);
    kx_dot(a.x, b.y, a.y, b.x, a.z, b.w, a.w, b.z, u.y, u.w);
    return kx_split(u);
}
// the same, two elements at a time
struct KxW { f2x x, y, ny, xl, yl, nyl; };     // the outer factor of each of the two elements
struct KxU { f2x xh, yh, xl, yl; };
__device__ __forceinline__ KxW kx_w(float4 a, float4 b) {
    return KxW{f2_pack(a.x, b.x), f2_pack(a.y, b.y), f2_pack(-a.y, -b.y), f2_pack(a.z, b.z), f2_pack(a.w, b.w),
               f2_pack(-a.w, -b.w)};
}
__device__ __forceinline__ void kx_dot2(f2x a, f2x b, f2x c, f2x d, f2x al, f2x bl, f2x cl, f2x dl, f2x& hi, f2x& lo) {
    hi = f2_fma(c, d, f2_mul(a, b));
    lo = f2_fma(c, dl, f2_fma(cl, d, f2_fma(a, bl, f2_fma(al, b, f2_fma(cl, dl, f2_mul(al, bl))))));
}
__device__ __forceinline__ KxU kx_mul(const KxW& w, const KxU& a) {
    KxU u;
    kx_dot2(w.x, a.xh, w.ny, a.yh, w.xl, a.xl, w.nyl, a.yl, u.xh, u.xl);
    kx_dot2(w.x, a.yh, w.y, a.xh, w.xl, a.yl, w.yl, a.xl, u.yh, u.yl);
    return u;
}
// The four digits of two elements, digit i of element e in w[i][e] as the BF16 pair (Re, Im).  Adding 1.5 x
// 2^23 units rounds to a multiple of the unit, the remainder is exact; the low part joins after the
// first digit, where the remainder is below 2^-8 and the sum is good to 2^-33 (the second digit then
// reaches 160 at most, still exact).  The last digit is the remainder cut to BF16: at most 2^-31 off, as far as
// a rounded one of unit 2^-31, and its products only meet the last accumulator.
__device__ __forceinline__ void kx_digits(const KxU& u, uint32_t (&w)[4][2]) {
    const float M[3] = {98304.0f, 384.0f, 1.5f};   // 1.5 x 2^16, 2^8, 2^0
    f2x rx = u.xh, ry = u.yh;
    #pragma unroll
    for (int i = 0; i < 4; ++i) {
        f2x sx = rx, sy = ry;
        if (i < 3) {
            const f2x m = f2_dup(M[i]);
            sx = f2_sub(f2_add(rx, m), m);
            sy = f2_sub(f2_add(ry, m), m);
            rx = f2_sub(rx, sx);
            ry = f2_sub(ry, sy);
        }
        uint32_t x0, x1, y0, y1;
        f2_unpack(sx, x0, x1);
        f2_unpack(sy, y0, y1);
        w[i][0] = __byte_perm(x0, y0, 0x7632);     // upper halves: the digits are exact in BF16
        w[i][1] = __byte_perm(x1, y1, 0x7632);
        if (i == 0) { rx = f2_add(rx, u.xl); ry = f2_add(ry, u.yl); }
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

// antenna factor i < My: a_y, else a_z of element i - My, of a geometry record and its low parts, as a
// (hi, lo) pair (cis_pair, ~3e-11)
__device__ __forceinline__ float4 kx_antenna(const DevGeom& G, const float4* tab, float4 g, float2 gl, int i) {
    const bool y = i < G.My;
    const float c = y ? G.py_l[i] : G.pz_l[i - G.My], cl = y ? G.py_lo[i] : G.pz_lo[i - G.My];
    const float u = y ? g.z : g.w, ul = y ? gl.x : gl.y;
    const float p = __fmul_rn(c, u);
    const float e = fmaf(c, ul, fmaf(cl, u, fmaf(c, u, -p)));
    float2 hi, lo;
    cis_pair(tab, p, e, hi, lo);
    return make_float4(hi.x, hi.y, lo.x, lo.y);
}

// ---------------------------------------------------------------- operand digits of V~ and r0
// Block (s, j, part of the chunks): the columns' power-of-two scales (largest part in [1/2, 1)
// after scaling, less kx_headroom), then the four digit slices of its chunks of 16 elements as rows n < SW (Re h_n)
// and n >= SW (Im h_{n - SW}) against k = 2 e + part, K-major core matrices:
// [Re(v + v'), Im(v - v')] and [Im(v + v'), -Re(v - v')] for a symmetric layout (v' the mirrored
// element's, the middle element counted once), else [Re v, Im v] and [Im v, -Re v].  Column SW - 1
// is r0, unused columns are zero.  Bound: the FP64 conversions (64 PFs x 4 PAs x Nz = 160: 223 us with FP64
// maxima in four blocks per (s, j), 96 us with maxima of upper words and about four blocks per SM).
// With `whole` (the CUDA-core kernel's operand) the fixed-point numbers themselves go out instead of their
// digits, in units of 2^-29 of a column scaled to [1/2, 1): per chunk [16][SW] the factors of Re u and Im u
// in Re h, then in Im h.
__global__ void __launch_bounds__(256) k_kappa_digits(DevGeom G, DevState D, int S, int SCA, int SW, bool whole,
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
            uint32_t top = 0;                      // upper words of the magnitudes: the exponent decides
            #pragma unroll 4
            for (int k = lane; k < Nh; k += 32) {
                double o[4];
                combo(v, k, o);
                #pragma unroll
                for (int i = 0; i < 4; ++i) top = max(top, (uint32_t)__double2hiint(o[i]) & 0x7fffffffu);
            }
            top = __reduce_max_sync(0xffffffffu, top);
            // the next upper word bounds the largest magnitude
            const double m = top < 0x7ff00000u ? __hiloint2double((int)(top + 1), 0) * (r0 ? 1.0 : isq) : 0.0;
            if (!(m < INFINITY) || top >= 0x7ff00000u) {
                inv = NAN;                         // an observation that is not finite: neither are the log ratios
            } else if (top > 0 && m > 0.0) {
                int e;
                frexp(m, &e);
                e += kx_headroom(Nh);
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
            const double f = sc[c] * (whole ? ldexp(1.0, 29 + kx_headroom(Nh)) : 2147483648.0);
            #pragma unroll
            for (int i = 0; i < 4; ++i) q[i] = __double2ll_rn(o[i] * f);
            q[3] = -q[3];
        }
        if (whole) {
            reinterpret_cast<int4*>(out + (size_t)kc * 4 * slice)[e * SW + c] = make_int4((int)q[0], (int)q[1], (int)q[2], (int)q[3]);
            continue;
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

// The element factors split into an inner table and an outer factor: with yz the inner one is a_y a_z and the
// outer one the frequency's (see launch_kappa), else a_z and b_f a_y.  VEC: largest of 4, 2, 1 that
// divides the inner length (elements between possible changes of the outer factor).  btab: the
// frequency factors stay in shared memory (else they are formed where a row of elements begins).
// TA: A goes through tensor memory (two words per element and digit pair, the accumulators leave half of it
// free up to 32 columns of V~), else through shared memory.  nsa, nsb: slots of the A and the B ring.
template <int VEC, bool TA>
__global__ void __launch_bounds__(KX_T, 1) k_kappa_x(DevGeom G, DevParams Pm, DevState D, int S, int SW, int nsa, int nsb, int yz,
                                                     int btab) {
    extern __shared__ __align__(1024) unsigned char smx[];
    const int P = Pm.P, J = G.J, Nz = G.Nz, My = G.My, Mz = G.Mz, Nm = My * Mz, Nf = G.Nf;
    const int Nh = kx_elements(G), Fh = btab ? kx_freqs(G) : 0;
    const int N1 = 2 * SW, NCk = kx_chunks(Nh);
    const int Mi = yz ? Nm : Mz, Mo = yz ? 1 : My;                       // inner and outer elements of a frequency
    const int nfac = kx_factors(G, yz) + Fh;
    const uint32_t bbytes = kx_bbytes(SW), bring = TA ? 0 : nsa * KX_A;
    // steering factors of the 128 particles: a_y [My] without yz, the inner table (pairs of elements for
    // VEC > 1), b [Fh]
    float4* fy = reinterpret_cast<float4*>(smx + bring + (size_t)nsb * bbytes);
    float4* fz = fy + (size_t)(yz ? 0 : My) * 128;
    float4* fb = fz + (size_t)((Mi + 1) & ~1) * 128;
    float4* ctab = fy + (size_t)nfac * 128;                              // [256]
    float4* exs = ctab + 256;                                            // [KX_NG][128] |h|^2 (grid, rest), dev
    float4* exr = exs + KX_NG * 128;                                     // [128] u^H r0
    float* ssc = reinterpret_cast<float*>(exr + 128);                    // [3][64] column scales (unit mod 3: fetched one unit ahead, read one behind)
    uint64_t* mb = reinterpret_cast<uint64_t*>(ssc + 3 * 64);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(mb + 4 * KX_NS_MAX + 4);
    volatile int* sbad = reinterpret_cast<volatile int*>(tslot + 1);
    const uint32_t afull = tc::smem_u32(mb), aempty = afull + 8 * KX_NS_MAX;   // A slot filled; its MMAs done
    const uint32_t bfull = aempty + 8 * KX_NS_MAX, bempty = bfull + 8 * KX_NS_MAX;
    const uint32_t maccf = bempty + 8 * KX_NS_MAX, macce = maccf + 16;         // accumulator set complete; read
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int nacc = 8 * N1 <= (TA ? KX_ACOL : 512) ? 2 : 1;             // accumulator sets of 4 N1 columns
    uint32_t ncols = TA ? 512 : 32;
    while (ncols < (uint32_t)(nacc * 4 * N1)) ncols *= 2;
    if (warp == 0) tc::tmem_alloc(tslot, ncols);
    if (tid == 0) {
        for (int i = 0; i < KX_NS_MAX; ++i) {
            tc::mbar_init(afull + 8 * i, KX_PT / 64);        // the warps of the chunk's team
            tc::mbar_init(aempty + 8 * i, 1);
            tc::mbar_init(bfull + 8 * i, 1);
            tc::mbar_init(bempty + 8 * i, 1);
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
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tslot, 0);
    // a wait that gives up marks the block bad: nobody waits any more, every loop runs out
    auto wait = [&](uint32_t mbar, uint32_t parity) {
        if (tc::mbar_try(mbar, parity & 1u)) return true;
        for (int i = 0; i < KX_WAIT; ++i) {
            if (*sbad) return false;
            if (tc::mbar_try(mbar, parity & 1u)) return true;
        }
        *sbad = 1;
        return false;
    };
    const int ptiles = (P + 127) / 128, items = S * ptiles;
    const int nit = (int)blockIdx.x < items ? (items - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int units = nit * J;                   // (item, j) in order
    const uint32_t ring = tc::smem_u32(smx);
    if (warp == KX_PT / 32 + 1) {
        // ---- copying thread: the chunks of B, in order; those of an item are contiguous
        if (lane == 0) {
            int st = 0, use = 0, loaded = 0;
            bool ok = true;
            for (int it = 0; it < nit && ok; ++it) {
                const int s = (blockIdx.x + it * gridDim.x) / ptiles;
                const unsigned char* src = D.kB + (size_t)s * J * NCk * bbytes;
                for (int c = 0; c < J * NCk; ++c, src += bbytes) {
                    const uint32_t bar = bfull + 8 * st;
                    if (use > 0 && !(ok = wait(bempty + 8 * st, use - 1))) break;
                    tc::mbar_expect_tx(bar, bbytes);
                    tc::bulk_g2s(ring + bring + st * bbytes, src, bbytes, bar);
                    ++loaded;
                    if (++st == nsb) { st = 0; ++use; }
                }
            }
            // after a wait that gave up: let the copies in flight land (bounded)
            if (!ok || *sbad)
                for (int m = max(0, loaded - nsb); m < loaded; ++m) tc::mbar_wait(bfull + 8 * (m % nsb), (m / nsb) & 1, KX_WAIT);
        }
        __syncwarp();
    } else if (warp == KX_PT / 32) {
        // ---- issuing warp.  The MMAs take their descriptors from uniform registers: the loop is uniform over
        // the warp and one elected lane issues (a lane alone took ~180 clocks per MMA to move them)
        {
            // descriptors: the address is in the low word, which an offset leaves without a carry
            const uint64_t a0 = tc::smem_desc(ring, 128, KX_KC * 16), b0 = tc::smem_desc(ring + bring, 128, KX_KC * 16);
            const uint32_t hi = (uint32_t)(a0 >> 32);
            auto desc = [&](uint32_t lo) { return ((uint64_t)hi << 32) | lo; };
            // A's digit i against B's first 4 - i digit slices: at most 256 columns per MMA (a second part beyond 32
            // columns of V~ for the first digit, beyond 40 for the second)
            const uint32_t id0 = tc::idesc_bf16_f32(128, min(256, 4 * N1)), id1 = tc::idesc_bf16_f32(128, min(256, 3 * N1)),
                           id2 = tc::idesc_bf16_f32(128, 2 * N1), id3 = tc::idesc_bf16_f32(128, N1),
                           id02 = tc::idesc_bf16_f32(128, max(16, 4 * N1 - 256)), id12 = tc::idesc_bf16_f32(128, max(16, 3 * N1 - 256));
            const bool two1 = 3 * N1 > 256;
            int sa = 0, ua = 0, sb = 0, ub = 0, issued = 0;
            bool ok = true;
            // (every loop runs to its end, past a wait that gave up without issuing: it stays uniform)
            for (int u = 0; u < units; ++u) {
                const int set = nacc == 2 ? (u & 1) : 0, turn = nacc == 2 ? (u >> 1) : u;
                if (turn > 0) ok = __all_sync(0xffffffffu, ok && wait(macce + 8 * set, turn - 1));
                const uint32_t acc = tmem + (uint32_t)(set * 4 * N1), acc1 = acc + N1, acc2 = acc + 2 * N1, acc3 = acc + 3 * N1;
                for (int kc = 0; kc < NCk; ++kc) {
                    ok = __all_sync(0xffffffffu, ok && wait(bfull + 8 * sb, ub) && wait(afull + 8 * sa, ua));
                    tc::fence_after_sync();
                    const uint32_t da = (uint32_t)a0 + sa * (KX_A >> 4), db = (uint32_t)b0 + sb * (bbytes >> 4);
                    const uint32_t ts = tmem + KX_ACOL + sa * (2 * KX_KC);
                    if (ok && tc::elect_one()) {
                        #pragma unroll
                        for (int ks = 0; ks < KX_KC / 16; ++ks) {
                            const uint64_t b = desc(db + 16 * ks), b2 = desc(db + 16 * ks + 256 * KX_KC * 2 / 16);
                            auto mma = [&](int i, uint32_t col, uint64_t bd, uint32_t id, bool add) {
                                if constexpr (TA) tc::mma_bf16_ta(col, ts + i * (KX_KC / 2) + 8 * ks, bd, id, add);
                                else tc::mma_bf16(col, desc(da + i * (128 * KX_KC * 2 / 16) + 16 * ks), bd, id, add);
                            };
                            mma(0, acc, b, id0, kc > 0 || ks > 0);
                            if constexpr (!TA) mma(0, acc + 256, b2, id02, kc > 0 || ks > 0);
                            mma(1, acc1, b, id1, true);
                            if constexpr (!TA) if (two1) mma(1, acc1 + 256, b2, id12, true);
                            mma(2, acc2, b, id2, true);
                            mma(3, acc3, b, id3, true);
                        }
                        tc::mma_commit(aempty + 8 * sa);
                        tc::mma_commit(bempty + 8 * sb);
                        if (kc == NCk - 1) tc::mma_commit(maccf + 8 * set);
                    }
                    __syncwarp();
                    issued += ok ? 1 : 0;
                    if (++sa == nsa) { sa = 0; ++ua; }
                    if (++sb == nsb) { sb = 0; ++ub; }
                }
            }
            // after a wait that gave up: let the MMAs in flight land (bounded)
            if (!ok || *sbad)
                for (int m = max(0, issued - nsa); m < issued; ++m) tc::mbar_wait(aempty + 8 * (m % nsa), (m / nsa) & 1, KX_WAIT);
        }
        __syncwarp();
    } else {
        // ---- producers and epilogue
        const int grp = warp >> 2, row = tid & 127;
        const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const int team = grp >> 1, hh = grp & 1;  // a team fills every other chunk, eight elements per thread
        const uint32_t arow = (uint32_t)((row >> 3) * (KX_KC * 16) + (row & 7) * 16 + hh * 256);
        float GM = 1.5f;                          // grid of the |h|^2 sum: |h|^2 <= Nz
        for (int v = 1; v < 4 * Nz; v *= 2) GM *= 2.0f;
        // two chunks (32 elements) on, in (f, outer, inner)
        const int f_s = 32 / Nm, y_s = (32 - f_s * Nm) / Mi, m_s = 32 - f_s * Nm - y_s * Mi;
        float pA = 0.f, pDev = 0.f, pH0 = 0.f, pL0 = 0.f;   // previous unit: amplitude, |u|^2 - Nz (this group's part), carrier
        ff delta{0.f, 0.f};
        bool dead = false;                        // a wait gave up: nothing is stored or announced any more
        int e_it = -1, e_j = J - 1, e_s = 0, e_p = 0;   // item, PA, PF and particle of the epilogue's unit
        // reads the accumulators of unit u (in order), and one group per item evaluates Delta
        auto epilogue = [&](int u) {
            if (++e_j == J) {
                e_j = 0;
                ++e_it;
                const int item = blockIdx.x + e_it * gridDim.x;
                e_s = item / ptiles;
                e_p = (item - e_s * ptiles) * 128 + row;
            }
            const int it = e_it, j = e_j, s = e_s, p = e_p;
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
            if (!wait(maccf + 8 * set, use)) dead = true;
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
                        // g_0 + g_1 exactly (g_0, a multiple of 2^-14, is one of g_1's last place: |g_1| < 2^10), the
                        // rest onto the error
                        const f2x a = col2(0, q), b = col2(1, q), t = f2_add(a, b);
                        const f2x e = f2_add(f2_sub(b, f2_sub(t, a)), f2_add(col2(2, q), col2(3, q)));
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
            if (lane == 0 && !dead) kx_arrive(macce + 8 * set);
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
        int g_it = -1, g_j = J - 1, g_s = 0, g_p = 0;
        auto fetch = [&](int u) {                 // geometry record of unit u (in order)
            if (++g_j == J) {
                g_j = 0;
                ++g_it;
                const int item = blockIdx.x + g_it * gridDim.x;
                g_s = item / ptiles;
                g_p = (item - g_s * ptiles) * 128 + row;
            }
            const int j = g_j, s = g_s, p = g_p;
            const size_t gi = ((size_t)s * J + j) * P + min(p, P - 1);
            ngeo = D.geo[gi];
            ngl = D.geo_lo[gi];
            if (tid < 64) ssc[(u % 3) * 64 + tid] = tid < SW - 1 ? D.kSc[((size_t)s * J + j) * 64 + tid] : 0.f;
        };
        if (units > 0) fetch(0);
        int st = team, use = 0;                   // A slot and its turn of this team's next chunk (nsa >= 2)
        for (int u = 0; u < units; ++u) {
            const float4 grec = ngeo;
            const float2 grl = ngl;
            const float A = G.amp_c / (grec.x + grec.y);
            float dev = 0.f;
            auto cis = [&](float c, float e) {
                float2 hi, lo;
                cis_pair(ctab, c, e, hi, lo);
                return make_float4(hi.x, hi.y, lo.x, lo.y);
            };
            auto phase = [&](bool isz, int i, float& t, float& e) {
                const float c = isz ? G.pz_l[i] : G.py_l[i], cl = isz ? G.pz_lo[i] : G.py_lo[i];
                const float uu = isz ? grec.w : grec.z, ul = isz ? grl.y : grl.x;
                t = __fmul_rn(c, uu);
                e = fmaf(c, ul, fmaf(cl, uu, fmaf(c, uu, -t)));
            };
            auto inner = [&](int i) {             // a_z, or a_y a_z
                float t, e;
                if (!yz) {
                    phase(true, i, t, e);
                } else {
                    const int yi = i / Mz;
                    float t1, e1, t2, e2;
                    phase(false, yi, t1, e1);
                    phase(true, i - yi * Mz, t2, e2);
                    two_sum(t1, t2, t, e);
                    e += e1 + e2;
                }
                return cis(t, e);
            };
            auto conj4 = [](float4 a) { return make_float4(a.x, -a.y, a.z, -a.w); };
            auto put2 = [&](int m, float4 a, float4 b) {  // (hx, hx', hy, hy'), then the low parts
                fz[m * 128 + row] = make_float4(a.x, b.x, a.y, b.y);
                fz[(m + 1) * 128 + row] = make_float4(a.z, b.z, a.w, b.w);
            };
            auto freq = [&](int f) {              // b_f, without the carrier
                float h, l;
                ff_frac_mul2(grec.x, grec.y, G.fc_hi[f], G.fc_lo[f], h, l);
                return cis(-h, -l);
            };
            auto unit_dev = [&](float4 a) { return pair_unit_dev(make_float2(a.x, a.y), make_float2(a.z, a.w)); };
            const float fdup = G.sym ? 2.0f : 1.0f;
            kx_bar();                             // every group is done with the previous unit's factors
            // the antenna factors of a symmetric layout come in conjugate pairs: items of the inner table
            // (two elements each for VEC > 1), then a_y, then b
            constexpr int IV = VEC > 1 ? 2 : 1;
            const int nin = Mi / IV, hin = G.sym ? (nin + 1) / 2 : nin, hy = yz ? 0 : G.sym ? (My + 1) / 2 : My;
            const float win = (float)(Nf * Mo);
            for (int i = grp; i < hin + hy + Fh; i += KX_NG) {
                if (i < hin) {
                    const int m = IV * i, m2 = Mi - IV - m;       // the mirrored item
                    const float4 a = inner(m);
                    float d = unit_dev(a);
                    if (VEC > 1) {
                        const bool self = G.sym && m2 == m;
                        const float4 b = self ? conj4(a) : inner(m + 1);
                        d += unit_dev(b);
                        const float4 sa = kx_split(a), sb = kx_split(b);
                        put2(m, sa, sb);
                        if (G.sym && !self) { put2(m2, conj4(sb), conj4(sa)); d *= 2.0f; }
                    } else {
                        const float4 sa = kx_split(a);
                        fz[m * 128 + row] = sa;
                        if (G.sym && m2 != m) { fz[m2 * 128 + row] = conj4(sa); d *= 2.0f; }
                    }
                    dev = fmaf(win, d, dev);
                } else if (i < hin + hy) {
                    const int yi = i - hin, y2 = My - 1 - yi;
                    float t, e;
                    phase(false, yi, t, e);
                    const float4 a = cis(t, e), sa = kx_split(a);
                    const bool two = G.sym && y2 != yi;
                    fy[yi * 128 + row] = sa;
                    if (two) fy[y2 * 128 + row] = conj4(sa);
                    dev = fmaf((float)(Nf * Mz) * (two ? 2.0f : 1.0f), unit_dev(a), dev);
                } else {
                    // (the middle frequency is 0: no deviation)
                    const int f = i - hin - hy;
                    const float4 a = freq(f);
                    fb[f * 128 + row] = kx_split(a);
                    dev = fmaf((float)Nm * fdup, unit_dev(a), dev);
                }
            }
            kx_bar();
            if (u + 1 < units) fetch(u + 1);
            bool drained = u == 0;
            const int kc0 = team ^ (u & NCk & 1);  // this team's first chunk of the unit
            int f = (16 * kc0 + 8 * hh) / Nm, m = 16 * kc0 + 8 * hh - f * Nm, y = m / Mi;
            m -= y * Mi;
            for (int kc = kc0; kc < NCk; kc += 2) {
                // a slot of this unit's own ring turn frees only once the previous unit's
                // accumulators are read
                if (!drained && kc >= nsa) { epilogue(u - 1); drained = true; }
                const int k = 16 * kc + 8 * hh;
                uint32_t d[4][8];                 // [digit][element]
                if (k < Nh) {
                    int yy = y, mm = m, ff_ = f;
                    float4 b;
                    auto set_b = [&](int e) {
                        if (btab) { b = fb[ff_ * 128 + row]; return; }
                        b = freq(ff_);
                        const int cnt = min(min((ff_ + 1) * Nm, k + 8), Nh) - (k + e);
                        dev = fmaf((float)cnt * fdup, unit_dev(b), dev);
                        b = kx_split(b);
                    };
                    auto step = [&](int e, int by) {   // to element e (by elements on); true if the outer factor changed
                        mm += by;
                        if (mm < Mi) return false;
                        mm = 0;
                        if (++yy == Mo) {
                            yy = 0;
                            ++ff_;
                            if (k + e < Nh) set_b(e);
                        }
                        return k + e < Nh;
                    };
                    auto outer = [&]() { return yz ? b : kx_mul_split(b, fy[yy * 128 + row]); };
                    set_b(0);
                    float4 w = outer();
                    KxW w2;
                    if (VEC > 1) w2 = kx_w(w, w);
                    #pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        KxU a;
                        if (VEC > 1) {
                            const bool at = VEC == 4 ? q == 2 : q > 0;   // the outer factor may change here
                            if (at && step(2 * q, VEC)) {
                                w = outer();
                                w2 = kx_w(w, w);
                            }
                            const int m2 = VEC == 4 ? mm + 2 * (q & 1) : mm;
                            const float4 h = fz[m2 * 128 + row], l = fz[(m2 + 1) * 128 + row];
                            a = KxU{f2_pack(h.x, h.y), f2_pack(h.z, h.w), f2_pack(l.x, l.y), f2_pack(l.z, l.w)};
                        } else {
                            if (q > 0 && step(2 * q, 1)) w = outer();
                            const float4 a0 = fz[mm * 128 + row], w0 = w;
                            if (step(2 * q + 1, 1)) w = outer();
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
                    if (k + 8 > Nh) {             // elements past the last one
                        #pragma unroll
                        for (int e = 1; e < 8; ++e)
                            if (k + e >= Nh) d[0][e] = d[1][e] = d[2][e] = d[3][e] = 0u;
                    }
                } else {
                    #pragma unroll
                    for (int i = 0; i < 4; ++i)
                        #pragma unroll
                        for (int e = 0; e < 8; ++e) d[i][e] = 0u;
                }
                // the digits are formed before the slot is free, so that the wait costs little
                if (use > 0 && !wait(aempty + 8 * st, use - 1)) dead = true;
                if constexpr (TA) {
                    __syncwarp();
                    tc::fence_after_sync();
                    const uint32_t dst = tlane + KX_ACOL + st * (2 * KX_KC) + 8 * hh;
                    #pragma unroll
                    for (int i = 0; i < 4; ++i) tc::tmem_st8(dst + i * (KX_KC / 2), d[i]);
                    tc::tmem_st_wait();
                    tc::fence_before_sync();
                } else {
                    const uint32_t dst = ring + st * KX_A + arow;
                    #pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        kx_sts(dst + i * (128 * KX_KC * 2), d[i][0], d[i][1], d[i][2], d[i][3]);
                        kx_sts(dst + i * (128 * KX_KC * 2) + 128, d[i][4], d[i][5], d[i][6], d[i][7]);
                    }
                    tc::fence_async_smem();
                }
                __syncwarp();
                if (lane == 0 && !dead) kx_arrive(afull + 8 * st);
                st += 2;
                if (st >= nsa) { st -= nsa; ++use; }
                // two chunks on
                m += m_s;
                y += y_s;
                f += f_s;
                if (m >= Mi) { m -= Mi; ++y; }
                if (y >= Mo) { y -= Mo; ++f; }
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
// The same closed form without the tensor cores (a tile request can ask for it), in integers.  With the
// steering elements in units of 2^-30 and the columns of 2^-29 a sum of eight elements' products fits 64 bits
// exactly; every eight elements it is added, in units of 2^-47, to the column's running sum.
// Block: 64 particles of one PF, a warp per four columns, lane i the particles 2 i and 2 i + 1 (16 sums in
// registers).  While a chunk of 16 elements is multiplied, the next one's steering elements are formed (a
// thread per particle and row of Mz elements) and its columns fetched, in the other half of the
// buffers.  Bound: the integer multiply-adds (four per complex product) and the shared-memory reads of
// their operands.
// Measured (PF likelihood stage, J = 4, symmetric / general layout), and a thread per particle with the products as
// FP32 pairs over all elements: 10 PFs x 30000, Nz = 160: 1.19 / 2.21 ms (4.26); 64 x 20000: 22.6 / 40.3 (69.5);
// 32 x 20000, Nz = 1024: 29.0 / 56.9 (110).
constexpr int KCC_P = 64, KCC_E = 16, KCC_Q = 4;   // particles per block, elements per chunk, columns per warp
struct KccPlan { int quads, rows, dev; size_t smem; };
__host__ __device__ inline KccPlan kcc_plan(const DevGeom& G, int S) {
    KccPlan t;
    t.quads = (S + KCC_Q - 1) / KCC_Q;
    t.rows = (KCC_E - 1) / G.Mz + 2;               // rows of Mz elements that a chunk can touch
    t.dev = 2 * t.rows > G.My + G.Mz ? 2 * t.rows : G.My + G.Mz;
    t.smem = ((size_t)(G.My + G.Mz + 2) * KCC_P + 256 + 2 * (size_t)KCC_E * KCC_Q * t.quads) * sizeof(float4) +
             (2 * (size_t)KCC_E + t.quads + 1) * KCC_P * sizeof(float2) + (size_t)(t.dev + 1) * KCC_P * sizeof(float);
    return t;
}

__global__ void __launch_bounds__(32 * S_CAP_MAX / KCC_Q, 1) k_kappa_cc(DevGeom G, DevParams Pm, DevState D, int S, int SW) {
    extern __shared__ float4 smc[];
    const KccPlan pl = kcc_plan(G, S);
    const int P = Pm.P, J = G.J, Nz = G.Nz, My = G.My, Mz = G.Mz, Nm = My * Mz, nant = My + Mz, K = S - 1;
    const int Nh = kx_elements(G), NCk = kx_chunks(Nh), NC = KCC_Q * pl.quads;
    float4* fa = smc;                              // [nant][KCC_P] a_y, a_z, split
    float4* ctab = fa + (size_t)nant * KCC_P;      // [256]
    int4* vs = reinterpret_cast<int4*>(ctab + 256);   // [2][KCC_E][NC] factors of Re u and Im u in Re h, in Im h
    float4* sgeo = reinterpret_cast<float4*>(vs + 2 * (size_t)KCC_E * NC);   // [KCC_P]
    float4* exr = sgeo + KCC_P;                    // [KCC_P] u^H r0
    int2* us = reinterpret_cast<int2*>(exr + KCC_P);   // [2][KCC_E][KCC_P] u
    float2* ex = reinterpret_cast<float2*>(us + 2 * (size_t)KCC_E * KCC_P);  // [quads][KCC_P] |h|^2 (grid, rest)
    float2* sdl = ex + (size_t)pl.quads * KCC_P;   // [KCC_P] Delta over the PAs
    float* dv = reinterpret_cast<float*>(sdl + KCC_P);   // |.|^2 - 1: [nant][KCC_P] of factors, then [2][rows][KCC_P] of the rows' b_f
    float* sdv = dv + (size_t)pl.dev * KCC_P;      // [KCC_P] |u|^2 - Nz
    const int s = blockIdx.y, tid = threadIdx.x, T = blockDim.x, lane = tid & 31, quad = tid >> 5, p0 = blockIdx.x * KCC_P;
    for (int i = tid; i < 256; i += T) ctab[i] = D.ctab[i];
    const float* ph = D.phi[D.cur] + (size_t)s * 6 * P;
    const size_t chunk = kx_bbytes(SW);
    const float back = ldexpf(1.0f, -47 - kx_headroom(Nh)), dbl = G.sym ? 2.0f : 1.0f;
    float GM = 1.5f;
    for (int v = 1; v < 4 * Nz; v *= 2) GM *= 2.0f;
    for (int j = 0; j < J; ++j) {
        const size_t sj = (size_t)s * J + j;
        const unsigned char* B = D.kB + sj * NCk * chunk;
        const float* scl = D.kSc + sj * 64;
        __syncthreads();
        for (int t = tid; t < nant * KCC_P; t += T) {
            const int i = t / KCC_P, q = t % KCC_P;
            const size_t gi = sj * P + min(p0 + q, P - 1);
            const float4 grec = D.geo[gi];
            const float4 a = kx_antenna(G, ctab, grec, D.geo_lo[gi], i);
            dv[t] = (float)(i < My ? G.Nf * Mz : G.Nf * My) * pair_unit_dev(make_float2(a.x, a.y), make_float2(a.z, a.w));
            fa[t] = kx_split(a);
            if (i == 0) sgeo[q] = grec;
        }
        __syncthreads();
        for (int q = tid; q < KCC_P; q += T) {
            float d = 0.f;
            for (int i = 0; i < nant; ++i) d += dv[i * KCC_P + q];
            sdv[q] = d;
        }
        __syncthreads();
        // the steering elements (in units of 2^-30) and the columns of chunk kc
        auto fill = [&](int kc) {
            const int k0 = kc * KCC_E, k1 = min(k0 + KCC_E, Nh), r0 = k0 / Mz, nr = (k1 - 1) / Mz - r0 + 1;
            int2* u = us + (kc & 1) * KCC_E * KCC_P;
            float* d = dv + (kc & 1) * pl.rows * KCC_P;
            int4* v = vs + (kc & 1) * KCC_E * NC;
            const int4* src = reinterpret_cast<const int4*>(B + kc * chunk);
            for (int t = tid; t < KCC_E * NC; t += T) {
                const int e = t / NC, c = t - e * NC;
                v[t] = c < S ? src[e * SW + (c < K ? c : SW - 1)] : make_int4(0, 0, 0, 0);
            }
            for (int t = tid; t < nr * KCC_P; t += T) {
                const int r = r0 + t / KCC_P, q = t % KCC_P, f = r / My, y = r - f * My, ka = max(r * Mz, k0), kb = min(r * Mz + Mz, k1);
                const float4 g = sgeo[q];
                float h, l;
                float2 hi, lo;
                ff_frac_mul2(g.x, g.y, G.fc_hi[f], G.fc_lo[f], h, l);
                cis_pair(ctab, -h, -l, hi, lo);
                // once per frequency (a half-used middle frequency is 0: no deviation)
                d[t] = y == 0 && r * Mz >= k0 ? (float)Nm * dbl * pair_unit_dev(hi, lo) : 0.f;
                const float4 w = kx_mul_split(kx_split(make_float4(hi.x, hi.y, lo.x, lo.y)), fa[y * KCC_P + q]);
                for (int k = ka; k < kb; ++k) {
                    const float4 a = fa[(My + k - r * Mz) * KCC_P + q];
                    float4 x;
                    kx_dot(w.x, a.x, -w.y, a.y, w.z, a.z, -w.w, a.w, x.x, x.z);
                    kx_dot(w.x, a.y, w.y, a.x, w.z, a.w, w.w, a.z, x.y, x.w);
                    u[(k - k0) * KCC_P + q] = make_int2(__float2int_rn(x.x * 1073741824.0f) + __float2int_rn(x.z * 1073741824.0f),
                                                        __float2int_rn(x.y * 1073741824.0f) + __float2int_rn(x.w * 1073741824.0f));
                }
            }
            for (int t = tid + (k1 - k0) * KCC_P; t < KCC_E * KCC_P; t += T) u[t] = make_int2(0, 0);
        };
        long long tot[2][KCC_Q][2];
        #pragma unroll
        for (int i = 0; i < 2; ++i)
            #pragma unroll
            for (int q = 0; q < KCC_Q; ++q) tot[i][q][0] = tot[i][q][1] = 0;
        fill(0);
        __syncthreads();
        for (int kc = 0; kc < NCk; ++kc) {
            if (kc + 1 < NCk) fill(kc + 1);
            {   // deviations of this chunk's rows
                const int k0 = kc * KCC_E, nr = (min(k0 + KCC_E, Nh) - 1) / Mz - k0 / Mz + 1;
                const float* d = dv + (kc & 1) * pl.rows * KCC_P;
                for (int q = tid; q < KCC_P; q += T) {
                    float v = sdv[q];
                    for (int r = 0; r < nr; ++r) v += d[r * KCC_P + q];
                    sdv[q] = v;
                }
            }
            const int2* u2 = us + (kc & 1) * KCC_E * KCC_P + 2 * lane;
            const int4* v2 = vs + (kc & 1) * KCC_E * NC + quad * KCC_Q;
            #pragma unroll 1
            for (int half = 0; half < 2; ++half) {
                long long acc[2][KCC_Q][2];
                #pragma unroll
                for (int i = 0; i < 2; ++i)
                    #pragma unroll
                    for (int q = 0; q < KCC_Q; ++q) acc[i][q][0] = acc[i][q][1] = 0;
                #pragma unroll 2
                for (int e = 0; e < KCC_E / 2; ++e) {
                    const int4 u = *reinterpret_cast<const int4*>(u2 + (half * (KCC_E / 2) + e) * KCC_P);
                    #pragma unroll
                    for (int q = 0; q < KCC_Q; ++q) {
                        const int4 v = v2[(half * (KCC_E / 2) + e) * NC + q];
                        acc[0][q][0] += (long long)u.x * v.x + (long long)u.y * v.y;
                        acc[0][q][1] += (long long)u.x * v.z + (long long)u.y * v.w;
                        acc[1][q][0] += (long long)u.z * v.x + (long long)u.w * v.y;
                        acc[1][q][1] += (long long)u.z * v.z + (long long)u.w * v.w;
                    }
                }
                #pragma unroll
                for (int i = 0; i < 2; ++i)
                    #pragma unroll
                    for (int q = 0; q < KCC_Q; ++q) {
                        tot[i][q][0] += acc[i][q][0] >> 12;
                        tot[i][q][1] += acc[i][q][1] >> 12;
                    }
            }
            __syncthreads();
        }
        #pragma unroll
        for (int i = 0; i < 2; ++i) {
            float sg = 0.f, sr = 0.f;
            #pragma unroll
            for (int q = 0; q < KCC_Q; ++q) {
                const int c = quad * KCC_Q + q;
                if (c >= S) break;
                const float sc = scl[c < K ? c : SW - 1];
                float hi[2], lo[2];
                #pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const float t = __ll2float_rn(tot[i][q][v]);
                    hi[v] = t * back * sc;
                    lo[v] = __ll2float_rn(tot[i][q][v] - __float2ll_rn(t)) * back * sc;
                }
                if (c == K) { exr[2 * lane + i] = make_float4(hi[0], hi[1], lo[0], lo[1]); continue; }
                #pragma unroll
                for (int v = 0; v < 2; ++v) {
                    const float t = __fsub_rn(fmaf(hi[v], hi[v], GM), GM);
                    sg = __fadd_rn(sg, t);
                    sr += fmaf(2.0f * hi[v], lo[v], fmaf(hi[v], hi[v], -t));
                }
            }
            ex[quad * KCC_P + 2 * lane + i] = make_float2(sg, sr);
        }
        __syncthreads();
        for (int q = tid; q < KCC_P; q += T) {
            const int p = p0 + q, pp = min(p, P - 1);
            float sg = 0.f, sr = 0.f;
            for (int c = 0; c < pl.quads; ++c) {
                sg = __fadd_rn(sg, ex[c * KCC_P + q].x);   // multiples of the grid: exact
                sr += ex[c * KCC_P + q].y;
            }
            ff au;
            two_sum(__fsub_rn((float)Nz, sg), sdv[q] - sr, au.hi, au.lo);
            if (!(au.hi > 0.f)) au = ff{0.f, 0.f};
            const float4 g = sgeo[q], r = exr[q];
            float h0, l0;                          // the carrier: conj(e^{-i 2 pi d / lambda})
            ff_frac_mul2(g.x, g.y, G.inv_lam_hi, G.inv_lam_lo, h0, l0);
            float2 ch, cl;
            cis_pair(ctab, h0, l0, ch, cl);
            const cff pr = cff_mul(cff{ff{r.x, r.z}, ff{r.y, r.w}}, cff{ff{ch.x, cl.x}, ff{ch.y, cl.y}});
            const ff d = kx_delta(D.kC[sj], G.amp_c / (g.x + g.y), ph[3 * (size_t)P + pp], ph[4 * (size_t)P + pp],
                                  ph[5 * (size_t)P + pp], au, pr);
            const ff all = j == 0 ? d : ff_add(ff{sdl[q].x, sdl[q].y}, d);
            sdl[q] = make_float2(all.hi, all.lo);
            if (j == J - 1 && p < P) D.lw_y[(size_t)s * P + p] = ff_to_d(all);
        }
    }
}

// the (hi, lo) cis table of the steering factors, once per handle
__global__ void k_cis_table(float4* tab) { cis_table_fill(tab, threadIdx.x, blockDim.x); }
void launch_cis_table(const DevState& D, cudaStream_t st) { k_cis_table<<<1, 256, 0, st>>>(D.ctab); }

size_t kappa_operand_bytes(const DevGeom& G, int S_max) {
    return (size_t)S_max * G.J * kx_chunks(kx_elements(G)) * kx_bbytes(kx_sw(S_max));
}

int launch_kappa(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, int SCA, bool tensor,
                 const double* V64, cudaStream_t st) {
    const int SW = kx_sw(S);
    const double2* V = reinterpret_cast<const double2*>(V64);
    k_kappa_digits<<<dim3(S, G.J, max(1, min(4, 4 * sm_count() / (S * G.J)))), 256, 0, st>>>(G, D, S, SCA, SW, !tensor, V);
    if (!tensor) {
        const KccPlan t = kcc_plan(G, S);
        smem_allow_max((const void*)k_kappa_cc);
        k_kappa_cc<<<dim3((Pm.P + KCC_P - 1) / KCC_P, S), 32 * t.quads, t.smem, st>>>(G, Pm, D, S, SW);
        return 2;
    }
    // Up to 32 columns A goes through tensor memory: MMAs of few columns are bound by reading A from shared
    // memory there (128 x 256, 192, 128 and 64 columns: 333 clocks against 320 of tensor memory; 64, 48,
    // 32 and 16: 172 against 82), and the ring leaves room for the frequency factors.
    // The inner table holds a_y a_z where at least eight frequencies use it (its My Mz / 2 sincos per
    // particle against a product of pairs per four elements); the frequency factors stay in shared
    // memory where more than four elements share one.  Both only where two slots of each ring still fit,
    // and without them two always do (128 KB of rings and 80 KB of factors for the largest array and
    // SW = 64); the rings take what is left, up to four slots, A's first (its turn-around is longer).
    const bool ta = SW <= 32;
    const size_t asl = ta ? 0 : KX_A, bsl = kx_bbytes(SW), limit = 227 * 1024;
    const int Nm = G.My * G.Mz, Fh = kx_freqs(G);
    auto fits = [&](int yz, int fb) { return kx_smem_fixed(kx_factors(G, yz) + fb) + 2 * (asl + bsl) <= limit; };
    const int yz = G.Nf >= 8 && fits(1, Nm > 4 ? Fh : 0);
    const int btab = Nm > 4 && fits(yz, Fh);
    const size_t fixed = kx_smem_fixed(kx_factors(G, yz) + (btab ? Fh : 0));
    int nsa = KX_NS_MAX, nsb = KX_NS_MAX;
    if (!ta) nsb = 2;
    while (nsb > 2 && fixed + nsb * bsl > limit) --nsb;
    while (nsa > 2 && fixed + nsa * asl + nsb * bsl > limit) --nsa;
    while (nsb < KX_NS_MAX && fixed + nsa * asl + (nsb + 1) * bsl <= limit) ++nsb;
    const size_t smem = fixed + nsa * asl + nsb * bsl;
    const int items = S * ((Pm.P + 127) / 128), grid = items < sm_count() ? items : sm_count();
    auto go = [&](auto kernel) {
        smem_allow_max((const void*)kernel);
        kernel<<<grid, KX_T, smem, st>>>(G, Pm, D, S, SW, nsa, nsb, yz, btab);
    };
    const int Mi = yz ? Nm : G.Mz;
    if (Mi % 4 == 0) ta ? go(k_kappa_x<4, true>) : go(k_kappa_x<4, false>);
    else if (Mi % 2 == 0) ta ? go(k_kappa_x<2, true>) : go(k_kappa_x<2, false>);
    else ta ? go(k_kappa_x<1, true>) : go(k_kappa_x<1, false>);
    return 2;
}

}  // namespace bp
