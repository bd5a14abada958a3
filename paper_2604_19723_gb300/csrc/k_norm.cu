// Beliefs, normalisation, estimates, pruning, resampling, regularisation.
//   Sec. IV-D "Beliefs" / Sec. S-III: log w~ = log w_pred + sum_j log(message).
//   Sec. S-IV: C_y,s = sum_p w~_y,s + (1 - W_s) prod_j kappa~(., 0); the PF
//   log-likelihoods here are already relative to prod_j kappa~(., 0), so the
//   null term is log(1 - W_s).  FP64 log-sum-exp throughout.
//   Sec. II-C: MMSE estimates, declaration, pruning (never the LoS).
//   Systematic resampling (Arulampalam et al. 2002, Alg. 2) and Gaussian
//   kernel regularisation with h_opt = (4/(P(d+2)))^(1/(d+4)) (Musso et al. 2001).
#include "bp_internal.cuh"
#include "bp_kernels.cuh"

namespace bp {

// log weight of particle p in belief b, and a pointer to its state dims
struct BeliefView {
    int kind;       // 0 MT, 1 PF, 2 eta
    int index;      // s or j
    int dims;       // 6 or 1
};

__device__ inline BeliefView belief_of(int b, const DevParams& Pm, int J) {
    if (b == 0) return BeliefView{0, 0, 6};
    if (b <= Pm.S_max) return BeliefView{1, b - 1, 6};
    return BeliefView{2, b - 1 - Pm.S_max, 1};
}

// prediction weights, log-likelihoods and (in turn) log weights / normalised weights of a belief
__device__ inline const double* belief_w(const DevState& D, const BeliefView& v, int P) {
    return v.kind == 0 ? D.w_x : (v.kind == 1 ? D.w_alpha : D.w_eta) + (size_t)v.index * P;
}
__device__ inline const double* belief_l(const DevState& D, const BeliefView& v, int P) {
    return v.kind == 0 ? D.lw_x : (v.kind == 1 ? D.lw_y : D.lw_eta) + (size_t)v.index * P;
}
__device__ inline double* belief_wn(const DevState& D, const BeliefView& v, int P) {
    return v.kind == 0 ? D.wn_x : (v.kind == 1 ? D.wn_y : D.wn_eta) + (size_t)v.index * P;
}

__device__ inline void belief_state(const DevState& D, const BeliefView& v, int P, int p, double* out) {
    if (v.kind == 0) {
        const float* x = D.x[D.cur];
        for (int k = 0; k < 6; ++k) out[k] = x[(size_t)k * P + p];
    } else if (v.kind == 1) {
        const float* ph = D.phi[D.cur] + (size_t)v.index * 6 * P;
        for (int k = 0; k < 6; ++k) out[k] = ph[(size_t)k * P + p];
    } else {
        out[0] = D.eta[D.cur][(size_t)v.index * P + p];
    }
}

// active beliefs: b in {0} U {1..S} U {1+S_max .. S_max+J}
__device__ inline int active_belief(int a, int S, int S_max) { return a <= S ? a : 1 + S_max + (a - S - 1); }

// log weights of every particle (kept in the buffer of the normalised weights) and the block
// maxima.  FP64 logarithms set the time here (GB300 issues FP64 at 1/64 of the FP32 rate): after
// resampling a belief's weights are all equal, so the logarithm of a block's first weight serves
// every particle that has the same one.
__global__ void k_norm_max(DevGeom G, DevParams Pm, DevState D, int S, int NB) {
    const int b = active_belief(blockIdx.y, S, Pm.S_max);
    const BeliefView v = belief_of(b, Pm, G.J);
    const int P = Pm.P;
    const int per = (P + NB - 1) / NB;
    const int p0 = blockIdx.x * per, p1 = min(P, p0 + per);
    const double *w = belief_w(D, v, P), *l = belief_l(D, v, P);
    double* o = belief_wn(D, v, P);
    double m = -INFINITY;
    if (p0 < p1) {
        const double w0 = w[p0], lw0 = log(w0);
        for (int p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
            const double wp = w[p];
            const double t = (wp == w0 ? lw0 : log(wp)) + l[p];
            o[p] = t;
            m = fmax(m, t);
        }
    }
    __shared__ double red[32];
    m = warp_max_d(m);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        double t = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : -INFINITY;
        t = warp_max_d(t);
        if (threadIdx.x == 0) D.red_part[((size_t)b * NB + blockIdx.x) * RED_W] = t;
    }
}

// Weights more than NORM_SKIP nats below the largest are left out of the sums: P e^-60 < 2^-53 for
// every P this library takes, so they are below the rounding of a sum that is at least 1.
constexpr double NORM_SKIP = 60.0;
__global__ void k_norm_sum(DevGeom G, DevParams Pm, DevState D, int S, int NB, double* part) {
    const int b = active_belief(blockIdx.y, S, Pm.S_max);
    const BeliefView v = belief_of(b, Pm, G.J);
    const int P = Pm.P;
    double M = -INFINITY;
    for (int i = 0; i < NB; ++i) M = fmax(M, D.red_part[((size_t)b * NB + i) * RED_W]);
    double ref[6];
    belief_state(D, v, P, 0, ref);
    const int per = (P + NB - 1) / NB;
    const int p0 = blockIdx.x * per, p1 = min(P, p0 + per);
    const double* lw = belief_wn(D, v, P);
    double acc[32];
    #pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0;
    const int d = v.dims;
    if (M > -INFINITY) {
        for (int p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
            const double t = lw[p] - M;
            if (t < -NORM_SKIP) continue;
            const double w = exp(t);
            double xs[6];
            belief_state(D, v, P, p, xs);
            acc[0] += w;
            acc[28] += w * w;
            if (d == 1) {
                const double x = xs[0] - ref[0];
                acc[1] += w * x;
                acc[7] += w * x * x;
                continue;
            }
            #pragma unroll
            for (int k = 0; k < 6; ++k) {
                xs[k] -= ref[k];
                acc[1 + k] += w * xs[k];
            }
            int q = 7;
            #pragma unroll
            for (int r = 0; r < 6; ++r)
                #pragma unroll
                for (int c = r; c < 6; ++c) acc[q++] += w * xs[r] * xs[c];
        }
    }
    __shared__ double red[32][RED_W + 1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // the sums of a warp all at once: halving the values while the lanes pair up (31 FP64 additions instead of
    // 145; lane i ends with the i-th sum).  An idle warp's are zero.
    if (__any_sync(0xffffffffu, acc[0] != 0.0)) {
        #pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const bool up = lane & o;
            #pragma unroll
            for (int i = 0; i < o; ++i) {
                const double keep = up ? acc[i + o] : acc[i], give = up ? acc[i] : acc[i + o];
                acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
            }
        }
    }
    if (lane < RED_W) red[wid][lane] = acc[0];
    __syncthreads();
    if (threadIdx.x < RED_W) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w][threadIdx.x];
        part[((size_t)b * NB + blockIdx.x) * RED_W + threadIdx.x] = s;
    }
}

__device__ inline void mt_mask(const DevParams& Pm, bool* a) {
    for (int k = 0; k < 6; ++k) a[k] = true;
    if (Pm.motion_dims == 2) { a[2] = false; a[5] = false; }
}
__device__ inline void pf_mask(const DevParams& Pm, int s, bool* a) {
    for (int k = 0; k < 6; ++k) a[k] = true;
    if (s == 0) { a[0] = a[1] = a[2] = false; }
    else if (Pm.motion_dims == 2) a[2] = false;
    if (Pm.zero_mean) { a[4] = a[5] = false; }
}

// two warps per active belief: the first combines the partials (lane i the i-th sum, in block order), then its
// lane 0 forms the normaliser while the second forms mean, covariance and the jitter factor, lanes over
// their rows (one lane for everything took 36 us against 13, most of it FP64 square roots and divisions in turn)
__global__ void __launch_bounds__(64) k_norm_final(DevGeom G, DevParams Pm, DevState D, int S, int NB, const double* part) {
    const int b = active_belief(blockIdx.x, S, Pm.S_max);
    const BeliefView v = belief_of(b, Pm, G.J);
    const int P = Pm.P, lane = threadIdx.x & 31;
    __shared__ double acc[RED_W], Cs[6][6];
    double M = -INFINITY;
    if (threadIdx.x < 32) {
        for (int i = lane; i < NB; i += 32) M = fmax(M, D.red_part[((size_t)b * NB + i) * RED_W]);
        M = warp_max_d(M);
        if (lane < RED_W) {
            double t = 0.0;
            #pragma unroll 4
            for (int i = 0; i < NB; ++i) t += part[((size_t)b * NB + i) * RED_W + lane];
            acc[lane] = t;
        }
    }
    __syncthreads();
    double* rec = D.bel + bel_rec(Pm.S_max, G.J, b);
    if (threadIdx.x < 32) {
        if (lane != 0) return;
        const double lse = (acc[0] > 0) ? M + log(acc[0]) : -INFINITY;
        double logC = lse;
        if (v.kind == 1) {
            const double W = D.W[v.index];
            const double ln = (W < 1.0) ? log1p(-W) : -INFINITY;
            const double mx = fmax(lse, ln);
            logC = (mx == -INFINITY) ? -INFINITY : mx + log(exp(lse - mx) + exp(ln - mx));
            const double ps = (logC == -INFINITY) ? 0.0 : exp(lse - logC);
            D.p_s[v.index] = ps;
        }
        rec[0] = M; rec[1] = lse; rec[2] = logC;
        rec[3] = (acc[0] > 0) ? acc[28] / (acc[0] * acc[0]) : 1.0;   // sum of squared normalised weights
        return;
    }
    const int d = v.dims;
    const bool some = acc[0] > 0;
    double ref[6];
    belief_state(D, v, P, 0, ref);
    // lane k < 6: component k of the mean; lane t < 21: entry (r, c) of the covariance (active dimensions only)
    double mean = 0.0;
    if (some && lane < d) mean = acc[1 + lane] / acc[0];
    bool act[6];
    if (v.kind == 0) mt_mask(Pm, act);
    else if (v.kind == 1) pf_mask(Pm, v.index, act);
    else { act[0] = true; for (int k = 1; k < 6; ++k) act[k] = false; }
    int dact = 0;
    for (int k = 0; k < d; ++k) if (act[k]) ++dact;
    int r = 0, c = lane;
    while (r < 5 && c >= 6 - r) { c -= 6 - r; ++r; }
    c += r;
    c = min(c, 5);
    const double mr = __shfl_sync(0xffffffffu, mean, r), mc = __shfl_sync(0xffffffffu, mean, c);
    if (lane < 21) {
        bool on = some && r < d && c < d;
        for (int k = 0; k < 6; ++k) if ((k == r || k == c) && !act[k]) on = false;
        Cs[r][c] = Cs[c][r] = on ? acc[d == 1 ? 7 : 7 + lane] / acc[0] - mr * mc : 0.0;
    }
    double rk = 0.0;
    #pragma unroll
    for (int k = 0; k < 6; ++k) if (k == lane && k < d) rk = ref[k];
    if (lane < 6) rec[4 + lane] = lane < d ? (some ? mean + rk : 0.0) : 0.0;
    __syncwarp();
    // Cholesky factor, lane i its row i (columns of non-positive pivots stay zero); h_opt L goes out
    const int row = min(lane, 5);
    double Lr[6] = {0, 0, 0, 0, 0, 0};
    #pragma unroll
    for (int k = 0; k < 6; ++k) {
        double x = Cs[row][k];
        #pragma unroll
        for (int m = 0; m < k; ++m) x -= Lr[m] * __shfl_sync(0xffffffffu, Lr[m], k);
        const double piv = __shfl_sync(0xffffffffu, x, k);
        if (k < d && piv > 0.0) {                 // uniform
            const double lk = sqrt(piv);
            if (lane == k) Lr[k] = lk;
            else if (lane > k && lane < d) Lr[k] = x / lk;
        }
    }
    const double h = Pm.h_opt[dact];
    float* Lf = D.Lchol + (size_t)b * 36;
    if (lane < 6) {
        #pragma unroll
        for (int k = 0; k < 6; ++k) Lf[lane * 6 + k] = (float)((Pm.regularize ? h : 0.0) * Lr[k]);
    }
    if (lane == 0) rec[10] = dact;
}

// estimates, declaration, pruning map: a thread per PF, the survivors numbered by ballot
__global__ void __launch_bounds__(S_CAP_MAX) k_estimate(DevGeom G, DevParams Pm, DevState D, int S) {
    const int J = G.J, SM = Pm.S_max, s = threadIdx.x, lane = s & 31;
    const EstLayout E{SM, J};
    double* est = D.est;
    bool kept = false;
    if (s < S) {
        const double* rs = D.bel + bel_rec(SM, J, 1 + s);
        const double ps = D.p_s[s];
        est[E.p_s() + s] = ps;
        for (int k = 0; k < 6; ++k) est[E.phi_hat() + 6 * s + k] = rs[4 + k];
        double prod = 1.0;
        for (int j = 0; j < J; ++j) {
            const double pr = D.bel[BEL_PPR + s * J + j];
            est[E.p_pr() + s * J + j] = pr;
            prod *= (1.0 - pr);
        }
        const double pany = 1.0 - prod;
        est[E.p_any() + s] = pany;
        est[E.declared() + s] = (ps > Pm.T_dec) ? 1.0 : 0.0;
        kept = (s == 0) || Pm.T_pru <= 0.0 || !(ps < Pm.T_pru || pany < Pm.T_pru);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, kept);
    __shared__ int first;
    if (s == 0) first = __popc(bal);
    __syncthreads();
    const int at = __popc(bal & ((1u << lane) - 1u)) + (s >= 32 ? first : 0);
    if (kept) D.ctrl[4 + at] = s;
    if (s == S_CAP_MAX - 1) {
        const int keep = at + (kept ? 1 : 0);
        D.ctrl[1] = keep;
        est[E.S_next()] = keep;
    }
    if (s < J) est[E.eta_hat() + s] = (D.bel + bel_rec(SM, J, 1 + SM + s))[4];
    if (s != 0) return;
    const double* r0 = D.bel + bel_rec(SM, J, 0);
    est[E.n()] = D.step[0];
    est[E.S()] = S;
    est[E.repaired()] = D.flags[0];
    for (int k = 0; k < 6; ++k) est[E.x_hat() + k] = r0[4 + k];
    est[E.ess()] = 1.0 / r0[3];
    est[E.skipped()] = D.ctrl[2];
    int status = 0;
    if (!(r0[2] > -INFINITY)) status = BP_ERR_NUMERIC;
    // a NaN or Inf in z reaches |e|^2 of its PA first; report it as such
    for (int j = 0; j < J; ++j)
        if (!isfinite(D.nu_c[2 * j])) status = EST_STATUS_BAD_Z;
    est[E.status()] = status;
    D.ctrl[3] = status;
}

// particles per tile of the cumulative weights (at most CDF_TILES tiles) and the tile count
constexpr int CDF_SUB = 2048, CDF_TILES = 256;
__host__ __device__ inline int cdf_tile(int P) { return CDF_SUB * ((P + CDF_SUB * CDF_TILES - 1) / (CDF_SUB * CDF_TILES)); }
__host__ __device__ inline int cdf_tiles(int P) { return (P + cdf_tile(P) - 1) / cdf_tile(P); }
// block sum in a fixed order, in every thread
__device__ inline double block_sum_256(double v, double* red) {
    v = warp_sum_d(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.0;
    #pragma unroll
    for (int w = 0; w < 8; ++w) v += red[w];
    return v;
}

// normalised weights of every active belief (before resampling), in place of the log weights, and
// their tile sums
__global__ void __launch_bounds__(256) k_norm_weights(DevGeom G, DevParams Pm, DevState D, int S, double* tsum) {
    const int P = Pm.P;
    const int b = active_belief(blockIdx.y, S, Pm.S_max);
    const BeliefView v = belief_of(b, Pm, G.J);
    const double logC = (D.bel + bel_rec(Pm.S_max, G.J, b))[2];
    double* w = belief_wn(D, v, P);
    const int tile = cdf_tile(P), p0 = blockIdx.x * tile, p1 = min(P, p0 + tile);
    double acc = 0.0;
    for (int p = p0 + threadIdx.x; p < p1; p += 256) {
        const double t = w[p] - logC;
        // e^t is 0 in FP64 below -745.2
        const double e = (logC > -INFINITY) ? (t < -746.0 ? 0.0 : exp(t)) : 0.0;
        w[p] = e;
        acc += e;
    }
    __shared__ double red[8];
    acc = block_sum_256(acc, red);
    if (threadIdx.x == 0) tsum[(size_t)b * CDF_TILES + blockIdx.x] = acc;
}

int launch_normalize(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, cudaStream_t st) {
    const int P = Pm.P;
    int NB = (P + 2047) / 2048;
    if (NB > 64) NB = 64;
    const int nb = 1 + S + G.J;
    double* part = D.red_part + (size_t)bel_count(Pm.S_max, G.J) * 64 * RED_W;
    k_norm_max<<<dim3(NB, nb), 256, 0, st>>>(G, Pm, D, S, NB);
    k_norm_sum<<<dim3(NB, nb), 256, 0, st>>>(G, Pm, D, S, NB, part);
    k_norm_final<<<nb, 64, 0, st>>>(G, Pm, D, S, NB, part);
    k_estimate<<<1, S_CAP_MAX, 0, st>>>(G, Pm, D, S);
    k_norm_weights<<<dim3(cdf_tiles(P), nb), 256, 0, st>>>(G, Pm, D, S, D.tsum);
    return 5;
}

// ---------------------------------------------------------------- systematic resampling
// belief of resampling slot a: the MT, the kept PFs in their new order, then eta; false if idle
struct ResampleSlot { int b, kind, index; };
__device__ inline bool resample_slot(const DevParams& Pm, const DevState& D, int J, int a, ResampleSlot& r) {
    const int S_next = D.ctrl[1], SM = Pm.S_max;
    if (a == 0) { r = ResampleSlot{0, 0, 0}; return true; }
    if (a <= S_next) {
        const int s = D.ctrl[4 + a - 1];
        if (!bp_in_range(s, SM, D.kerr)) return false;
        r = ResampleSlot{1 + s, 1, s};
        return true;
    }
    if (a <= S_next + J) { const int j = a - S_next - 1; r = ResampleSlot{1 + SM + j, 2, j}; return true; }
    return false;
}

// cumulative weights (FP64, not normalised) of every kept belief: block (tile, slot) scans its tile
// from the sum of the tiles before it
__global__ void __launch_bounds__(256) k_cdf(DevGeom G, DevParams Pm, DevState D, const double* tsum, double* cdf_all) {
    const int P = Pm.P, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    ResampleSlot r;
    if (!resample_slot(Pm, D, G.J, blockIdx.y, r)) return;
    const double* w = belief_wn(D, BeliefView{r.kind, r.index, 0}, P);
    double* cdf = cdf_all + (size_t)blockIdx.y * P;
    const double* ts = tsum + (size_t)r.b * CDF_TILES;
    __shared__ double red[8];
    double run = block_sum_256(tid < (int)blockIdx.x ? ts[tid] : 0.0, red);
    const int tile = cdf_tile(P), p0 = blockIdx.x * tile, p1 = min(P, p0 + tile);
    for (int q0 = p0; q0 < p1; q0 += CDF_SUB) {
        const int q = q0 + 8 * tid;
        double x[8], loc = 0.0;
        #pragma unroll
        for (int i = 0; i < 8; ++i) {
            loc += (q + i < p1) ? w[q + i] : 0.0;
            x[i] = loc;
        }
        double inc = loc;
        #pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
        }
        __syncthreads();
        if (lane == 31) red[wid] = inc;
        __syncthreads();
        double off = run, tot = 0.0;
        #pragma unroll
        for (int v = 0; v < 8; ++v) {
            if (v < wid) off += red[v];
            tot += red[v];
        }
        off += inc - loc;
        #pragma unroll
        for (int i = 0; i < 8; ++i)
            if (q + i < p1) cdf[q + i] = off + x[i];
        run += tot;
    }
}

// resampling index, gather and jitter into the other buffer, weights of the new belief and (PFs) the PR
// table: a thread per (output particle, slot).  Particle i takes the first k with CDF_k >= (U + i)/P.
__global__ void __launch_bounds__(256) k_resample(DevGeom G, DevParams Pm, DevState D, const double* cdf_all) {
    const int P = Pm.P, J = G.J, i = blockIdx.x * blockDim.x + threadIdx.x;
    const int n = D.step[0], nxt = 1 - D.cur, a = blockIdx.y;
    ResampleSlot r;
    if (!resample_slot(Pm, D, J, a, r)) return;
    if (r.kind == 1 && blockIdx.x == 0 && threadIdx.x < J)
        D.p_pr[(a - 1) * J + threadIdx.x] = D.bel[BEL_PPR + r.index * J + threadIdx.x];
    if (i >= P) return;
    const double* cdf = cdf_all + (size_t)a * P;
    const double tot = cdf[P - 1];
    const double U = u32d(draw(Pm, (uint32_t)((r.kind << 16) | r.index), n, RNG_RESAMPLE, 0, 0).x);
    int src = i;                               // equal weights where the belief has none
    if (tot > 0.0) {
        const double u = (U + (double)i) / (double)P * tot;
        int lo = 0, hi = P - 1;
        while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            if (cdf[mid] >= u) hi = mid; else lo = mid + 1;
        }
        src = lo;
    }
    D.idx[(size_t)r.b * P + i] = src;
    if (!bp_in_range(src, P, D.kerr)) src = i;
    const float* L = D.Lchol + (size_t)r.b * 36;
    if (r.kind == 2) {
        float e[1];
        normals8(Pm, i, n, RNG_JITTER_ETA, r.index, 1, e);
        D.eta[nxt][(size_t)r.index * P + i] = fabsf(D.eta[D.cur][(size_t)r.index * P + src] + L[0] * e[0]);
        D.w_eta[(size_t)r.index * P + i] = 1.0 / P;
        return;
    }
    float e[6];
    normals8(Pm, i, n, r.kind == 0 ? RNG_JITTER_MT : RNG_JITTER_PF, r.index, 6, e);
    const float* in = r.kind == 0 ? D.x[D.cur] : D.phi[D.cur] + (size_t)r.index * 6 * P;
    float* out = r.kind == 0 ? D.x[nxt] : D.phi[nxt] + (size_t)(a - 1) * 6 * P;
    for (int k = 0; k < 6; ++k) {
        float jit = 0.f;
        for (int c = 0; c <= k; ++c) jit += L[k * 6 + c] * e[c];
        float v = in[(size_t)k * P + src] + jit;
        if (r.kind == 1 && k == 3) v = fabsf(v);
        out[(size_t)k * P + i] = v;
    }
    if (r.kind == 0) D.w_x[i] = 1.0 / P;
    else D.w_y[(size_t)(a - 1) * P + i] = D.p_s[r.index] / P;
}

void launch_resample(const DevGeom& G, const DevParams& Pm, const DevState& D, int S, double* cdf, cudaStream_t st) {
    const int nb = 1 + S + G.J;
    k_cdf<<<dim3(cdf_tiles(Pm.P), nb), 256, 0, st>>>(G, Pm, D, D.tsum, cdf);
    k_resample<<<dim3((Pm.P + 255) / 256, nb), 256, 0, st>>>(G, Pm, D, cdf);
}

}  // namespace bp
