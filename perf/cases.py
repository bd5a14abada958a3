"""Performance cases of the particle BP filter: what a program that uses this package has it do.

Every case goes through the public entry points (bp.Filter, bp.Batch, bp.Mlp).  A "step" case is
one time step of a tracking program: restore the belief from its checkpoint in pinned host memory,
predict, update with an observation, read the estimates.  Successive passes take successive
observations of a step (new noise, visibility and spurious paths) from the same belief, as a
Monte Carlo evaluation of one step does, and a program that serves several terminals with one
handle.  A "batch" case steps many independent filters of uneven sizes together; a "train" case
is a few Adam steps of the proposal network on minibatches, after which the parameters are read.

Observations come from the generative signal model in FP64 (plain torch, below).  Initial beliefs
lie around the truth: 1 cm for terminal and surfaces, amplitudes within 10 %, noise variances
within 30 % of their true values.  Where a filter holds more features than there are surfaces, the
others are near-duplicates a few centimetres off, which births leave behind.  The estimates are
weighted means of the FP32 particles, formed from FP32 likelihoods; the program logs them in the
particles' own type, FP32; the updated belief stays in the handle, on the GPU, as it does between
the steps of a run.

`exact` restates the whole step in FP64: Philox counters, prediction and birth, message table,
existence tests, likelihoods, normalisation, estimates.
"""
import math

import numpy as np
import torch

from paper_2604_19723_gb300 import bp
from paper_2604_19723_gb300 import workload as W

OBS = 8                 # observations a program has queued
ARRAYS = ((1, 1), (2, 2), (3, 2), (2, 4), (3, 3), (5, 3), (4, 4), (4, 8), (8, 8))
EXACT_FLOPS = 5.0e12    # FP64 flops of the restated step that fit about 20 s
DRAW_COST = 5.0e11      # P J Nz S^2 of the largest drawn step (the largest listed one: 1.1e12)


def _step(name, **kw):
    c = dict(kind="step", J=4, Nf=10, My=4, Mz=4, B=200e6, P=30000, S=5, S_max=16, K=4, Q=0, T_pru=0.0, sigma_v=0.5,
             sigma_mu=3e-3, sigma_sfv=1e-4, planar=False, zero_mean=False, proposal=False, N_g=4096, learned=False,
             visibility=1.0, clutter=0, snr_db=20.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one array, planar motion, births and pruning, ten spurious paths: the smallest filter, one
        # kernel launch after another
        _step("track_1pa_1k", J=1, P=1000, S=7, Q=1, T_pru=0.1, sigma_v=0.1, planar=True, visibility=0.9, clutter=10),
        # the paper's first experiment: four arrays, 30 000 particles, and about twice as many features as
        # surfaces, which is where its runs settle
        _step("exp1_30k", S=9, Q=1, T_pru=0.1),
        # the paper's second experiment (fast terminal, 100 MHz) with new features drawn from the birth
        # proposal, the configuration of the Monte Carlo evaluation
        _step("exp2_proposal_15k", B=100e6, P=15000, S=7, Q=1, T_pru=0.1, sigma_v=7.7, sigma_mu=3e-2, sigma_sfv=4e-3,
              proposal=True),
        # odd sizes throughout and the zero-mean amplitude variant: three 3 x 3 arrays, 7 frequencies
        _step("ragged_zm_21x4999", J=3, Nf=7, My=3, Mz=3, P=4999, S=21, S_max=21, K=20, zero_mean=True, visibility=0.9,
              clutter=20),
        # many frequencies on a small array, a feature count between the powers of two
        _step("wideband_40x8k", Nf=75, My=2, Mz=2, P=8192, S=40, S_max=40, K=39, visibility=0.8),
        # the learned terminal proposal at its operating point: a tenth of the particles
        _step("learned_64x10k", P=10000, S=64, S_max=64, K=63, learned=True, visibility=0.8, clutter=200),
        # the benchmark's workload: 64 features held fixed, 100 000 particles, 200 spurious paths
        _step("scale_64x100k", P=100000, S=64, S_max=64, K=63, visibility=0.8, clutter=200),
        # the mixed-precision stress shape: 8 x 8 arrays, 16 frequencies, 30 dB
        _step("stress_32x262k", Nf=16, My=8, Mz=8, P=262144, S=32, S_max=32, K=31, visibility=0.8, clutter=500, snr_db=30.0),
        # independent filters of uneven sizes stepped together (graphs, shared workspaces)
        dict(name="batch_16", kind="batch", n=16, mix=21),
        # training the proposal network: sixteen minibatches, then the parameters
        dict(name="train_16x4096", kind="train", B=4096, steps=16),
    ]


def draw(rng):
    u = rng.random()
    if u < 0.1:
        return dict(kind="batch", n=rng.randint(3, 16), mix=rng.randrange(1, 10000))
    if u < 0.2:
        return dict(kind="train", B=int(round(math.exp(rng.uniform(math.log(200), math.log(16384))))),
                    steps=rng.randint(4, 24))
    My, Mz = rng.choice(ARRAYS)
    Nf = rng.randint(3, max(3, min(75, 1024 // (My * Mz))))
    J = rng.randint(1, 4)
    births = rng.random() < 0.35
    S = rng.randint(2, 12) if births else int(round(math.exp(rng.uniform(math.log(2), math.log(64)))))
    P = int(round(math.exp(rng.uniform(math.log(500), math.log(131072)))))
    cost = float(J) * Nf * My * Mz * (16 if births else S) ** 2
    P = max(400, min(P, int(DRAW_COST / cost)))
    fast = rng.random() < 0.3
    K = min(S - 1, 4) if births else max(1, (S - 1) // 2) if rng.random() < 0.25 else S - 1
    return _step(None, J=J, Nf=Nf, My=My, Mz=Mz, P=P, S=S, K=K, S_max=16 if births else S, Q=1 if births else 0,
                 T_pru=0.1 if births else 0.0, sigma_v=7.7 if fast else 0.5, sigma_mu=3e-2 if fast else 3e-3,
                 sigma_sfv=4e-3 if fast else 1e-4, planar=rng.random() < 0.15, zero_mean=rng.random() < 0.2,
                 proposal=births and rng.random() < 0.5, N_g=rng.choice((1024, 4096)),
                 visibility=rng.choice((0.8, 0.9, 1.0)), clutter=rng.choice((0, 0, 10, 50, 200)),
                 snr_db=rng.choice((15.0, 20.0, 30.0)))


# ---------------------------------------------------------------- inputs
def _params(c):
    z = 0.0 if c["planar"] else 1.0
    return W.Params(T=0.1, sigma_v=c["sigma_v"], sigma_mu=c["sigma_mu"], sigma_sfv=c["sigma_sfv"], Q=c["Q"],
                    T_pru=c["T_pru"], motion_dims=2 if c["planar"] else 3, zero_mean=int(c["zero_mean"]),
                    birth_proposal=int(c["proposal"]), N_g=c["N_g"], p_min=(-3.5, -1.0, -z), p_max=(4.5, 4.5, z))


def _geometry(c):
    return W.make_geometry(J=c["J"], Nf=c["Nf"], My=c["My"], Mz=c["Mz"], B=c["B"])


def _dev(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device="cuda")


def _steering(g, j, p, sfv):
    """psi^(j) for terminal positions p (n, 3) and surfaces sfv ((n, 3), None: line of sight): (n, Nz)."""
    pa, R = _dev(g.p_pa[j]), _dev(g.R_pa[j])
    if sfv is None:
        r = p - pa
    else:
        nn = (sfv * sfv).sum(1, keepdim=True)
        va = pa - (2.0 * (sfv @ pa)[:, None] / nn - 1.0) * sfv
        r = p - va
        r = r - 2.0 * (sfv * r).sum(1, keepdim=True) / nn * sfv
    loc = r @ R
    d = loc.norm(dim=1)
    lam = g.c / g.fc
    f = _dev(g.freqs())
    cyc = -(g.fc + f)[None, :] * d[:, None] / g.c
    ym = (loc[:, 1] / d)[:, None] * _dev(g.p_y) / lam
    zm = (loc[:, 2] / d)[:, None] * _dev(g.p_z) / lam

    def cis(t):
        t = 2.0 * math.pi * (t - torch.round(t))
        return torch.complex(torch.cos(t), torch.sin(t))

    a = (cis(ym)[:, :, None] * cis(zm)[:, None, :]).reshape(len(d), -1)
    b = cis(cyc) * (lam / (4.0 * math.pi * d))[:, None]
    return (b[:, :, None] * a[:, None, :]).reshape(len(d), -1)


def _inputs(c, seed):
    """OBS observations (OBS, J, Nz) complex64 of step 1 and the belief of step 0, from the seed alone."""
    g, prm = _geometry(c), _params(c)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rng = np.random.default_rng(seed)
    rand = lambda *s: torch.rand(*s, generator=gen, device="cuda", dtype=torch.float64)    # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64)  # noqa: E731
    J, P, S, K, Nz = c["J"], c["P"], c["S"], c["K"], g.Nz
    # the truth: a terminal inside the room, the room's walls and random surfaces, amplitudes 1 and 1/2
    x0 = np.r_[0.5 + rng.uniform(-1, 1), 1.75 + rng.uniform(-1, 1), 0.0 if c["planar"] else 0.1, 0.2, -0.1, 0.0]
    x1 = x0.copy()
    x1[:3] += prm.T * x0[3:]
    walls = W.room_sfvs(prm.p_min, prm.p_max)
    sfv = walls[:K] if K <= 4 else np.concatenate([walls, W.random_sfvs(rng, K - 4, prm.p_min, prm.p_max)])
    rho_abs = np.r_[1.0, np.full(K, 0.5)]
    rho = rho_abs * np.exp(1j * rng.uniform(-np.pi, np.pi, K + 1))
    vis = torch.as_tensor(rng.random((OBS, J, K + 1)) < c["visibility"], device="cuda")
    at, surf, rt, power = _dev(x1[None, :3]), _dev(sfv), torch.as_tensor(rho, device="cuda"), 0.0
    z = torch.zeros(OBS, J, Nz, dtype=torch.complex128, device="cuda")
    for j in range(J):
        paths = torch.cat([_steering(g, j, at, None), _steering(g, j, at.expand(K, 3), surf)])    # (K + 1, Nz)
        power += float((rt @ paths).abs().square().mean()) / J
        z[:, j] = (rt * vis[:, j]) @ paths
    eta = power / 10.0 ** (c["snr_db"] / 10.0)                  # sum-channel SNR
    box_lo, box_hi = _dev(2.0 * np.asarray(prm.p_min)), _dev(2.0 * np.asarray(prm.p_max))
    for i, n in enumerate(rng.poisson(c["clutter"], OBS)):      # spurious paths
        v = box_lo + (box_hi - box_lo) * rand(int(n), 3)
        v = v[v.norm(dim=1) > 1.0]
        for j in range(J if len(v) else 0):
            a = torch.polar(torch.full_like(v[:, 0], 0.05), 2.0 * math.pi * rand(len(v)))
            z[i, j] += a @ _steering(g, j, at.expand(len(v), 3), v)
    z += math.sqrt(eta / 2.0) * torch.complex(randn(OBS, J, Nz), randn(OBS, J, Nz))
    # the belief of step 0
    x = _dev(x0)[:, None] + _dev([0.01] * 3 + [0.05] * 3)[:, None] * randn(6, P)
    if c["planar"]:
        x[2], x[5] = 0.0, 0.0
    phi = torch.zeros(S, 6, P, dtype=torch.float32, device="cuda")
    for s in range(S):
        k = 0 if s == 0 else 1 + (s - 1) % K
        if s:
            centre = sfv[k - 1] + (rng.normal(0.0, 0.03, 3) if s > K else 0.0)
            phi[s, :3] = (_dev(centre)[:, None] + 0.01 * randn(3, P)).float()
            if c["planar"]:
                phi[s, 2] = float(sfv[k - 1, 2])
        phi[s, 3] = (rho_abs[k] ** 2 * (0.5 + rand(P))).float()
        if not c["zero_mean"]:
            m = rho[k] + 0.1 * rho_abs[k] / math.sqrt(2.0) * torch.complex(randn(P), randn(P))
            phi[s, 4], phi[s, 5] = m.real.float(), m.imag.float()
    p_s = rng.uniform(0.3, 0.99, S)
    host = lambda a: torch.as_tensor(a).pin_memory().numpy()                                # noqa: E731
    st = W.StateArrays(n=0, S=S, x=host(x.float().cpu()), phi=host(phi.cpu()),
                       eta=host((eta * torch.exp(0.3 * randn(J, P))).float().cpu()), w_x=host(np.full(P, 1.0 / P)),
                       w_y=host(np.repeat(p_s[:, None] / P, P, axis=1)), w_eta=host(np.full((J, P), 1.0 / P)),
                       p_pr=rng.uniform(0.2, 0.99, (S, J)))
    return g, prm, z.to(torch.complex64), st


def _batch_members(c):
    """The scenarios of the batched workload as step cases, in batch order."""
    out = []
    for d in W.batched_scenarios(c["n"], seed=c["mix"]):
        g = d["geom"]
        out.append(_step(None, J=g.J, Nf=g.Nf, My=g.My, Mz=g.Mz, P=d["P"], S=d["S"], S_max=d["S"], K=d["S"] - 1, visibility=0.8))
    return out


# ---------------------------------------------------------------- the program's side
def prepare(case, seed):
    c = case
    if c["kind"] == "train":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n = c["B"] * c["steps"]
        X = torch.randn(n, 16, generator=gen, device="cuda")
        mean = 0.5 * torch.tanh(X[:, :3])
        T = mean + 0.7 * torch.randn(n, 3, generator=gen, device="cuda")
        return dict(case=c, net=bp.Mlp(W.mlp_init(seed)), X=X.split(c["B"]), T=T.split(c["B"]),
                    loss=torch.zeros(c["steps"], device="cuda"))
    if c["kind"] == "batch":
        members = [_inputs(m, seed + 1000 * i) for i, m in enumerate(_batch_members(c))]
        b = bp.Batch([(g, prm, st.x.shape[1], st.S, st.S, seed + i) for i, (g, prm, _, st) in enumerate(members)])
        z = torch.zeros(OBS, b.z_floats(), device="cuda")
        for i, (g, _, zi, _) in enumerate(members):
            o = b.z_offset(i)
            z[:, o:o + 2 * g.J * g.Nz] = torch.view_as_real(zi).reshape(OBS, -1)
        return dict(case=c, batch=b, member=[b.member(i) for i in range(len(b))], start=[m[3] for m in members], z=z,
                    now=torch.zeros_like(z[0]), i=0)
    g, prm, z, st = _inputs(c, seed)
    f = bp.Filter(g, prm, P=c["P"], S_max=c["S_max"], seed=seed)
    if c["learned"]:
        f.set_mt_proposal(bp.Mlp(W.mlp_init(seed)))
    return dict(case=c, filter=f, z=z, start=st, i=0)


def _log(e):
    return dict(x_hat=e["x_hat"].astype(np.float32), eta_hat=e["eta_hat"].astype(np.float32),
                p_s=e["p_s"].astype(np.float32), phi_hat=e["phi_hat"].astype(np.float32),
                p_pr=e["p_pr"].astype(np.float32), declared=e["declared"], S_next=int(e["S_next"]))


def _join(logs):
    """The members' logs as one: concatenated along the features (or arrays)."""
    return {k: np.concatenate([np.atleast_1d(lg[k]).reshape(-1) for lg in logs]) for k in logs[0]}


def run(state):
    c = state["case"]
    if c["kind"] == "train":
        for k, (X, T) in enumerate(zip(state["X"], state["T"])):
            state["net"].train_step(X, T, 1e-3, loss_out=state["loss"][k:k + 1])
        return dict(params=state["net"].params(), loss=state["loss"])
    i = state["i"] % OBS
    state["i"] += 1
    if c["kind"] == "batch":
        for m, st in zip(state["member"], state["start"]):
            m.set_state(st)
        state["now"].copy_(state["z"][i])
        state["batch"].step(state["now"])
        return _join([_log(m.estimate()) for m in state["member"]])
    f = state["filter"]
    f.set_state(state["start"])
    f.step(state["z"][i])
    return _log(f.estimate())


# ---------------------------------------------------------------- what a pass cannot do without
def _step_work(c):
    P, J, S, Nz = float(c["P"]), c["J"], c["S"] + c["Q"], c["Nf"] * c["My"] * c["Mz"]
    nfac = c["Nf"] + c["My"] + c["Mz"]
    particles = P * (6 + 6 * S + J)
    flops = P * J * (S * Nz * 8 * S              # projections of every steering vector on the other features
                     + S * Nz * 2 * 8            # its products with the residual and the message table's sums
                     + S * S / 2 * 8 * nfac      # the terminal likelihood's Gram matrix
                     + S * Nz * 8                # its residual
                     + S ** 3 / 6 * 8            # its factorisation
                     + S * nfac * 20)            # steering factors
    if c["proposal"]:
        flops += c["N_g"] * J * Nz * 8.0
    if c["learned"]:
        flops += P * 12288
    return dict(bytes=2 * 4 * particles + 8 * J * Nz, flops=flops)


def work(case):
    if case["kind"] == "train":
        n = case["B"] * case["steps"]
        return dict(bytes=n * 19 * 4.0 + 6288 * 4.0, flops=n * 3 * 12288.0)
    if case["kind"] == "batch":
        each = [_step_work(m) for m in _batch_members(case)]
        return {k: sum(e[k] for e in each) for k in ("bytes", "flops")}
    return _step_work(case)


# ---------------------------------------------------------------- the same in 64 bits
def _philox(item, n, purpose, sub, block, seed):
    """Philox4x32-10 words of counters (item, n, purpose << 16 | sub, block), key = seed."""
    M, mask = (0xD2511F53, 0xCD9E8D57), 0xFFFFFFFF
    c = [item, torch.full_like(item, n), torch.full_like(item, (purpose << 16) | sub), torch.full_like(item, block)]
    k0, k1 = seed & mask, (seed >> 32) & mask
    for _ in range(10):
        p0, p1 = c[0] * M[0], c[2] * M[1]      # the low 64 bits are kept, as two 32-bit words
        c = [((p1 >> 32) & mask) ^ c[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return c


def _u24(x):
    return ((x >> 8).double() + 0.5) * 2.0 ** -24


def _normals(item, n, purpose, sub, count, seed):
    out = []
    for block in range((count + 3) // 4):
        w = _philox(item, n, purpose, sub, block, seed)
        for a, b in ((0, 1), (2, 3)):
            r, t = torch.sqrt(-2.0 * torch.log(_u24(w[a]))), 2.0 * math.pi * _u24(w[b])
            out += [r * torch.cos(t), r * torch.sin(t)]
    return out[:count]


def _uniforms(item, n, purpose, sub, count, seed):
    out = []
    for block in range((count + 3) // 4):
        out += [_u24(w) for w in _philox(item, n, purpose, sub, block, seed)]
    return out[:count]


def _gamma(item, n, purpose, sub, shape, scale, seed):
    """Marsaglia-Tsang, one Philox block per attempt."""
    d = shape - 1.0 / 3.0
    cc = 1.0 / math.sqrt(9.0 * d)
    out, done = shape * scale, torch.zeros_like(item, dtype=torch.bool)
    for a in range(16):
        w = _philox(item, n, purpose, sub, a, seed)
        u = [(v.double() + 0.5) * 2.0 ** -32 for v in w[:3]]
        x = torch.sqrt(-2.0 * torch.log(u[0])) * torch.cos(2.0 * math.pi * u[1])
        v = (1.0 + cc * x) ** 3
        ok = (v > 0) & (torch.log(u[2]) < 0.5 * x * x + d - d * v + d * torch.log(v.clamp_min(1e-300)))
        out = torch.where(ok & ~done, d * v * scale, out)
        done |= ok
        if bool(done.all()):
            break
    return out


def _store(a):
    """Particles are FP32."""
    return a.float().double()


def _mean_weighted(rows, w):
    return rows @ (w / w.sum())


def _propose(prm, g, z, x, phi, w_x, w_alpha, S, seed):
    """The new features' positions and weights from the coherent Bartlett spectrum of the residual."""
    P = x.shape[1]
    xh = _mean_weighted(x[:3], w_x)
    pos = [_mean_weighted(phi[s, :3], w_alpha[s]) for s in range(S)]
    res = []
    for j in range(g.J):
        A = torch.cat([_steering(g, j, xh[None], None if s == 0 else pos[s][None]) for s in range(S)]).T
        q = torch.linalg.qr(A)[0]
        res.append(z[j] - q @ (q.conj().T @ z[j]))
    lo0, hi0 = 2.0 * np.asarray(prm.p_min), 2.0 * np.asarray(prm.p_max)
    item = torch.arange(prm.N_g, device="cuda")
    for s in range(S, phi.shape[0]):
        q = s - S
        lo, hi = lo0.copy(), hi0.copy()
        wd = (hi0[0] - lo0[0]) / prm.Q
        lo[0] = lo0[0] + q * wd
        hi[0] = lo[0] + wd
        lo, hi = _dev(lo), _dev(hi)
        cand = lo + (hi - lo) * torch.stack(_uniforms(item, 1, 13, q, 3, seed), 1)
        acc = sum(_steering(g, j, xh.expand(len(cand), 3), cand) @ res[j].conj() / g.Nz for j in range(g.J))
        cost = acc.abs().square()
        if not float(cost.sum()) > 0:
            continue
        m = cand[int(cost.argmax())]
        C = ((cand - m) * (cost / cost.sum())[:, None]).T @ (cand - m)
        L = torch.zeros_like(C)
        for k in range(3):
            piv = float(C[k, k] - (L[k, :k] ** 2).sum())
            if piv > 0:
                L[k, k] = math.sqrt(piv)
                for i in range(k + 1, 3):
                    L[i, k] = (C[i, k] - (L[i, :k] * L[k, :k]).sum()) / L[k, k]
        e = torch.stack(_normals(torch.arange(P, device="cuda"), 1, 14, s, 3, seed))
        at = m[:, None] + L @ e
        ok = ((at >= lo[:, None]) & (at <= hi[:, None])).all(0)
        w = torch.where(ok, torch.exp(0.5 * (e[torch.diagonal(L) > 0] ** 2).sum(0)), torch.zeros_like(at[0]))
        if float(w.sum()) > 0:
            phi[s, :3] = _store(at)
            w_alpha[s] = prm.mu_B / prm.Q / (1.0 + prm.mu_B / prm.Q) * w / w.sum()


def _exact_step(c, seed, filter_seed):
    g, prm, z, st = _inputs(c, seed)
    z = z[0].to(torch.complex128)
    J, P, S_old, Nz, T = c["J"], c["P"], c["S"], g.Nz, prm.T
    S = min(S_old + prm.Q, c["S_max"])
    item = torch.arange(P, device="cuda")
    sd = filter_seed
    # prediction and birth
    x, eta = _dev(st.x), _dev(st.eta)
    w = prm.sigma_v * torch.stack(_normals(item, 1, 1, 0, 3, sd))
    if c["planar"]:
        w[2] = 0.0
    x = _store(torch.cat([x[:3] + T * x[3:] + 0.5 * T * T * w, x[3:] + T * w]))
    eta = torch.stack([_store(_gamma(item, 1, 2, j, prm.c_eta, eta[j] / prm.c_eta, sd)) for j in range(J)])
    phi = torch.zeros(S, 6, P, dtype=torch.float64, device="cuda")
    phi[:S_old] = _dev(st.phi)
    for s in range(S_old):
        e = _normals(item, 1, 3, s, 5, sd)
        if s:
            for k in range(2 if c["planar"] else 3):
                phi[s, k] += prm.sigma_sfv * e[k]
        phi[s, 3] = _gamma(item, 1, 4, s, prm.c_gamma, phi[s, 3] / prm.c_gamma, sd)
        if c["zero_mean"]:
            phi[s, 4:] = 0.0
        else:
            phi[s, 4] += prm.sigma_mu / math.sqrt(2.0) * e[3]
            phi[s, 5] += prm.sigma_mu / math.sqrt(2.0) * e[4]
    pB = prm.mu_B / max(prm.Q, 1) / (1.0 + prm.mu_B / max(prm.Q, 1))
    lo, hi = 2.0 * np.asarray(prm.p_min), 2.0 * np.asarray(prm.p_max)
    for s in range(S_old, S):
        u = _uniforms(item, 1, 5, s, 6, sd)
        wd = (hi[0] - lo[0]) / prm.Q
        for k in range(3):
            phi[s, k] = (lo[0] + (s - S_old) * wd + wd * u[0]) if k == 0 else lo[k] + (hi[k] - lo[k]) * u[k]
        phi[s, 3] = prm.gamma_max * u[3]
        if not c["zero_mean"]:
            r = prm.mu_max * torch.sqrt(u[4])
            phi[s, 4], phi[s, 5] = r * torch.cos(2.0 * math.pi * u[5]), r * torch.sin(2.0 * math.pi * u[5])
    phi = _store(phi)
    w_x, w_eta = _dev(st.w_x), _dev(st.w_eta)
    w_al = torch.full((S, P), pB / P, dtype=torch.float64, device="cuda")
    w_al[:S_old] = prm.pS * _dev(st.w_y)
    zeta = torch.full((S, J), prm.pB_pr, dtype=torch.float64, device="cuda")
    zeta[:S_old] = prm.pS_pr * _dev(st.p_pr) + prm.pR_pr * (1.0 - _dev(st.p_pr))
    if c["proposal"]:
        _propose(prm, g, z, x, phi, w_x, w_al, S_old, sd)
    gam, mu = phi[:, 3], torch.complex(phi[:, 4], phi[:, 5])
    m2 = mu.abs().square()
    Ws, eb = w_al.sum(1), (w_eta * eta).sum(1)
    pr, lk, li, ln = torch.zeros(S, J, device="cuda").double(), torch.zeros(S, P, device="cuda").double(), \
        torch.zeros(P, device="cuda").double(), torch.zeros(J, P, device="cuda").double()
    chunk = max(1, int(2.0e8) // (Nz * S))
    parts = [slice(a, min(P, a + chunk)) for a in range(0, P, chunk)]
    for j in range(J):
        pi, e = zeta[:, j] * Ws, float(eb[j])
        amp1, amp2 = torch.sqrt(gam + m2 * (1.0 - pi)[:, None]), torch.sqrt(gam + m2 * (1.0 - Ws)[:, None])
        tab = torch.zeros(S, 3, Nz, dtype=torch.complex128, device="cuda")
        ps = lambda s, q: _steering(g, j, x[:3, q].T, None if s == 0 else phi[s, :3, q].T)   # noqa: E731
        for q in parts:                                     # message table, terminal likelihood
            Psi = torch.stack([ps(s, q) for s in range(S)], 1)                               # (p, S, Nz)
            cf = (w_x[q] * torch.stack([amp1[:, q] + 0j, amp2[:, q] + 0j, mu[:, q]])).transpose(0, 1)
            tab += torch.einsum("sip,psn->sin", cf, Psi)
            d = torch.sqrt(pi[:, None] * (gam[:, q] + m2[:, q] * (1.0 - pi)[:, None])).T     # (p, S)
            r = z[j] - torch.einsum("ps,psn->pn", (pi[:, None] * mu[:, q]).T, Psi)
            M = d[:, :, None] * Psi
            G = M.conj() @ M.transpose(1, 2)
            L = torch.linalg.cholesky(torch.eye(S, device="cuda") + G / e)
            y = torch.linalg.solve_triangular(L, M.conj() @ r[:, :, None], upper=False)[:, :, 0]
            li[q] += -(r.abs().square().sum(1) / e - y.abs().square().sum(1) / e ** 2) \
                - 2.0 * torch.log(torch.diagonal(L, dim1=1, dim2=2).real).sum(1) - Nz * math.log(math.pi * e)
            del Psi, M, G, L, y
        m, mw = (Ws * zeta[:, j])[:, None] * tab[:, 0], Ws[:, None] * tab[:, 1]
        mu4 = Ws[:, None] * tab[:, 2]
        mu3 = zeta[:, j, None] * mu4
        for s in range(S):                                  # existence tests, feature likelihoods
            o = [k for k in range(S) if k != s]
            Mo = m[o].T
            B = torch.eye(S - 1, device="cuda", dtype=torch.complex128) + Mo.conj().T @ Mo / e
            V = torch.linalg.solve_triangular(torch.linalg.cholesky(B), Mo.conj().T, upper=False).conj().T
            e0 = z[j] - mu3[o].sum(0)

            def form(a, b):                                 # a^H A^-1 b, A = eta I + Mo Mo^H, rows a, b
                return ((a.conj() * b).sum(-1) - ((a @ V.conj()).conj() * (b @ V.conj())).sum(-1) / e) / e

            def quad(v, r, q):                              # log CN up to what both hypotheses share
                den = 1.0 + q * form(v, v).real
                return q * form(v, r).abs().square() / den - form(r, r).real - torch.log(den)

            null = -form(e0, e0).real
            llr = quad(mw[s], e0 - mu4[s], 1.0) - null
            pr[s, j] = torch.sigmoid(torch.log(zeta[s, j]) - torch.log1p(-zeta[s, j]) + llr)
            qa = (gam[s] + m2[s] * (1.0 - zeta[s, j])) * zeta[s, j]
            for a in range(0, P, max(1, int(2.0e8) // Nz)):
                q = slice(a, min(P, a + max(1, int(2.0e8) // Nz)))
                v = ps(s, q)
                lk[s, q] += quad(v, e0[None] - zeta[s, j] * mu[s, q][:, None] * v, qa[q]) - null
        lam, U = torch.linalg.eigh(m.conj() @ m.T)          # noise likelihood
        r = z[j] - mu3.sum(0)
        b2 = (U.conj().T @ (m.conj() @ r)).abs().square()
        lam = lam.clamp_min(0.0)
        den = eta[j][None, :] + lam[:, None]
        ln[j] = -(r.abs().square().sum() - (b2[:, None] / den).sum(0)) / eta[j] - torch.log(den).sum(0) \
            - (Nz - S) * torch.log(eta[j]) - Nz * math.log(math.pi)
    wx = torch.softmax(torch.log(w_x) + li, 0)
    we = torch.softmax(torch.log(w_eta) + ln, 1)
    lw = torch.log(w_al) + lk
    lse = torch.logsumexp(lw, 1)
    tot = torch.logaddexp(lse, torch.log1p(-Ws.clamp_max(1.0)))
    wy = torch.softmax(lw, 1)
    out = dict(x_hat=x @ wx, eta_hat=(we * eta).sum(1), p_s=torch.exp(lse - tot), p_pr=pr,
               phi_hat=torch.einsum("skp,sp->sk", phi, wy))
    return {**{k: v.cpu().numpy() for k, v in out.items()}, "declared": None, "S_next": None}


def _exact_flops(c):
    return 16.0 * c["P"] * c["J"] * c["Nf"] * c["My"] * c["Mz"] * (c["S"] + c["Q"]) ** 2


def _exact_train(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n = c["B"] * c["steps"]
    X = torch.randn(n, 16, generator=gen, device="cuda")
    T = 0.5 * torch.tanh(X[:, :3]) + 0.7 * torch.randn(n, 3, generator=gen, device="cuda")
    X, T = X.double(), T.double()
    th = _dev(W.mlp_init(seed).astype(np.float64))
    m1, m2, loss = torch.zeros_like(th), torch.zeros_like(th), []
    for k in range(c["steps"]):
        x, t = X[k * c["B"]:(k + 1) * c["B"]], T[k * c["B"]:(k + 1) * c["B"]]
        p = th.clone().requires_grad_(True)
        h, o = x, 0
        for i, (fi, fo) in enumerate(((16, 64), (64, 64), (64, 16))):
            h = h @ p[o:o + fi * fo].reshape(fo, fi).T + p[o + fi * fo:o + fi * fo + fo]
            o += fi * fo + fo
            h = torch.relu(h) if i < 2 else h
        lo = (0.5 * ((t - h[:, :3]) * torch.exp(-h[:, 3:6])) ** 2 + h[:, 3:6]).sum()
        gr = torch.autograd.grad(lo / c["B"], p)[0]
        m1, m2 = 0.9 * m1 + 0.1 * gr, 0.999 * m2 + 0.001 * gr * gr
        th = th - 1e-3 * (m1 / (1.0 - 0.9 ** (k + 1))) / (torch.sqrt(m2 / (1.0 - 0.999 ** (k + 1))) + 1e-8)
        loss.append(float(lo))
    return dict(params=th.cpu().numpy(), loss=np.asarray(loss))


def exact(case, seed):
    c = case
    if c["kind"] == "train":
        return _exact_train(c, seed)
    if c["kind"] == "batch":
        members = _batch_members(c)
        if sum(_exact_flops(m) for m in members) > EXACT_FLOPS:
            return None
        logs = [_exact_step(m, seed + 1000 * i, seed + i) for i, m in enumerate(members)]
        keep = [k for k in logs[0] if logs[0][k] is not None]
        return {**_join([{k: lg[k] for k in keep} for lg in logs]), "declared": None, "S_next": None}
    if c["learned"] or _exact_flops(c) > EXACT_FLOPS:      # the network's draws have no 64-bit value
        return None
    return _exact_step(c, seed, seed)
