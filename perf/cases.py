"""The work that users of the library have it do, as measurable cases.

Every case calls the public binding the way a program does:

  step    draw proposals of one lattice and run the Metropolis-Hastings scan of its
          chains over them (the loop of Algorithm 1), in FP64, FP32 or BF16
  logq    log q and energy of given configurations (chain states under a new proposal)
  tune    log q of accepted states and its gradient with respect to the tensors
  batch   one graph-replayed step of many disorder samples of uneven size
  sweep   the same with a Metropolis sweep between proposals (equilibration runs)
  frozen  one frozen-line move of chains on tori (environments rebuilt for every move)
  build   the environments of one lattice, its first proposals and log Z~
  cube    proposals and the scan on a cubic lattice

Sizes follow the repository's workloads: the 8 x 8 ferromagnet, the 32 x 32 +-J glass, the
batches of Gaussian glasses, the fully frustrated lattice that is tuned, the wide critical
ferromagnet at chi = 64 (cut to a strip whose environment builds in a second), the
equilibration and torus runs, and the cube.
"""
import math

import numpy as np
import torch

from paper_2104_13264_gb300 import autograd, batched, binding, frozen, instances


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: a single chain on a small ferromagnet, launches and latency count
        dict(name="chain_8x8_f64", kind="step", model="ferro", Ly=8, Lx=8, beta=0.44, chi=8, precision="f64",
             B=10000, chains=1),
        # FP64 proposals of a ragged glass in random fields (dense tensors, odd sizes)
        dict(name="glass_23x29_f64", kind="step", model="field", Ly=23, Lx=29, beta=0.8, chi=13, precision="f64",
             B=5000, chains=50),
        # the production form of a mid-sized glass: 65536 proposals per launch in FP32
        dict(name="glass_32x32_f32", kind="step", model="pm", Ly=32, Lx=32, beta=1.0, chi=16, precision="f32",
             B=65536, chains=256),
        # re-evaluating chain states after the proposal changed
        dict(name="villain_24x45_logq", kind="logq", model="villain", Ly=24, Lx=45, beta=1.5, chi=32,
             precision="f32", B=16384),
        # one gradient of a tuning run
        dict(name="villain_12x48_tune", kind="tune", model="villain", Ly=12, Lx=48, beta=1.5, chi=32, B=8192),
        # the wide critical lattice at chi = 64 on the tensor cores, a full launch
        dict(name="strip_8x96_bf16", kind="step", model="ferro", Ly=8, Lx=96, beta=0.4407, chi=64,
             precision="bf16", B=65536, chains=64),
        # one large-chi member of a disorder batch on the tensor cores: few tiles, latency counts
        dict(name="glass_20x40_bf16", kind="step", model="gauss", Ly=20, Lx=40, beta=2.0, chi=32,
             precision="bf16", B=4096, chains=16),
        # a batch of glasses of uneven L and chi in one persistent launch
        dict(name="batch_f32", kind="batch", n=48, Lmin=16, Lmax=32, chimax=32, beta=2.0, precision="f32", B=4096,
             chains=16),
        # equilibration: one proposal and one sweep per chain and iteration, FP64, low temperature
        dict(name="equilibrate_f64", kind="sweep", n=64, Lmin=32, Lmax=32, chimax=16, beta=1.0 / 0.212,
             precision="f64", B=32, chains=32),
        # chains on tori: every move builds one environment per chain
        dict(name="torus_24", kind="frozen", D=4, C=16, L=24, beta=1.0 / 0.212, chi=16),
        # one environment build of the frustrated lattice
        dict(name="build_16x48", kind="build", model="villain", Ly=16, Lx=48, beta=1.5, chi=32, B=1024),
        # three dimensions, bond basis
        dict(name="cube_8", kind="cube", L=8, T=4.5, D=2, chi=2, precision="f32", B=8192, chains=64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "logq", "tune", "batch", "sweep", "frozen", "build", "cube"])
    model = rng.choice(["ferro", "pm", "gauss", "field", "villain"])
    beta = {"ferro": 0.44, "pm": 1.0, "gauss": 2.0, "field": 0.8, "villain": 1.5}[model]
    if kind == "step":
        precision = rng.choice(["f64", "f32", "bf16"])
        if precision == "bf16":
            Ly, Lx, chi = rng.randint(6, 20), rng.randint(24, 96), rng.randint(24, 64)
            cap, B = 2.0e12, _log_int(rng, 2048, 65536)
            while Ly * Lx * chi ** 3 > 5e7:       # the environment builds in about a second
                Ly, chi = max(6, Ly - 1), chi - 2
        elif precision == "f32":
            Ly, Lx, chi = rng.randint(12, 40), rng.randint(12, 48), rng.randint(6, 32)
            cap, B = 1.0e11, _log_int(rng, 4096, 65536)
        else:
            Ly, Lx, chi = rng.randint(6, 32), rng.randint(6, 32), rng.randint(4, 16)
            cap, B = 1.2e10, _log_int(rng, 1000, 16384)
        chains = rng.choice([1, 16, 50, 256])
        B = int(max(500, min(B, cap / _flops(Ly, Lx, chi)))) // chains * chains
        B = max(B, chains)
        return dict(kind=kind, model=model, Ly=Ly, Lx=Lx, beta=beta, chi=chi, precision=precision, B=B, chains=chains)
    if kind == "logq":
        Ly, Lx, chi = rng.randint(12, 32), rng.randint(12, 48), rng.randint(8, 32)
        B = int(max(300, min(_log_int(rng, 1024, 32768), 1.0e11 / _flops(Ly, Lx, chi))))
        return dict(kind=kind, model=model, Ly=Ly, Lx=Lx, beta=beta, chi=chi, precision="f32", B=B)
    if kind == "tune":
        Ly, Lx, chi = rng.randint(8, 16), rng.randint(16, 48), rng.randint(8, 32)
        B = int(max(300, min(_log_int(rng, 1024, 8192), 2.0e10 / _flops(Ly, Lx, chi))))
        return dict(kind=kind, model=rng.choice(["pm", "villain", "field"]), Ly=Ly, Lx=Lx, beta=1.0, chi=chi, B=B)
    if kind == "batch":
        Lmin = rng.randint(12, 24)
        return dict(kind=kind, n=rng.randint(16, 48), Lmin=Lmin, Lmax=Lmin + rng.randint(2, 8),
                    chimax=rng.choice([8, 16, 24]), beta=2.0, precision="f32", B=16 * _log_int(rng, 32, 256),
                    chains=16)
    if kind == "sweep":
        L = rng.randint(16, 32)
        chains = 2 * rng.randint(8, 16)
        return dict(kind=kind, n=rng.randint(16, 64), Lmin=L, Lmax=L, chimax=rng.randint(8, 16), beta=1.0 / 0.212,
                    precision="f64", B=chains, chains=chains)
    if kind == "frozen":
        return dict(kind=kind, D=rng.randint(1, 4), C=2 * rng.randint(4, 8), L=rng.randint(12, 24), beta=1.0 / 0.212,
                    chi=rng.randint(8, 16))
    if kind == "build":
        Ly, Lx, chi = rng.randint(8, 20), rng.randint(16, 48), rng.randint(8, 32)
        while Ly * Lx * chi ** 3 > 2e7:
            Ly, Lx = max(8, Ly - 1), Lx - 1
        return dict(kind=kind, model=model, Ly=Ly, Lx=Lx, beta=beta, chi=chi, B=_log_int(rng, 64, 1024))
    return dict(kind=kind, L=rng.randint(4, 8), T=rng.choice([4.0, 4.5, 5.0]), D=2, chi=2, precision="f32",
                B=64 * rng.randint(16, 128), chains=64)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _instance(case, seed):
    m, Ly, Lx, beta, chi = case["model"], case["Ly"], case["Lx"], case["beta"], case["chi"]
    if m == "ferro":
        return instances.ferromagnet(Ly, Lx, beta, chi)
    if m == "villain":
        return instances.villain(Ly, Lx, beta, chi)
    if m == "pm":
        return instances.ea_pm(Ly, Lx, beta, chi, seed=seed)
    return instances.ea_gauss(Ly, Lx, beta, chi, seed=seed, hscale=0.3 if m == "field" else 0.0)


def _batch_instances(case, seed):
    g = np.random.default_rng([case["n"], case["Lmin"], case["Lmax"], 23])   # sizes belong to the case
    Ls = g.integers(case["Lmin"], case["Lmax"] + 1, size=case["n"])
    chis = g.choice([c for c in (8, 16, 24, 32) if c <= case["chimax"]], size=case["n"])
    if case["kind"] == "sweep":
        chis[:] = case["chimax"]
    return [instances.ea_gauss(int(L), int(L), case["beta"], int(c), seed=seed * 1009 + i)
            for i, (L, c) in enumerate(zip(Ls, chis))]


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed, k=0)
    if kind == "step":
        env = binding.Env.from_instance(_instance(case, seed), precisions=(case["precision"],))
        st.update(env=env, chain=binding.init_chains(env, case["chains"], seed=seed + 1, precision=case["precision"]))
    elif kind == "logq":
        env = binding.Env.from_instance(_instance(case, seed), precisions=("f64", case["precision"]))
        st.update(env=env, spins=binding.sample(env, case["B"], seed=seed, precision="f64")[0])
    elif kind == "tune":
        inst = _instance(case, seed)
        env = binding.Env.from_instance(inst, precisions=("f64", "f32"))
        spins = binding.sample(env, case["B"], seed=seed, precision="f64")[0]
        params = torch.tensor(_padded(_build(inst)[0], case), dtype=torch.float32, device="cuda").flatten()
        st.update(env=env, spins=spins, params=params.requires_grad_(True),
                  weights=torch.full((case["B"],), 1.0 / case["B"], dtype=torch.float64, device="cuda"))
    elif kind in ("batch", "sweep"):
        envs = binding.build_envs_batched(_batch_instances(case, seed), precisions=(case["precision"],))
        tile = 64 if kind == "sweep" else 128
        runner = batched.BatchRunner(envs, case["B"], chains=case["chains"], precision=case["precision"], tile=tile,
                                     order="cost", seed=seed, sweeps=1 if kind == "sweep" else 0)
        runner.capture()
        st.update(runner=runner)
    elif kind == "frozen":
        L, D, C = case["L"], case["D"], case["C"]
        Jh, Jv, h, _ = instances.gaussian_ea_torus_batch(n=D, L=L, T=1.0 / case["beta"], seed=seed)
        g = np.random.default_rng([seed, 29])
        start = g.choice(np.array([-1, 1], dtype=np.int8), size=(D, C, L, L))
        st.update(chains=frozen.FrozenLineChains(Jh, Jv, h, case["beta"], case["chi"], start, seed=seed))
    elif kind == "build":
        st.update(inst=_instance(case, seed))
    else:
        inst = instances.cubic_uniform(case["L"], 1.0 / case["T"], case["D"], case["chi"])
        env = binding.Env3D.from_instance(inst, gauge="bond")
        st.update(env=env, chain=binding.init_chains3d(env, case["chains"], seed=seed + 1,
                                                       precision=case["precision"]))
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(state):
    case, seed, k = state["case"], state["seed"], state["k"]
    kind = case["kind"]
    state["k"] = k + 1
    if kind == "step":
        B, C = case["B"], case["chains"]
        env, chain = state["env"], state["chain"]
        sp, lq, E, fl = binding.sample(env, B, seed=seed, sample_offset=k * B, precision=case["precision"])
        acc = binding.mh_step(env, C, B // C, (sp, lq, E), chain, seed=seed, step_offset=k * (B // C))
        return sp, lq, E, fl, acc, chain[0], chain[1], chain[2]
    if kind == "logq":
        return binding.logq(state["env"], state["spins"], precision=case["precision"])
    if kind == "tune":
        lq = autograd.logq(state["params"], state["env"], state["spins"])
        (g,) = torch.autograd.grad((state["weights"] * lq).sum(), state["params"])
        return lq.detach(), g
    if kind in ("batch", "sweep"):
        r = state["runner"]
        r.step()
        return (*r.prop, *r.chain, r.accepted, r.n_accepted)
    if kind == "frozen":
        c = state["chains"]
        acc = c.step()
        return acc, c.spins, c.energy()
    if kind == "build":
        env = binding.Env.from_instance(state["inst"])
        out = binding.sample(env, case["B"], seed=seed, sample_offset=k * case["B"])
        logZ = env.info()["logZ"]
        env.free()
        return (*out, logZ)
    B, C = case["B"], case["chains"]
    env, chain = state["env"], state["chain"]
    sp, lq, E, fl = binding.sample3d(env, B, seed=seed, sample_offset=k * B, precision=case["precision"])
    acc = binding.mh_step3d(env, C, B // C, (sp, lq, E), chain, seed=seed, step_offset=k * (B // C))
    return sp, lq, E, fl, acc, chain[0], chain[1], chain[2]


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _bond(chi, Lx, Ly, r, c):
    return 1 if c <= 0 or c >= Lx else min(chi, 1 << min(c, Lx - c, Ly - r, 30))


def _flops(Ly, Lx, chi):
    """Multiply-adds x 2 of one proposal: a right and a left contraction per site, both spin
    values; the right sweep of row 0 depends on no spin and is shared by all proposals."""
    return float(sum((4 if r == 0 else 8) * _bond(chi, Lx, Ly, r, c) * _bond(chi, Lx, Ly, r, c + 1)
                     for r in range(Ly) for c in range(Lx)))


def _tensor_values(Ly, Lx, chi):
    return sum(2 * _bond(chi, Lx, Ly, r, c) * _bond(chi, Lx, Ly, r, c + 1) for r in range(Ly) for c in range(Lx))


def _build_flops(Ly, Lx, chi):
    """One QR and one SVD factorisation per site of the doubled MPS (m x n: 2 m n min)."""
    f = 0.0
    for r in range(Ly - 1):
        for c in range(Lx):
            m, n = 2 * _bond(chi, Lx, Ly, r + 1, c), 2 * _bond(chi, Lx, Ly, r + 1, c + 1)
            f += 2 * (2 * m) * n * min(2 * m, n) + 4 * m * (2 * _bond(chi, Lx, Ly, r, c + 1)) * m
    return f


def work(case):
    kind = case["kind"]
    size = {"f64": 8, "f32": 4, "bf16": 4}.get(case.get("precision", "f32"), 4)
    if kind in ("step", "logq", "tune"):
        Ly, Lx, chi, B = case["Ly"], case["Lx"], case["chi"], case["B"]
        t = size * _tensor_values(Ly, Lx, chi)
        if kind == "tune":
            return dict(bytes=float(2 * t + B * (Ly * Lx + 16)), flops=3.0 * B * _flops(Ly, Lx, chi))
        return dict(bytes=float(t + B * (Ly * Lx + 21)), flops=B * _flops(Ly, Lx, chi))
    if kind in ("batch", "sweep"):
        L = (case["Lmin"] + case["Lmax"]) // 2
        chis = [c for c in (8, 16, 24, 32) if c <= case["chimax"]] if kind == "batch" else [case["chimax"]]
        rows = case["n"] * (case["B"] + (case["chains"] if kind == "sweep" else 0))
        f = sum(_flops(L, L, c) for c in chis) / len(chis)
        t = size * case["n"] * sum(_tensor_values(L, L, c) for c in chis) / len(chis)
        return dict(bytes=float(t + rows * (L * L + 21)), flops=rows * f)
    if kind == "frozen":
        n, L = case["D"] * case["C"], case["L"] - 1
        return dict(bytes=float(n * (8 * _tensor_values(L, L, case["chi"]) + 2 * L * L)),
                    flops=n * (_build_flops(L, L, case["chi"]) + 2 * _flops(L, L, case["chi"])))
    if kind == "build":
        Ly, Lx, chi = case["Ly"], case["Lx"], case["chi"]
        return dict(bytes=float(8 * _tensor_values(Ly, Lx, chi) + case["B"] * Ly * Lx),
                    flops=_build_flops(Ly, Lx, chi) + case["B"] * _flops(Ly, Lx, chi))
    # a site of the cube is absorbed into a boundary MPS of bond chi, compressed, and drawn
    n, d, x = case["L"] ** 3, 2 * case["D"], case["chi"]
    return dict(bytes=float(n * (4 * 2 * d ** 4 + case["B"])), flops=float(case["B"] * n * 8 * x * x * d * d * d))


# ---------------------------------------------------------------------------
# the same values in 64 bits, from numpy and torch alone
# ---------------------------------------------------------------------------
_SPIN = np.array([-1.0, 1.0])


def _build(inst):
    """Row environments by successive SVD (numpy, LAPACK): M[r][c] and log Z~."""
    Ly, Lx = inst.h.shape
    Jh, Jv, h, beta = inst.Jh, inst.Jv, inst.h, inst.beta
    M, logs = [None] * Ly, 0.0
    for r in range(Ly - 1, -1, -1):
        row = []
        for c in range(Lx):
            if r == Ly - 1:
                t = np.ones((1, 2, 1))
            else:
                t = np.einsum("ts,asb->atb", np.exp(beta * Jv[r, c] * np.outer(_SPIN, _SPIN)), M[r + 1][c])
            t = t * np.exp(beta * h[r, c] * _SPIN)[None, :, None]
            if c > 0:       # the copy of the left neighbour's spin
                G = np.exp(beta * Jh[r, c - 1] * np.outer(_SPIN, _SPIN))
                t = (t[:, None] * G[None, :, :, None]).reshape(2 * t.shape[0], 2, t.shape[2])
            if c < Lx - 1:  # the copy of this site's spin
                t = (t[:, :, :, None] * np.eye(2)[None, :, None, :]).reshape(t.shape[0], 2, 2 * t.shape[2])
            row.append(t)
        for c in range(Lx - 1):
            a, _, b = row[c].shape
            Q, R = np.linalg.qr(row[c].reshape(2 * a, b))
            row[c] = Q.reshape(a, 2, -1)
            s = np.abs(R).max()
            logs += math.log(s)
            row[c + 1] = np.tensordot(R / s, row[c + 1], 1)
        for c in range(Lx - 1, 0, -1):
            a, _, b = row[c].shape
            U, S, Vh = np.linalg.svd(row[c].reshape(a, 2 * b), full_matrices=False)
            k = _bond(inst.chi, Lx, Ly, r, c)
            row[c] = Vh[:k].reshape(k, 2, b)
            logs += math.log(S[0])
            row[c - 1] = np.tensordot(row[c - 1], U[:, :k] * (S[:k] / S[0]), 1)
        s = np.linalg.norm(row[0])
        row[0] = row[0] / s
        logs += math.log(s)
        M[r] = row
    v = np.ones(1)
    for t in M[0]:
        v = v @ t.sum(axis=1)
        logs += math.log(np.abs(v).max())
        v = v / np.abs(v).max()
    return M, logs + math.log(v[0])


def _padded(M, case):
    """[Ly][Lx][P][2][P], zero outside the bond dimensions."""
    Ly, Lx = case["Ly"], case["Lx"]
    P = (max(_bond(case["chi"], Lx, Ly, r, c) for r in range(Ly) for c in range(Lx + 1)) + 3) & ~3
    out = np.zeros((Ly, Lx, P, 2, P))
    for r in range(Ly):
        for c in range(Lx):
            a, _, b = M[r][c].shape
            out[r, c, :a, :, :b] = M[r][c]
    return out


def _uniform(seed, site, sample):
    """The 53 leading bits of the draw of (site, sample): Philox4x32-10, stream 0."""
    lo = 0xFFFFFFFF
    w = [torch.full_like(sample, site >> 1), sample & lo, (sample >> 32) & lo, torch.zeros_like(sample)]
    k0, k1 = seed & lo, (seed >> 32) & lo
    for i in range(10):
        if i:
            k0, k1 = (k0 + 0x9E3779B9) & lo, (k1 + 0xBB67AE85) & lo
        p0, p1 = w[0] * 0xD2511F53, w[2] * 0xCD9E8D57
        w = [((p1 >> 32) & lo) ^ w[1] ^ k0, p1 & lo, ((p0 >> 32) & lo) ^ w[3] ^ k1, p0 & lo]
    x0, x1 = (w[2], w[3]) if site & 1 else (w[0], w[1])
    return ((x1 << 21) | (x0 >> 11)).double() * 2.0 ** -53


def _evaluate(inst, T, B, spins=None, seed=0):
    """log q, energy and spins of B configurations: drawn, or given. T[r][c]: float64 tensors."""
    Ly, Lx = inst.h.shape
    dev = T[0][0].device
    pm = torch.tensor([-1.0, 1.0], dtype=torch.float64, device=dev)
    lq = torch.zeros(B, dtype=torch.float64, device=dev)
    E = torch.zeros(B, dtype=torch.float64, device=dev)
    sample = torch.arange(B, dtype=torch.int64, device=dev)
    one = torch.ones(B, 1, dtype=torch.float64, device=dev)
    above, rows = None, []

    def unit(v):
        return v / v.detach().abs().amax(dim=1, keepdim=True).clamp_min(1e-300)

    for r in range(Ly):
        f = [None if r == 0 else torch.exp(inst.beta * float(inst.Jv[r - 1, c]) * above[:, c:c + 1] * pm)
             for c in range(Lx)]
        R = [None] * (Lx + 1)
        R[Lx] = one
        for c in range(Lx - 1, 0, -1):
            u = torch.einsum("asb,nb->nas", T[r][c], R[c + 1])
            R[c] = unit(u.sum(dim=2) if r == 0 else (u * f[c][:, None, :]).sum(dim=2))
        left, cur = one, []
        for c in range(Lx):
            u = torch.einsum("na,asb->nsb", left, T[r][c])
            if r > 0:
                u = u * f[c][:, :, None]
            w = torch.einsum("nsb,nb->ns", u, R[c + 1]).clamp_min(0.0)
            p = w / w.sum(dim=1, keepdim=True)
            if spins is None:
                s = (_uniform(seed, r * Lx + c, sample) < p[:, 1].detach()).long()
            else:
                s = (spins[:, r, c] > 0).long()
            lq = lq + torch.log(p.gather(1, s[:, None])[:, 0])
            left = unit(u.gather(1, s[:, None, None].expand(-1, 1, u.shape[2]))[:, 0])
            sv = 2.0 * s - 1.0
            loc = torch.full_like(sv, float(inst.h[r, c]), dtype=torch.float64)
            if c > 0:
                loc = loc + float(inst.Jh[r, c - 1]) * cur[-1]
            if r > 0:
                loc = loc + float(inst.Jv[r - 1, c]) * above[:, c]
            E = E - sv * loc
            cur.append(sv.double())
        above = torch.stack(cur, dim=1)
        rows.append(above)
    return lq, E, torch.stack(rows, dim=1)


def exact(case, seed):
    kind = case["kind"]
    # a batch or a torus move is dozens of builds, and a cube's proposal a boundary compression
    # per row and sample: minutes in numpy
    if kind not in ("step", "logq", "tune", "build"):
        return None
    inst = _instance(case, seed)
    M, logZ = _build(inst)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    T = [[torch.tensor(t, device=dev) for t in row] for row in M]
    B = case["B"]
    if kind == "build":
        lq, E, _ = _evaluate(inst, T, B, seed=seed)
        return None, lq, E, None, logZ
    if kind == "step":
        lq, E, _ = _evaluate(inst, T, B, seed=seed)
        return None, lq, E, None, None, None, None, None
    if kind == "logq":
        lq, E, _ = _evaluate(inst, T, B, seed=seed)
        return lq, E, None
    # tune: the tensors are the FP32 parameters the program holds, the states those that the
    # built proposal draws
    with torch.no_grad():
        _, _, spins = _evaluate(inst, T, B, seed=seed)
    T = [[t.float().double().requires_grad_(True) for t in row] for row in T]
    lq, _, _ = _evaluate(inst, T, B, spins=spins)
    g = torch.autograd.grad(lq.mean(), [t for row in T for t in row])
    Lx = case["Lx"]
    g = [[x.cpu().numpy() for x in g[r * Lx:(r + 1) * Lx]] for r in range(case["Ly"])]
    return lq.detach(), torch.tensor(_padded(g, case)).flatten()
