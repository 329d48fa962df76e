"""The work this library is used for, as cases that can be timed and compared.

A flow solver calls the library once per flow step: it advances the chemistry of every cell of its (sub)domain,
by the network with its out-of-distribution guard (``chem_step_ann_props``) or by the plain stiff method
(``chem_step_stiff``), and evaluates the properties the transport equations need (``props_eval``). Beside the
flow step, training data are integrated (``chem_step_stiff``), the network is trained (``mlp_train_step``), and
the network or one of its layers is evaluated alone (``chem_mlp_forward_prec``, ``chem_dense_bf16``).

Sizes: the workloads the repository names (c1: 9 species / 20 reactions, 4,096 cells; c2: 30 / 180, up to
4,194,304 cells, network 1600/800/400; c5: 53 / 325, network 2048/1024/512), subdomains of a few thousand cells,
where launches and latency count, and odd sizes. Cell states follow ``synth.states_profiles`` (c2, c5) and
``synth.states_dirichlet`` (c1), drawn on the device.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_05800_gb300 import binding, synth

DT = 1.0e-6
HIDDEN = {"c1": (256, 128, 64), "c2": (1600, 800, 400), "c5": (2048, 1024, 512)}
# integrator settings of the plain method and of the guard's fallback (loose), of the training data (data), and
# of the library's defaults (tight)
LOOSE = dict(rtol=1e-2, atol_Y=1e-8, atol_T=1e-2, h0=1e-9, max_steps=10000, mode=binding.CHEM_ODE_MIXED)
DATA = dict(rtol=1e-4, atol_Y=1e-10, atol_T=1e-4, h0=1e-9, max_steps=20000)
TIGHT = dict(rtol=1e-6, atol_Y=1e-12, atol_T=1e-6, h0=1e-9, max_steps=10000)
SETTINGS = {"loose": LOOSE, "data": DATA, "tight": TIGHT}
DTYPES = {"f32": binding.CHEM_F32, "f64": binding.CHEM_F64, "f64_in_f32": binding.CHEM_F64_IN_F32}
GUARD_STATES = 2097152      # training states the guard's grids are fitted on
NORM_STATES = 65536         # states the input statistics are taken from
TRAIN_PAIRS = 65536


def listed():
    return [
        # the smallest workload in double precision: the properties of a small box of cells
        {"name": "props c1 f64 4096", "kind": "props", "mech": "c1", "dtype": "f64", "n": 4096, "transport": True},
        # thermal and transport properties of a whole field from the FP64 state, once per flow step
        {"name": "props c2 2M", "kind": "props", "mech": "c2", "dtype": "f64_in_f32", "n": 2097152,
         "transport": True},
        # the larger mechanism on a subdomain of odd size, in single precision
        {"name": "props c5 f32 300001", "kind": "props", "mech": "c5", "dtype": "f32", "n": 300001,
         "transport": True},
        # thermodynamics alone (cp and h), as an energy equation needs between transport updates
        {"name": "thermo c2 1000003", "kind": "props", "mech": "c2", "dtype": "f64_in_f32", "n": 1000003,
         "transport": False},
        # the plain method on the small mechanism with the library's default tolerances
        {"name": "stiff c1 tight 4096", "kind": "stiff", "mech": "c1", "n": 4096, "setting": "tight"},
        # the plain method at its throughput setting
        {"name": "stiff c2 loose 65536", "kind": "stiff", "mech": "c2", "n": 65536, "setting": "loose"},
        # the learned flow step of a whole field: guard, network, fallback, properties
        {"name": "step c2 4M", "kind": "step", "mech": "c2", "prec": "bf16", "n": 4194304, "chunk": 1048576,
         "off": 0.0, "props": True, "tune": True},
        # the same with 2 % of the cells off the trained manifold: the fallback integrates them
        {"name": "step c2 off-manifold 262144", "kind": "step", "mech": "c2", "prec": "bf16", "n": 262144,
         "chunk": 262144, "off": 0.02, "props": False, "tune": False},
        # the learned flow step of a small subdomain: launches and latency
        {"name": "step c2 2500", "kind": "step", "mech": "c2", "prec": "bf16", "n": 2500, "chunk": 4096, "off": 0.0,
         "props": True, "tune": False},
        # the larger mechanism's network alone, in E4M3
        {"name": "forward c5 fp8 500001", "kind": "forward", "mech": "c5", "prec": "fp8", "n": 500001,
         "chunk": 262144},
        # one hidden layer (the 1600 -> 800 layer of the c2 network) on a chunk of cells
        {"name": "dense gelu 262144x800x1600", "kind": "dense", "M": 262144, "N": 800, "K": 1600, "act": 1},
        # one training step at the usual batch
        {"name": "train c2 4096", "kind": "train", "mech": "c2", "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["props", "props", "stiff", "stiff", "step", "step", "forward", "dense", "train"])
    if kind == "props":
        mech = rng.choice(["c1", "c2", "c2", "c5"])
        dtype = rng.choice(["f32", "f64_in_f32", "f64_in_f32", "f64"])
        top = {"c1": 2000000, "c2": 2000000, "c5": 600000}[mech]
        if dtype == "f64":
            top = 20000
        return {"kind": kind, "mech": mech, "dtype": dtype, "n": _log_int(rng, 1000, top),
                "transport": rng.random() < 0.8}
    if kind == "stiff":
        mech = rng.choice(["c1", "c2", "c2", "c5"])
        setting = rng.choice(["loose", "loose", "data", "tight"])
        top = {"c1": {"loose": 60000, "data": 30000, "tight": 8000}, "c2": {"loose": 60000, "data": 8000, "tight": 800},
               "c5": {"loose": 8000, "data": 1000, "tight": 100}}[mech][setting]
        return {"kind": kind, "mech": mech, "n": _log_int(rng, 20, top), "setting": setting}
    if kind == "step":
        mech = rng.choice(["c2", "c2", "c5"])
        n = _log_int(rng, 1000, 2000000 if mech == "c2" else 500000)
        off = rng.choice([0.0, 0.0, 0.01])
        if off:
            n = min(n, 200000)
        return {"kind": kind, "mech": mech, "prec": rng.choice(["bf16", "bf16", "fp8"]), "n": n,
                "chunk": rng.choice([65536, 262144]), "off": off, "props": rng.random() < 0.7, "tune": False}
    if kind == "forward":
        mech = rng.choice(["c2", "c5"])
        return {"kind": kind, "mech": mech, "prec": rng.choice(["bf16", "fp8"]), "n": _log_int(rng, 1000, 500000),
                "chunk": rng.choice([65536, 262144])}
    if kind == "dense":
        return {"kind": kind, "M": _log_int(rng, 1000, 262144), "N": 8 * rng.randint(4, 200),
                "K": 8 * rng.randint(4, 200), "act": rng.choice([0, 1, 1])}
    return {"kind": kind, "mech": rng.choice(["c2", "c2", "c5"]), "batch": 8 * rng.randint(32, 512)}


# --------------------------------------------------------------------------------------------------------------------
# cell states and networks
# --------------------------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, dtype=torch.float64, device="cuda")


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=torch.float64, device="cuda")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _mole_to_mass(X, W):
    Y = X * W[:, None]
    return Y / Y.sum(0, keepdim=True)


def _profiles(m, n, ld, g):
    """The stratified premixed profiles of synth.states_profiles, drawn on the device: (p [ld], S [N + 1][ld]) with
    the state's rows T, Y_1 .. Y_N in S."""
    r, E = m.roles, m.elements
    fuel, ox, bath, water, co2 = r.get("fuel", r["h2"]), r["oxidizer"], r["bath"], r["water"], r.get("co2")
    nC = int(m.elem[fuel, E.index("C")]) if "C" in E else 0
    nH = int(m.elem[fuel, E.index("H")])
    o2 = nC + nH / 4.0
    W = _dev(m.W)
    phi = 0.5 + 0.7 * _rand(g, n)
    c = _rand(g, n)
    Xu = torch.zeros(m.N, n, dtype=torch.float64, device="cuda")
    Xu[fuel], Xu[ox], Xu[bath] = phi / o2, 1.0, 3.76
    burnt = torch.clamp(1.0 / phi, max=1.0) * Xu[fuel]
    Xb = Xu.clone()
    Xb[fuel] -= burnt
    Xb[ox] = torch.clamp(Xb[ox] - burnt * o2, min=0.0)
    Xb[water] += burnt * nH / 2.0
    if co2 is not None:
        Xb[co2] += burnt * nC
    Yu, Yb = _mole_to_mass(Xu, W), _mole_to_mass(Xb, W)
    dh = -((Yb - Yu) * _dev(m.hf298 / m.W)[:, None]).sum(0)
    Tb = torch.clamp(300.0 + dh / 1400.0, 1200.0, 2700.0)
    S = torch.zeros(m.N + 1, ld, dtype=torch.float64, device="cuda")
    S[0, :n] = 300.0 + c * (Tb - 300.0)
    Y = (1.0 - c) * Yu + c * Yb
    del Xu, Xb, Yu, Yb
    amp = 10.0 ** np.random.default_rng(7000 + m.N).uniform(-6.0, -2.0, m.N)
    bump = 4.0 * c * (1.0 - c)
    for k in range(m.N):
        if k not in (fuel, ox, bath, water, co2):
            Y[k] += amp[k] * bump * (0.5 + _rand(g, n)) + 1e-12
    Y *= torch.exp(0.05 * _randn(g, m.N, n))
    S[1:, :n] = Y / Y.sum(0, keepdim=True)
    p = torch.zeros(ld, dtype=torch.float64, device="cuda")
    p[:n] = synth.P_ATM
    return p, S


def _states(m, n, ld, seed):
    if m.name == "c1":
        T, p, Y = synth.states_dirichlet(m, n, seed, ld)
        return _dev(p), _dev(np.concatenate([T[None], Y]))
    return _profiles(m, n, ld, _gen(seed))


def _off_manifold(S, n, frac, g):
    """synth.perturb_off_manifold on the device: a fraction of the cells, T +- 300 K and Y exp(0.2 xi)."""
    idx = torch.randperm(n, generator=g, device="cuda")[:int(round(frac * n))]
    sign = torch.where(_rand(g, idx.numel()) < 0.5, -1.0, 1.0)
    S[0, idx] = torch.clamp(S[0, idx] + 300.0 * sign, min=250.0)
    Y = S[1:, idx] * torch.exp(0.2 * _randn(g, S.shape[0] - 1, idx.numel()))
    S[1:, idx] = Y / Y.sum(0, keepdim=True)


def _features(p, S, n):
    return torch.cat([S[:1, :n], p[None, :n], (torch.clamp(S[1:, :n], min=0.0) ** 0.1 - 1.0) / 0.1])


def _norm(m):
    """Z-score statistics of one sample of training states: inputs from the states, outputs at the size of the change
    over dt (a few per mille of a species' spread). The same for every seed of a mechanism, as a trained network's."""
    p, S = _states(m, NORM_STATES, NORM_STATES, 424242)
    x = _features(p, S, NORM_STATES)
    sd = x.std(1, correction=0)
    sd[sd < 1e-12] = 1.0
    out = [k for k in range(m.N) if k != m.bath]
    sdu = 5e-3 * S[1:].std(1, correction=0)[out] + 1e-12
    return [v.cpu().numpy() for v in (x.mean(1), sd, torch.zeros_like(sdu), sdu)]


_NORM, _GUARD = {}, {}


def _net(dm, m, chunk, max_batch, seed):
    net = binding.Mlp(dm, hidden=HIDDEN[m.name], dt=DT, seed=seed, chunk=chunk, max_batch=max_batch)
    if m.name not in _NORM:
        _NORM[m.name] = _norm(m)
    net.set_norm(*_NORM[m.name])
    return net


def _fit_guard(net, dm, m):
    if m.name not in _GUARD:      # the training states, held once for all networks of this process
        _GUARD[m.name] = _states(m, GUARD_STATES, GUARD_STATES, 2103)
    p, S = _GUARD[m.name]
    binding.chem_mlp_fit_ood_multi(net, dm, GUARD_STATES, GUARD_STATES, S[0], p, S[1:],
                                   [m.roles["oxidizer"], m.roles["co2"]], nbins=64, min_count=1)


# --------------------------------------------------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "dense":
        g = _gen(seed)
        M, N, K = case["M"], case["N"], case["K"]
        f = dict(generator=g, dtype=torch.float32, device="cuda")
        x = torch.nn.functional.gelu(torch.randn(M, K, **f)).to(torch.bfloat16)
        W = ((2.0 * torch.rand(N, K, **f) - 1.0) * (1.7 / math.sqrt(K))).to(torch.bfloat16)
        b = (2.0 * torch.rand(-(-N // 16) * 16, **f) - 1.0) / math.sqrt(K)
        y = torch.zeros(M, N, dtype=torch.bfloat16 if case["act"] else torch.float32, device="cuda")
        return {"case": case, "x": x, "W": W, "b": b, "y": y}
    m = synth.get_mech(case["mech"])
    dm = binding.Mech(m)
    st = {"case": case, "m": m, "mech": dm}
    if kind == "train":
        n = TRAIN_PAIRS
        g = _gen(seed)
        st["ld"] = n
        st["p"], st["S"] = _profiles(m, n, n, g)
        Y1 = st["S"][1:] * torch.exp(0.02 * _randn(g, m.N, n))
        st["Y1"] = Y1 / Y1.sum(0, keepdim=True)
        st["idx"] = torch.randperm(n, generator=g, device="cuda")[:case["batch"]].to(torch.int32)
        st["loss"] = torch.zeros(4, dtype=torch.float32, device="cuda")
        net = binding.Mlp(dm, hidden=HIDDEN[m.name], dt=DT, seed=seed, chunk=4096, max_batch=4096)
        binding.chem_mlp_fit_norm(net, n, n, st["S"][0], st["p"], st["S"][1:], st["Y1"])
        st["net"] = net
        st["grads"] = binding.grad_buffers(net)
        for t in st["grads"]:
            t.owner = net      # views of the handle's memory: the handle lives as long as they do
        st["first"] = net.get_params()
        return st
    n = case["n"]
    ld = st["ld"] = synth.padded_ld(n)
    st["p"], S0 = _states(m, n, ld, seed)
    if kind == "props":
        dt = torch.float64 if case["dtype"] == "f64" else torch.float32
        if case["dtype"] == "f32":
            st["p"], S0 = st["p"].float(), S0.float()
        st["S"] = S0
        out = torch.zeros(4 + m.N, ld, dtype=dt, device="cuda")
        st["cp"], st["h"], st["mu"], st["lam"], st["Dk"] = out[0], out[1], out[2], out[3], out[4:]
        return st
    if kind == "stiff":
        st["S0"], st["S"] = S0, torch.zeros_like(S0)
        st["status"] = torch.zeros(ld, dtype=torch.int32, device="cuda")
        st["opts"] = binding.make_opts(**SETTINGS[case["setting"]])
        return st
    net = st["net"] = _net(dm, m, case["chunk"], 4096, seed)
    if case["prec"] == "fp8":
        k = min(n, 16384)
        pc, Sc = _profiles(m, k, synth.padded_ld(k), _gen(seed + 1))
        binding.chem_mlp_calibrate_fp8(net, k, Sc.shape[1], Sc[0], pc, Sc[1:])
    st["prec"] = binding.CHEM_PREC_FP8 if case["prec"] == "fp8" else binding.CHEM_PREC_BF16
    if kind == "forward":
        st["S"] = S0
        st["u"] = torch.zeros(n, -(-(m.N - 1) // 8) * 8, dtype=torch.float32, device="cuda")
        return st
    if case["off"]:
        _off_manifold(S0, n, case["off"], _gen(seed + 2))
    _fit_guard(net, dm, m)
    if case["tune"]:
        binding.chem_mlp_autotune(net, min(case["chunk"], 262144))
    st["S0"], st["S"] = S0, torch.zeros_like(S0)
    st["status"] = torch.zeros(ld, dtype=torch.int32, device="cuda")
    st["opts"] = binding.make_opts(**LOOSE)
    if case["props"]:
        out = torch.zeros(4 + m.N, ld, dtype=torch.float32, device="cuda")
        st["props"] = [out[0], out[1], out[2], out[3], out[4:]]
    else:
        st["props"] = [None] * 5
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "dense":
        M, N, K = case["M"], case["N"], case["K"]
        binding.chem_dense_bf16(M, N, K, st["x"], K, st["W"], K, st["b"], case["act"], st["y"], N)
        return st["y"]
    if kind == "train":
        S = st["S"]
        binding.mlp_train_step(st["net"], case["batch"], st["idx"], st["ld"], S[0], st["p"], S[1:], st["Y1"], 1e-5,
                               st["loss"])
        return [st["loss"][:1], st["grads"]]
    n, ld, S, p = case["n"], st["ld"], st["S"], st["p"]
    if kind == "props":
        t = case["transport"]
        binding.props_eval(st["mech"], n, ld, DTYPES[case["dtype"]], S[0], p, S[1:], st["cp"], st["h"],
                           st["mu"] if t else None, st["lam"] if t else None, st["Dk"] if t else None)
        return [st["cp"], st["h"]] + ([st["mu"], st["lam"], st["Dk"]] if t else [])
    if kind == "forward":
        binding.chem_mlp_forward_prec(st["net"], st["prec"], n, ld, S[0], p, S[1:], st["u"], st["u"].shape[1])
        return st["u"]
    # the chemistry steps advance the state in place; the solver keeps the state before the step
    S.copy_(st["S0"])
    if kind == "stiff":
        binding.chem_step_stiff(st["mech"], n, ld, DT, st["opts"], S[0], p, S[1:], st["status"])
        return [S[0], S[1:], st["status"]]
    binding.chem_step_ann_props(st["mech"], st["net"], n, ld, DT, st["prec"], st["opts"], S[0], p, S[1:],
                                st["status"], *st["props"])
    return [S[0], S[1:], st["status"]] + [v for v in st["props"] if v is not None]


def _step_flops(m, settings_steps):
    """Operations of one cell's integration: attempted steps times one step of the four-stage Rosenbrock method
    (3 right-hand sides, the analytic Jacobian, the factorisation and four solves; exp and log counted as 20)."""
    N, R, n = m.N, m.R, m.N + 1
    ntb, ntroe = int((m.rtype != 0).sum()), int((m.rtype == 2).sum())
    rhs = 20 * N + 52 * R + 2 * N * ntb + 130 * ntroe
    jac = 4 * n * n + 12 * N * ntb + 72 * R
    return settings_steps * (3 * rhs + jac + 2.0 / 3.0 * n ** 3 + 8 * n * n)


STEPS = {"loose": 13, "data": 55, "tight": 190}     # attempted steps a cell takes in dt, about


def work(case):
    kind = case["kind"]
    if kind == "dense":
        M, N, K = case["M"], case["N"], case["K"]
        return {"bytes": 2.0 * (M * K + N * K) + M * N * (2.0 if case["act"] else 4.0), "flops": 2.0 * M * N * K}
    m = synth.get_mech(case["mech"])
    N = m.N
    w = [N + 2] + list(HIDDEN[m.name]) + [N - 1]
    mac = sum(a * b for a, b in zip(w[:-1], w[1:]))
    if kind == "train":
        B = case["batch"]
        nw = mac + sum(w[1:])
        return {"bytes": B * (2 * N + 2) * 8.0 + nw * 4.0 * 8, "flops": B * 2.0 * (3 * mac - w[0] * w[1])}
    n = case["n"]
    props = 16.0 * N * N + 30.0 * N
    if kind == "props":
        i, o = {"f32": (4, 4), "f64": (8, 8), "f64_in_f32": (8, 4)}[case["dtype"]]
        if not case["transport"]:
            return {"bytes": n * ((N + 1.0) * i + 2 * o), "flops": n * 24.0 * N}
        return {"bytes": n * ((N + 2.0) * i + (4 + N) * o), "flops": n * props}
    if kind == "stiff":
        return {"bytes": n * (2 * N + 3) * 8.0, "flops": n * _step_flops(m, STEPS[case["setting"]])}
    if kind == "forward":
        return {"bytes": n * ((N + 2) * 8.0 + (N - 1) * 4.0), "flops": n * 2.0 * mac}
    # the copy of the state before the step, the step, the fallback of the off-manifold cells, the properties
    fl = n * (2.0 * mac + 24.0 * N * 4) + n * case["off"] * _step_flops(m, 2 * STEPS["loose"])
    by = n * ((N + 1) * 8.0 * 2 + (2 * N + 3) * 8.0 + 4.0)
    if case["props"]:
        fl += n * props
        by += n * (4 + N) * 4.0
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------------------------------------------------
# the same in plain torch, 64 bits
# --------------------------------------------------------------------------------------------------------------------

def _gelu(z):
    return 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))


def _exact_props(m, S, p, transport):
    """NASA-7 cp and h, Wilke viscosity, conductivity with Eucken species values and Wilke weights, and
    Hirschfelder-Curtiss diffusivities, species by species."""
    T, Y = S[0].double(), S[1:].double()
    R, W = synth.R_GAS, _dev(m.W)
    lo, hi = _dev(m.nasa_lo), _dev(m.nasa_hi)
    high = T >= synth.T_MID
    S1 = (Y / W[:, None]).sum(0)
    X = Y / W[:, None] / S1
    cp, h = torch.zeros_like(T), torch.zeros_like(T)
    cpR = []
    for k in range(m.N):
        a = [torch.where(high, hi[k, j], lo[k, j]) for j in range(6)]
        c = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4])))
        hk = T * (a[0] + T * (a[1] / 2 + T * (a[2] / 3 + T * (a[3] / 4 + T * a[4] / 5)))) + a[5]
        cpR.append(c)
        cp += Y[k] / W[k] * c * R
        h += Y[k] / W[k] * hk * R
    if not transport:
        return cp, h
    x = torch.log(T / 1000.0)
    vf, df = _dev(m.visc_fit), _dev(m.diff_fit)
    mu_k = [torch.exp(sum(vf[k, j] * x ** j for j in range(5))) for k in range(m.N)]
    mu, lam, Dk = torch.zeros_like(T), torch.zeros_like(T), torch.zeros_like(Y)
    for k in range(m.N):
        den, res, all_g = torch.zeros_like(T), torch.zeros_like(T), torch.zeros_like(T)
        for j in range(m.N):
            phi = (1.0 + torch.sqrt(mu_k[k] / mu_k[j]) * (W[j] / W[k]) ** 0.25) ** 2 / torch.sqrt(8.0 * (1.0 + W[k] / W[j]))
            den += X[j] * phi
            if j != k:
                g = sum(df[k, j, i] * x ** i for i in range(5))
                res += g * X[j]
                all_g += g
        mu += X[k] * mu_k[k] / den
        lam += X[k] * mu_k[k] / W[k] * (cpR[k] + 1.25) * R / den
        pure = (1.0 - X[k]) < 1e-12
        Dk[k] = torch.where(pure, T ** 1.5 / (p.double() * all_g / max(1, m.N - 1)), (1.0 - Y[k]) * T ** 1.5 / (p.double() * res))
    return cp, h, mu, lam, Dk


def _exact_layers(m, flat):
    w = [m.N + 2] + list(HIDDEN[m.name]) + [m.N - 1]
    return [(_dev(a), _dev(b)) for a, b in synth.unflatten(flat, w)]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("stiff", "step"):        # adaptive integration of every cell: minutes without this library
        return None
    st = prepare(case, seed)
    if kind == "dense":
        x, W = st["x"].double(), st["W"].double()
        y = torch.cat([c @ W.T + st["b"][:case["N"]].double() for c in x.split(32768)])
        return _gelu(y) if case["act"] else y
    m = st["m"]
    if kind == "props":
        n, ld = case["n"], st["ld"]
        got = [[], [], [], [], []]
        for c0 in range(0, n, 1 << 20):
            c1 = min(n, c0 + (1 << 20))
            for out, v in zip(got, _exact_props(m, st["S"][:, c0:c1], st["p"][c0:c1], case["transport"])):
                out.append(v)
        return [torch.nn.functional.pad(torch.cat(v, -1), (0, ld - n)) for v in got if v]
    if kind == "forward":
        n = case["n"]
        mu_x, sd_x = (_dev(v) for v in st["net"].get_norm()[:2])
        layers = _exact_layers(m, st["net"].get_params())
        u = torch.zeros(n, st["u"].shape[1], dtype=torch.float64, device="cuda")
        for c0 in range(0, n, 65536):
            c1 = min(n, c0 + 65536)
            z = ((_features(st["p"][c0:c1], st["S"][:, c0:c1], c1 - c0).T - mu_x) / sd_x)
            for i, (W, b) in enumerate(layers):
                z = z @ W.T + b
                z = _gelu(z) if i < 3 else z
            u[c0:c1, :m.N - 1] = z
        return u
    # training: the loss of the first step and its gradients at the initial parameters, rows padded to 8
    rows = st["idx"].long()
    mu_x, sd_x, mu_u, sd_u = (_dev(v) for v in st["net"].get_norm())
    z = (_features(st["p"][rows], st["S"][:, rows], rows.numel()).T - mu_x) / sd_x
    out = [k for k in range(m.N) if k != m.bath]
    target = ((st["Y1"] - st["S"][1:])[out][:, rows].T - mu_u) / sd_u
    layers = [(W.requires_grad_(), b.requires_grad_()) for W, b in _exact_layers(m, st["first"])]
    for i, (W, b) in enumerate(layers):
        z = z @ W.T + b
        z = _gelu(z) if i < 3 else z
    loss = (z - target).abs().sum() / rows.numel()
    loss.backward()
    grads = []
    for (W, b), gb in zip(layers, st["grads"][1::2]):
        W, b = W.grad, b.grad
        grads += [torch.nn.functional.pad(W, (0, -W.shape[1] % 8)).reshape(-1),
                  torch.nn.functional.pad(b, (0, gb.numel() - b.numel()))]
    return [loss.detach()[None], grads]
