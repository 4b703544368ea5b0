"""What this library is asked to do in earnest, as cases that can be timed and compared.

A case is one call sequence of a user's program on inputs that lie on the GPU (or in pinned host
memory where the case says so): a block of molecular-dynamics samples is pushed into a handle
whose basis and bins are loaded, and the result of the method is read.  `listed()` names the
cases, `draw()` gives more of the same ranges, `prepare()` makes what the program has in hand
before the call, `run()` is one pass, `work()` counts what a pass cannot do without, and
`exact()` gives the results in 64 bits from plain torch.

Inputs follow the recipes of paper_2102_03691_gb300/synth.py (Maxwell-Boltzmann velocities,
Gaussian virials, both AR(1) in time, natural or single isotopes, i.i.d. uniform frequencies),
drawn on the GPU.  The basis is an orthonormal cosine basis with random signs of the degrees of
freedom and random mode order: plane-wave-like as lattice modes are, and quick to make.

The Green-Kubo, HNEMA and SHC read-outs come from the library as doubles that hold results of
single-precision currents; the passes hand them on in single precision, as a program that stores
or plots them does.  Which d-axis split the library's autotuner picks, and with it the order of
the single-precision sums, may differ between two processes.
"""
import math

import numpy as np
import torch

from paper_2102_03691_gb300.mhc import ModalHeatCurrent, ModalHeatCurrentGroup, SpectralHeatCurrent

DEV = "cuda"
KB = 8.617333262145179e-5          # eV/K
A2_PS2_PER_EV_AMU = 9648.533212331  # 1 eV/amu in A^2/ps^2
WMK = 1602.176634                  # 1 eV/(ps A K) in W/(m K)
T_K, FE = 300.0, (1e-5, 0.0, 0.0)
SI = (27.9769265, 0.922, 28.9764947, 0.047, 29.9737702, 0.031)
RHO = 0.9                          # AR(1) coefficient of v and W between samples

# Atom counts of the uneven batch of 16 CNT-like systems (synth.cnt_group_sizes()).
CNT16 = "3200,1800,680,1720,3240,520,3200,1640,2480,2960,3280,3720,920,4000,3720,2000"


def listed():
    return [
        # the smallest call: a small cell, a short block, GKMA with its window read; launches and
        # host time count
        dict(name="gkma_small", kind="push", N=64, M=192, K=32, B=8, L=8, precision="fp16x3",
             read="window"),
        # ordinary: Si-like 512 atoms, the whole 1000-step run as one block, kappa(tau) curves read
        dict(name="gkma_si_n512", kind="push", N=512, M=1536, K=1000, B=100, L=200,
             precision="fp16x3", read="tau"),
        # the same system streamed from pinned host memory, as an MD engine on the host hands it over
        dict(name="gkma_si_n512_host", kind="push", N=512, M=1536, K=1000, B=100, L=200,
             precision="fp16x3", read="window", host=True),
        # odd and ragged in every size, a mode subset, the binding's default precision
        dict(name="gkma_ragged_n1003", kind="push", N=1003, M=2777, K=77, B=37, L=123,
             precision="bf16x3", read="window"),
        # graphene-like HNEMA in blocks of 128 steps
        dict(name="hnema_graphene_n4096", kind="push", N=4096, M=12288, K=128, B=200, L=0,
             precision="fp16x3", read="hnema"),
        # the same in FP32
        dict(name="hnema_graphene_n4096_fp32", kind="push", N=4096, M=12288, K=128, B=200, L=0,
             precision="fp32", read="hnema"),
        # the in-plane / out-of-plane split of the same system
        dict(name="hnema_graphene_n4096_direction", kind="push", N=4096, M=12288, K=128, B=200,
             L=0, precision="fp16x3", read="hnema", direction=True),
        # the 8000-atom Si system with all its modes, GKMA with 500 lags
        dict(name="gkma_si_n8000", kind="push", N=8000, M=24000, K=256, B=64, L=500,
             precision="fp16x3", read="window"),
        # mode subset of a 20000-atom system: the largest call
        dict(name="gkma_subset_n20000", kind="push", N=20000, M=6000, K=512, B=64, L=1000,
             precision="fp16x3", read="window"),
        # bin-bin cross-correlations over a whole run of four blocks, with their read-out
        dict(name="xcorr_si_n512", kind="xcorr", N=512, M=1536, K=250, B=64, L=200, blocks=4,
             precision="fp16x3"),
        # 16 systems of uneven size in one grouped push
        dict(name="hnema_cnt_group16", kind="group", sizes=CNT16, K=256, B=52,
             precision="fp16x3"),
        # spectral heat current of 8000 atoms: 250 lags, a 241-frequency spectrum
        dict(name="shc_si_n8000", kind="shc", N=8000, K=256, nc=250, n_freq=241,
             precision="fp16x3"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["gkma", "gkma", "hnema", "fp32", "direction", "host", "xcorr", "group", "shc"])
    if kind == "shc":
        return dict(kind="shc", N=_log(rng, 100, 9000), K=rng.randint(16, 256),
                    nc=rng.randint(20, 300), n_freq=rng.randint(60, 300),
                    precision=rng.choice(["fp16x3", "bf16x3"]))
    if kind == "group":
        n = rng.randint(2, 16)
        sizes = [40 * rng.randint(12, 100) for _ in range(n)]
        if rng.random() < 0.3:
            sizes[0] += rng.randint(1, 39)
        return dict(kind="group", sizes=",".join(map(str, sizes)), K=rng.randint(32, 256),
                    B=rng.randint(10, 60), precision=rng.choice(["fp16x3", "bf16x3"]))
    if kind == "xcorr":
        N = _log(rng, 60, 700)
        return dict(kind="xcorr", N=N, M=3 * N, K=rng.randint(32, 256), B=rng.randint(4, 72),
                    L=rng.randint(8, 250), blocks=rng.randint(1, 4), precision="fp16x3")
    # single handles; FP32 and the direction split up to the graphene size, the rest up to Si-8000
    top = {"fp32": 3500, "direction": 4100, "host": 1500}.get(kind, 8000)
    N = _log(rng, 60, top)
    if rng.random() < 0.5:
        N = max(64, N // 4 * 4)
    M = 3 * N if rng.random() < 0.6 else rng.randint(max(1, N // 2), 3 * N)
    K = rng.randint(100, 1000) if N < 700 else rng.randint(16, 128 if kind in ("fp32", "direction") else 256)
    hnema = kind in ("hnema", "direction", "fp32") and rng.random() < 0.7
    c = dict(kind="push", N=N, M=M, K=K, B=rng.randint(8, 200), L=0 if hnema else rng.randint(8, 500),
             precision="fp32" if kind == "fp32" else rng.choice(["fp16x3", "fp16x3", "bf16x3"]),
             read="hnema" if hnema else rng.choice(["window", "tau"]))
    if kind == "direction":
        c["direction"] = True
    if kind == "host":
        c["host"] = True
    return c


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _basis(N, M, g):
    """Orthonormal E [3N][M] float32: s_d c_n cos(pi (2 d + 1) n / (2 D)) for M of the D
    wave numbers n in random order, s_d a random sign."""
    D = 3 * N
    tab = torch.cos(torch.arange(4 * D, device=DEV, dtype=torch.float64) * (math.pi / (2 * D)))
    tab = (tab * math.sqrt(2.0 / D)).float()
    n = torch.randperm(D, generator=g, device=DEV)[:M]
    sign = (torch.randint(0, 2, (D,), generator=g, device=DEV) * 2 - 1).float()
    scale = torch.where(n == 0, math.sqrt(0.5), 1.0).float()
    E = torch.empty((D, M), device=DEV)
    step = max(1, (1 << 26) // M)
    for d0 in range(0, D, step):
        d = torch.arange(d0, min(D, d0 + step), device=DEV)
        E[d0:d0 + step] = tab[((2 * d + 1)[:, None] * n[None, :]) % (4 * D)]
    E *= sign[:, None]
    E *= scale[None, :]
    return E


def _masses(N, si, g):
    if not si:
        return np.full(N, 12.011)
    u = torch.rand(N, generator=g, device=DEV, dtype=torch.float64).cpu().numpy()
    return np.where(u < SI[1], SI[0], np.where(u < SI[1] + SI[3], SI[2], SI[4]))


def _samples(mass, K, g):
    """v [K][N][3], W [K][N][9] float32: AR(1) sequences written as one matrix product."""
    N = len(mass)
    k = torch.arange(K, device=DEV, dtype=torch.float64)
    a = torch.where(k[:, None] >= k[None, :], RHO ** (k[:, None] - k[None, :]).clamp(min=0), 0.0)
    a[:, 1:] *= math.sqrt(1.0 - RHO * RHO)
    a = a.float()
    sv = torch.from_numpy(np.sqrt(KB * T_K / mass * A2_PS2_PER_EV_AMU)).to(DEV).float()
    v = (a @ torch.randn(K, 3 * N, generator=g, device=DEV)).view(K, N, 3) * sv[None, :, None]
    W = (a @ torch.randn(K, 9 * N, generator=g, device=DEV)).view(K, N, 9)
    return v.contiguous(), W.contiguous()


def _f_max(case):
    return 16.0 if case.get("L", 0) or case["kind"] == "xcorr" else 52.0


def _system(N, M, K, f_max, si, g, blocks=1):
    mass = _masses(N, si, g)
    E = _basis(N, M, g)
    f = torch.rand(M, generator=g, device=DEV, dtype=torch.float64).cpu().numpy() * f_max
    data = [_samples(mass, K, g) for _ in range(blocks)]
    return mass, E, f, data


def _volume(N, case):
    return N * (20.02 if _f_max(case) == 16.0 or case["kind"] == "shc" else 8.77)


DT = 0.01        # ps between samples (SHC: 0.002)
DT_SHC = 0.002


def _inputs(case, seed):
    """What both prepare() and exact() start from."""
    g = _gen(seed)
    kind = case["kind"]
    if kind == "shc":
        mass = _masses(case["N"], True, g)
        return mass, _samples(mass, case["K"], g)
    if kind == "group":
        return [_system(n, 3 * n, case["K"], _f_max(case), False, g)
                for n in map(int, case["sizes"].split(","))]
    return _system(case["N"], case["M"], case["K"], _f_max(case), _f_max(case) == 16.0, g,
                   case.get("blocks", 1))


def _window(case):
    hi = (case["L"] - 1) * DT
    return 0.8 * hi, hi


def _handle(case, N, mass, E, f, **kw):
    h = ModalHeatCurrent(precision=case["precision"], k_max=case["K"], n_lags=case.get("L", 0),
                         dt_ps=DT, T_K=T_K, V_A3=_volume(N, case), F_e=FE, **kw)
    h.set_modes(E, mass, f)
    h.set_bins_uniform(0.0, _f_max(case), case["B"])
    return h


def prepare(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    f64 = dict(device=DEV, dtype=torch.float64)
    if kind == "shc":
        s = SpectralHeatCurrent(case["N"], case["nc"], k_max=case["K"], dt_ps=DT_SHC, T_K=T_K,
                                V_A3=_volume(case["N"], case), F_e=FE, precision=case["precision"])
        return dict(case=case, shc=s, v=data[1][0], W=data[1][1],
                    f=np.linspace(0.0, 60.0, case["n_freq"]),
                    kappa=torch.empty((9, case["n_freq"]), **f64))
    if kind == "group":
        hs = [_handle(case, len(m), m, E, f) for m, E, f, _ in data]
        n = sum(h.B * 3 for h in hs)
        return dict(case=case, hs=hs, group=ModalHeatCurrentGroup(hs),
                    v=[d[3][0][0] for d in data], W=[d[3][0][1] for d in data],
                    kappa=torch.empty(n, **f64), mean=torch.empty(n, **f64))
    mass, E, f, blocks = data
    h = _handle(case, case["N"], mass, E, f, direction=bool(case.get("direction")),
                xcorr=kind == "xcorr")
    if case.get("host"):
        blocks = [(v.cpu().pin_memory(), W.cpu().pin_memory()) for v, W in blocks]
    st = dict(case=case, h=h, blocks=blocks)
    rows = ((3,) if case.get("direction") else ()) + (case["B"],)
    if kind == "push":
        if case["read"] == "hnema":
            st["kappa"], st["mean"] = torch.empty(rows + (3,), **f64), torch.empty(rows + (3,), **f64)
        else:
            st["kw"] = torch.empty(rows + (3, 3), **f64)
            st["Jb"] = torch.empty((case["K"],) + rows + (3,), device=DEV)
            if case["read"] == "tau":
                st["kt"] = torch.empty(rows + (3, 3, case["L"]), **f64)
    return st


# ------------------------------------------------------------------------------ one pass
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "shc":
        s["shc"].push(s["v"], s["W"])
        return {"kappa": s["shc"].read_kappa(s["f"], 0, out=s["kappa"]).float()}
    if kind == "group":
        s["group"].push(s["v"], s["W"])
        s["group"].read_hnema(s["kappa"], s["mean"])
        return {"kappa": s["kappa"].float(), "mean": s["mean"].float()}
    h = s["h"]
    if kind == "xcorr":   # a whole run in blocks, then the pairs' window averages
        for v, W in s["blocks"]:
            h.push(v, W)
        _, kw = h.read_kappa_xcorr(*_window(case), with_tau=False)
        return {"kappa_xcorr": kw.astype(np.float32)}
    v, W = s["blocks"][0]
    h.push(v, W, async_inputs=bool(case.get("host")))
    if case["read"] == "hnema":
        h.read_hnema_into(s["kappa"], s["mean"])
        return {"kappa": s["kappa"].float(), "mean": s["mean"].float()}
    # GKMA: the block's binned currents (what the method writes out) and kappa
    h.read_binned_current(s["Jb"])
    kt = s.get("kt")
    h.read_kappa_gk_into(s["kw"], *_window(case), kappa_tau=kt)
    out = {"Jb": s["Jb"], "kappa_w": s["kw"].float()}
    if kt is not None:
        out["kappa_tau"] = kt.float()
    return out


# ------------------------------------------------------------------------------ what a pass needs
def work(case):
    """Bytes: the basis as single precision, the samples and the correlation state read once, the
    results (and that state) written once.  Flops: the method's products, 24 a mode, atom and
    step (Eqs. 13 and 16), 18 a bin and lag and step (Eq. 17), 18 an atom, lag and step (SHC)."""
    K = case["K"]
    if case["kind"] == "shc":
        N, nc = case["N"], case["nc"]
        return {"bytes": 48.0 * N * K + 36.0 * N * (nc - 1) + 8.0 * 9 * (2 * nc + case["n_freq"]),
                "flops": 18.0 * N * nc * K + 18.0 * nc * case["n_freq"]}
    if case["kind"] == "group":
        sizes = list(map(int, case["sizes"].split(",")))
        return {"bytes": sum(36.0 * n * n + 48.0 * n * K + 48.0 * case["B"] for n in sizes),
                "flops": sum(72.0 * n * n * K for n in sizes)}
    N, M, B, L = case["N"], case["M"], case["B"], case["L"]
    rows = B * (3 if case.get("direction") else 1)
    nb = case.get("blocks", 1)
    by = nb * (12.0 * N * M + 48.0 * N * K)
    fl = nb * 24.0 * M * N * K
    if L:
        by += nb * 2 * 72.0 * rows * L + 72.0 * rows
        fl += nb * 18.0 * rows * L * K
    if case["kind"] == "xcorr":
        by += nb * 2 * 72.0 * B * B * L + 72.0 * B * B
        fl += nb * 18.0 * B * B * L * K
        return {"bytes": by, "flops": fl}
    if case["read"] == "hnema":
        by += 48.0 * rows
    else:
        by += 12.0 * rows * K + (72.0 * rows * L if case["read"] == "tau" else 0.0)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------ 64-bit results
def _currents(case, mass, E, f, v, W):
    """Binned currents [K][rows][3] and the total current [K][3]."""
    N, K, B = len(mass), v.shape[0], case["B"]
    m = torch.from_numpy(mass).to(DEV)
    v, W = v.double(), W.double().view(K, N, 3, 3)
    J = torch.einsum("kiab,kib->ka", W, v)
    w = _f_max(case) / B
    b = np.minimum(np.floor(f / w).astype(np.int64), B - 1)
    dirs = 3 if case.get("direction") else 1
    Jb = torch.zeros((K, dirs, B, 3), device=DEV, dtype=torch.float64)
    xv = (v * m.sqrt()[None, :, None]).reshape(K, 3 * N)
    Wm = W / m.sqrt()[None, :, None, None]
    step = max(1, (1 << 28) // (3 * N))
    for n0 in range(0, E.shape[1], step):
        e = E[:, n0:n0 + step].double()
        ids = torch.from_numpy(b[n0:n0 + step]).to(DEV)
        x = xv @ e
        for a in range(3):
            for q in range(dirs):
                if dirs == 1:
                    y = Wm[:, :, a, :].reshape(K, 3 * N) @ e
                else:
                    y = Wm[:, :, a, q] @ e[q::3]
                Jb[:, q, :, a].index_add_(1, ids, x * y)
        del e
    return Jb.view(K, dirs * B, 3), J


def _hnema(case, N, Jb):
    mean = Jb.mean(0)
    return mean * (WMK / (T_K * _volume(N, case) * FE[0])), mean


def _correlate(A, B, L):
    """sum_{t >= l} A[t][i] B[t-l][j] for l < L: [L][i][j]."""
    T = A.shape[0]
    out = torch.zeros((L, A.shape[1], B.shape[1]), device=DEV, dtype=torch.float64)
    for l in range(min(L, T)):
        out[l] = A[l:].T @ B[:T - l]
    return out


def _green_kubo(case, C, T):
    """kappa(tau) [L][...] and its window average from the sums C [L][...] of T samples."""
    L = C.shape[0]
    cnt = torch.clamp(T - torch.arange(L, device=DEV, dtype=torch.float64), min=0)
    c = C * torch.where(cnt > 0, 1.0 / cnt.clamp(min=1), 0.0).view(-1, *([1] * (C.dim() - 1)))
    coef = WMK / (KB * T_K * T_K * _volume(case["N"], case)) * DT
    kt = torch.zeros_like(c)
    kt[1:] = torch.cumsum(0.5 * coef * (c[:-1] + c[1:]), 0)
    lo, hi = _window(case)
    pick = [l for l in range(L) if lo <= l * DT <= hi]
    return kt, kt[pick].mean(0) if pick else torch.zeros_like(kt[0])


def exact(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    if kind == "shc":
        v, W = (x.double() for x in data[1])
        N, K, nc = case["N"], case["K"], case["nc"]
        l = torch.arange(nc, device=DEV, dtype=torch.float64)
        cnt = K - l
        trap = torch.ones(nc, device=DEV, dtype=torch.float64)
        trap[0] = 0.5
        trap[-1] = 0.5
        f = torch.from_numpy(np.linspace(0.0, 60.0, case["n_freq"])).to(DEV)
        table = torch.cos(2.0 * math.pi * DT_SHC * l[:, None] * f[None, :])
        coef = WMK / (_volume(N, case) * T_K * FE[0])
        out = []
        for c in range(9):
            g = W[:, :, c] @ v[:, :, c % 3].T          # [tau][t]
            ks = torch.stack([torch.diagonal(g, q).sum() if q < K else g.new_zeros(()) for q in range(nc)])
            k = torch.where(cnt > 0, ks / cnt.clamp(min=1), 0.0)
            out.append(4.0 * coef * DT_SHC * ((trap * k) @ table))
        return {"kappa": torch.stack(out)}
    if kind == "group":
        got = [_hnema(case, len(m), _currents(case, m, E, f, *d[0])[0]) for m, E, f, d in data]
        return {"kappa": torch.cat([x[0].reshape(-1) for x in got]),
                "mean": torch.cat([x[1].reshape(-1) for x in got])}
    mass, E, f, blocks = data
    rows = ((3,) if case.get("direction") else ()) + (case["B"],)
    parts = [_currents(case, mass, E, f, v, W) for v, W in blocks]
    Jb, J = torch.cat([p[0] for p in parts]), torch.cat([p[1] for p in parts])
    if kind == "xcorr":
        B = case["B"]
        flat = Jb.reshape(Jb.shape[0], 3 * B)
        kw = _green_kubo(case, _correlate(flat, flat, case["L"]), Jb.shape[0])[1]
        return {"kappa_xcorr": kw.view(B, 3, B, 3).permute(0, 2, 1, 3).contiguous()}
    if case["read"] == "hnema":
        kappa, mean = _hnema(case, len(mass), Jb)
        return {"kappa": kappa.view(rows + (3,)), "mean": mean.view(rows + (3,))}
    R = Jb.shape[1]
    C = _correlate(Jb.reshape(Jb.shape[0], 3 * R), J, case["L"])
    kt, kw = _green_kubo(case, C, Jb.shape[0])
    out = {"Jb": Jb.view((Jb.shape[0],) + rows + (3,)), "kappa_w": kw.view(rows + (3, 3))}
    if case["read"] == "tau":
        out["kappa_tau"] = kt.permute(1, 2, 0).reshape(rows + (3, 3, case["L"])).contiguous()
    return out
