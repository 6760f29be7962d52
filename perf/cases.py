"""The work that users of the estimator have it do, as cases that can be timed and compared.

A case is a dict of plain values.  `prepare` makes what a user's program holds before the
call (device inputs, the plan, the ensemble or the network), `run` makes one pass through the
public entry points of `paper_2506_10526_gb300`, `work` counts what a pass cannot do without,
and `exact` restates the outputs in FP64 with plain torch and numpy.

Kinds:
  estimate   visibilities (gridded, or raw ones gridded first) -> folded MABS planes and the
             3D bispectrum of every closable ring triple, with the error bound when asked for
  reduce     accumulated collapse sums -> folded planes, 3D bispectrum and its three binnings
  mc         Monte Carlo: skies drawn on the GPU, a few runs of an ensemble, its statistics
  infer      bin features of a plan's grid and the surrogate's error bars for them
  train      normalisation, loss and gradient of a data set, and some training steps
"""
import math

import numpy as np
import torch

import paper_2506_10526_gb300 as bs

COARSE_FLAGS = (0, 1, 16, 30, 31)  # flagged channels of a 32-channel coarse band
PRECISIONS = {"fp32": bs.PREC_FP32, "bf16": bs.PREC_SPLIT_BF16, "fp16": bs.PREC_SPLIT_FP16}
WIDTH = 128  # hidden units of the surrogate


def listed():
    return [
        # one small field at the plainest settings: one image side, FP32, no flags; latency
        dict(name="tiny_fp32", kind="estimate", nt=64, nc=16, nb=8, spacing="linear", batch=1,
             precision="fp32", multires=False, flagged=False, symmetric=False, general=False,
             raw=0, bound=False),
        # the same field with coarse-band flags, split BF16 and error bounds: a production call
        dict(name="tiny_flagged_bf16", kind="estimate", nt=64, nc=16, nb=8, spacing="linear",
             batch=1, precision="bf16", multires=True, flagged=True, symmetric=False,
             general=False, raw=0, bound=True),
        # odd sizes: sides and channel counts that are no power of two, two realisations
        dict(name="odd_fp32", kind="estimate", nt=90, nc=27, nb=7, spacing="linear", batch=2,
             precision="fp32", multires=False, flagged=True, symmetric=False, general=False,
             raw=0, bound=False),
        # one 32-channel coarse band of the 256^2 MWA-like grid in plain FP32
        dict(name="mwa_coarse_band_fp32", kind="estimate", nt=256, nc=32, nb=20, spacing="log",
             batch=1, precision="fp32", multires=True, flagged=False, symmetric=False,
             general=False, raw=0, bound=False),
        # one 256-channel sub-band of the same grid in split BF16, channel symmetry: the
        # largest job, a whole channel cube
        dict(name="mwa_subband_bf16", kind="estimate", nt=256, nc=256, nb=20, spacing="log",
             batch=1, precision="bf16", multires=True, flagged=False, symmetric=True,
             general=False, raw=0, bound=False),
        # complex (non-Hermitian) visibilities in plain FP32, an odd channel count
        dict(name="general_fp32", kind="estimate", nt=100, nc=45, nb=9, spacing="log", batch=1,
             precision="fp32", multires=True, flagged=False, symmetric=False, general=True,
             raw=0, bound=False),
        # raw visibilities of 128 antennas: gridding, per-channel sampling, split FP16
        dict(name="raw_sampling_fp16", kind="estimate", nt=96, nc=64, nb=8, spacing="linear",
             batch=1, precision="fp16", multires=True, flagged=False, symmetric=False,
             general=False, raw=8128, bound=False),
        # what follows the accumulation over a whole 768-channel band, binnings included
        dict(name="reduce_band", kind="reduce", nt=64, nc=768, nb=12, spacing="log",
             flagged=True, n_k1=12, n_mu=5, n_t=5, lmax=4, n_cyl=20),
        # error bars of the flagged tiny configuration by Monte Carlo: many small realisations
        dict(name="mc_tiny", kind="mc", groups="64:16:8:linear:256:16:16:16", runs=2,
             flagged=True, precision="bf16"),
        # uneven shapes in one ensemble, the declared 32 x 16 x 64 channel blocks
        dict(name="mc_uneven", kind="mc",
             groups="128:64:16:log:4:32:16:64;256:64:12:log:2:32:16:64;64:72:20:log:4:32:16:64",
             runs=2, flagged=False, precision="bf16"),
        # error bars of every bin of a 60-channel band
        dict(name="surrogate_infer", kind="infer", nt=256, nc=60, nb=20, spacing="log",
             flagged=True),
        # training the surrogate on Monte Carlo variances
        dict(name="surrogate_train", kind="train", rows=122880, steps=24, batch=8192),
    ]


def draw(rng):
    """One more case: the kinds above, sizes spread over their ranges."""
    def spread(lo, hi, step=1):
        return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random() / step)) * step))

    kind = rng.choice(["estimate"] * 6 + ["reduce", "mc", "mc", "infer", "train"])
    while True:
        if kind == "estimate":
            variant = rng.choice(["plain", "plain", "flagged", "symmetric", "general", "raw"])
            c = dict(kind=kind, nt=spread(32, 256, 2), nc=spread(8, 160), nb=rng.randint(5, 20),
                     spacing=rng.choice(["linear", "log"]), batch=rng.choice([1, 1, 1, 2, 3]),
                     precision=rng.choice(["fp32", "bf16", "fp16"]),
                     multires=rng.random() < 0.75, flagged=variant == "flagged",
                     symmetric=variant == "symmetric", general=variant == "general",
                     raw=0, bound=variant in ("plain", "flagged") and rng.random() < 0.5)
            if c["symmetric"] and c["precision"] == "fp32":
                c["precision"] = "bf16"
            if c["precision"] != "fp32":  # several fields at once at these sizes: an ensemble
                c["batch"] = 1
                if c["general"]:
                    c.update(nb=rng.randint(4, 6), nc=spread(8, 24))
            if variant == "raw":
                c.update(raw=spread(2000, 8128), nt=spread(48, 96, 2), spacing="linear",
                         nb=rng.randint(5, 10), batch=1)
            w = work(c)
            rate = 1.5e13 if c["precision"] == "fp32" else 1e14
            if w["flops"] / rate > 0.5 or w["bytes"] > 1.5e9 or _field_bytes(c) > 8e9:
                continue
            return c
        if kind == "reduce":
            c = dict(kind=kind, nt=64, nc=spread(60, 768, 2), nb=rng.randint(6, 12),
                     spacing="log", flagged=rng.random() < 0.5, n_k1=rng.randint(6, 16),
                     n_mu=rng.randint(3, 8), n_t=rng.randint(3, 8), lmax=rng.choice([0, 2, 4]),
                     n_cyl=rng.randint(5, 24))
            return c
        if kind == "mc":
            groups = []
            for _ in range(rng.randint(1, 3)):
                nc = rng.choice([12, 16, 24, 32, 48, 60, 64, 72])
                nt = rng.choice([32, 48, 64, 96, 128])
                nb = rng.randint(6, 14)
                batch = max(1, min(64, int(spread(8, 64) * 16 * 64 // (nc * nt))))
                n1 = rng.choice([nc, max(8, nc // 2)])
                groups.append(f"{nt}:{nc}:{nb}:{rng.choice(['linear', 'log'])}:{batch}:{n1}:{n1}:{nc}")
            return dict(kind=kind, groups=";".join(groups), runs=rng.randint(1, 3),
                        flagged=rng.random() < 0.3, precision=rng.choice(["bf16", "bf16", "fp16"]))
        if kind == "infer":
            return dict(kind=kind, nt=rng.choice([64, 128, 256]), nc=spread(12, 60),
                        nb=rng.randint(6, 20), spacing="log", flagged=rng.random() < 0.7)
        return dict(kind=kind, rows=spread(10000, 122880), steps=rng.randint(8, 24),
                    batch=spread(1000, 8192))


# ---------------------------------------------------------------------------- geometry


def _edges(c):
    nt = c["nt"]
    if c["spacing"] == "linear":
        return np.linspace(0.0, nt / 2.0, c["nb"] + 1)
    return np.geomspace(4.41 * max(nt, 128) / 256.0, nt / 2.0, c["nb"] + 1)


def _flags(c):
    f = np.zeros(c["nc"], np.uint8)
    if c.get("flagged"):
        for k in range(c["nc"]):
            f[k] = k % 32 in COARSE_FLAGS
    return f


def _rings(c):
    """Ring label of every cell (-1: none) and each ring's largest component."""
    nt, h = c["nt"], c["nt"] // 2
    u = np.arange(nt) - h
    q = (u[:, None] ** 2 + u[None, :] ** 2).astype(np.float64)
    e2 = _edges(c) ** 2
    lab = np.searchsorted(e2, q, side="right") - 1
    lab[(lab >= c["nb"]) | (q == 0)] = -1
    lab[0, :] = lab[:, 0] = -1
    big = np.maximum(np.abs(u)[:, None], np.abs(u)[None, :])
    cmax = [int(big[lab == m].max()) if (lab == m).any() else -1 for m in range(c["nb"])]
    return lab, cmax


def _triples(nb):
    return [(i, j, l) for i in range(nb) for j in range(i, nb) for l in range(j, nb)]


def _side(need):
    b = 8
    while True:
        if b > need:
            return b
        if b * 3 // 2 > need:
            return b * 3 // 2
        b *= 2


def _closing(c):
    """Ring triples whose annuli can form a triangle, with the smallest alias-free image side."""
    lab, cmax = _rings(c)
    nt, h = c["nt"], c["nt"] // 2
    u = np.arange(nt) - h
    r = np.sqrt((u[:, None] ** 2 + u[None, :] ** 2).astype(np.float64))
    lo = [r[lab == m].min() if cmax[m] >= 0 else 0.0 for m in range(c["nb"])]
    hi = [r[lab == m].max() if cmax[m] >= 0 else 0.0 for m in range(c["nb"])]
    got = []
    for t, (i, j, l) in enumerate(_triples(c["nb"])):
        if min(cmax[i], cmax[j], cmax[l]) < 0 or lo[l] > hi[i] + hi[j] + 1e-9:
            continue
        need = max(cmax[i] + cmax[j] + cmax[l], 2 * max(cmax[i], cmax[j], cmax[l]))
        got.append((t, (i, j, l), _side(need)))
    return got


def _groups(c):
    out = []
    for g in c["groups"].split(";"):
        nt, nc, nb, spacing, batch, n1, n2, n3 = g.split(":")
        out.append(dict(nt=int(nt), nc=int(nc), nb=int(nb), spacing=spacing, batch=int(batch),
                        block=(0, int(n1), 0, int(n2), 0, int(n3)), flagged=c["flagged"],
                        symmetric=n1 == n2 == n3 and int(n1) >= 64))
    return out


def _field_bytes(c):
    """Image-plane fields of the largest side (FP32), an upper limit of a plan's own."""
    _, cmax = _rings(c)
    return 2.0 * c["batch"] * (4 if c["general"] else 1) * c["nb"] * c["nc"] * _side(3 * max(cmax)) ** 2 * 4


# ---------------------------------------------------------------------------- work


def _contract_flops(c, n1, n2, n3, symmetric):
    total = 0.0
    for _, (i, j, l), M in _closing(c):
        triples = float(n1) * n2 * n3
        if symmetric and (i == j or j == l):
            triples = 0.5 * n1 * n1 * (n1 + 1)
        total += 2.0 * M * M * triples
    return total


def work(case):
    c = case
    if c["kind"] == "estimate":
        ncl, nc = len(_closing(c)), c["nc"]
        comp = 2 if c["general"] else 1
        planes = c["batch"] * ncl * ((2 * nc - 1) ** 2 + nc * nc) * 8.0 * comp
        if c["bound"]:
            planes += c["batch"] * ncl * (2 * nc - 1) ** 2 * 8.0
        vis = c["batch"] * nc * c["nt"] ** 2 * 8.0
        if c["raw"]:
            vis = c["raw"] * (16.0 + nc * 9.0) + nc * c["nt"] ** 2 * 12.0
        real = 4.0 if c["general"] else 2.0 if c["raw"] else 1.0
        flops = real * c["batch"] * _contract_flops(c, nc, nc, nc, c["symmetric"])
        return {"bytes": vis + planes, "flops": flops}
    if c["kind"] == "reduce":
        ncl, n2, nc = len(_closing(c)), 2 * c["nc"] - 1, c["nc"]
        return {"bytes": ncl * 8.0 * (2.0 * n2 * n2 + nc * nc),
                "flops": ncl * (10.0 * nc * nc * math.log2(nc) + nc * nc * (2.0 + c["lmax"] + 1))}
    if c["kind"] == "mc":
        nbytes = flops = 0.0
        for g in _groups(c):
            nbytes += 2.0 * 8.0 * len(_triples(g["nb"])) * g["nc"] ** 2
            n = c["runs"] * g["batch"]
            cells = float(g["nc"]) * g["nt"] ** 2
            flops += n * (_contract_flops(g, g["block"][1], g["block"][3], g["block"][5], g["symmetric"])
                          + 15.0 * cells * math.log2(cells))
        return {"bytes": nbytes, "flops": flops}
    d = bs.MLP_FEATURES
    macs = d * WIDTH + WIDTH * WIDTH + WIDTH
    if c["kind"] == "infer":
        rows = len(_triples(c["nb"])) * c["nc"] ** 2
        live = len(_closing(c)) * c["nc"] ** 2
        return {"bytes": rows * (4.0 * d + 4.0), "flops": 2.0 * macs * live}
    rows = c["rows"] + c["steps"] * c["batch"]
    return {"bytes": (rows + c["rows"]) * 4.0 * (d + 1), "flops": 6.0 * macs * rows}


# ---------------------------------------------------------------------------- inputs


def _gen(seed, salt=0):
    return torch.Generator(device="cuda").manual_seed(1000003 * salt + int(seed))


def _sky(nt, nc, gen):
    """Visibilities of a weakly non-Gaussian sky with P(k) ~ k^-2, centred, complex128."""
    w = torch.randn((nc, nt, nt), device="cuda", generator=gen, dtype=torch.float64)
    g = torch.fft.ifftn(torch.fft.fftn(w) * _root_power(nt, nc)).real
    d = g + 0.5 * (g * g - 0.25)
    return torch.fft.fftshift(torch.fft.fft2(d), dim=(1, 2))


def _root_power(nt, nc):
    kz = 2 * math.pi * torch.fft.fftfreq(nc, device="cuda", dtype=torch.float64)
    kx = 2 * math.pi * torch.fft.fftfreq(nt, device="cuda", dtype=torch.float64)
    k2 = kz[:, None, None] ** 2 + kx[None, :, None] ** 2 + kx[None, None, :] ** 2
    p = torch.where(k2 > 0, 1.0 / torch.where(k2 > 0, k2, 1.0), 0.0)
    return torch.sqrt(p * (0.25 * p.numel() / p.sum()))


def _visibilities(c, seed):
    gen = _gen(seed, 1)
    out = torch.empty((c["batch"], c["nc"], c["nt"], c["nt"]), dtype=torch.complex64, device="cuda")
    for b in range(c["batch"]):
        v = _sky(c["nt"], c["nc"], gen)
        if c["general"]:
            v = v + 1j * _sky(c["nt"], c["nc"], gen)
        else:  # exactly Hermitian: V(-U) = conj V(U)
            m = v[:, 1:, 1:]
            m.copy_(0.5 * (m + m.flip((1, 2)).conj()))
        out[b] = v.to(torch.complex64)
    return out


def _raw(c, seed):
    """Baselines over the whole uv plane, and their visibilities: a smooth sky plus noise."""
    gen = _gen(seed, 2)
    nt, nbl, nc = c["nt"], c["raw"], c["nc"]
    uv = (torch.rand((nbl, 2), device="cuda", generator=gen, dtype=torch.float64) - 0.5) * (nt - 2)
    amp = 20.0 / (1.0 + 0.05 * (uv ** 2).sum(1, keepdim=True).sqrt())
    s = torch.complex(torch.randn((nbl, nc), device="cuda", generator=gen),
                      torch.randn((nbl, nc), device="cuda", generator=gen))
    vis = ((3.0 + s) * amp).to(torch.complex64)
    flags = (torch.rand((nbl, nc), device="cuda", generator=gen) < 0.15).to(torch.uint8)
    return uv, vis, flags


def _sampling(valid):
    """Unfolded number of channel triples at every (nu1 - nu3, nu2 - nu3)."""
    nc = len(valid)
    v = torch.from_numpy(np.asarray(valid, np.int64)).cuda()
    out = torch.zeros((2 * nc - 1, 2 * nc - 1), dtype=torch.int64, device="cuda")
    pair = v[:, None] * v[None, :]
    for n3 in range(nc):
        if valid[n3]:
            o = nc - 1 - n3
            out[o:o + nc, o:o + nc] += pair
    return out


def _sums(c, seed):
    """Collapse sums of a band: T A M^2 x (signal + noise) summed over the sampled triples."""
    n2 = 2 * c["nc"] - 1
    nnu = _sampling(1 - _flags(c))
    gen = _gen(seed, 3)
    sums = torch.zeros((1, len(_triples(c["nb"])), n2, n2), dtype=torch.float64, device="cuda")
    root = nnu.double().sqrt()
    d = (torch.arange(n2, device="cuda") - (c["nc"] - 1)).double()
    shape = 40.0 * torch.exp(-(d[:, None] ** 2 + d[None, :] ** 2 - d[:, None] * d[None, :]) / 800.0)
    for t, _, M in _closing(c):
        noise = torch.randn((n2, n2), device="cuda", generator=gen, dtype=torch.float32)
        sums[0, t] = (root * noise + nnu * shape) * float(M * M)
    return sums, nnu


def _binning(c, plan):
    kperp = 2 * np.pi * plan.ring_umean()
    kpar = (np.arange(c["nc"]) - c["nc"] // 2) * (2 * np.pi / c["nc"]) * 20.0
    kmax = float(np.sqrt(kperp.max() ** 2 + 4 * np.abs(kpar).max() ** 2))
    k1 = np.geomspace(0.9 * kperp.min(), 1.01 * kmax, c["n_k1"] + 1)
    return kperp, kpar, k1, _cyl_edges(c, kpar)


def _cyl_edges(c, kpar):
    return np.linspace(-0.9 * np.abs(kpar).max(), 0.9 * np.abs(kpar).max(), c["n_cyl"] + 1)


def _network(seed):
    """Parameters of a trained-looking network: [W1 | b1 | W2 | b2 | w3 | b3] and the
    normalisation [mu_x | sd_x | mu_y, sd_y]."""
    r = np.random.default_rng(int(seed) + 77)
    d, w = bs.MLP_FEATURES, WIDTH
    p = [r.normal(0, 1.0 / math.sqrt(d), w * d), r.normal(0, 0.1, w), r.normal(0, 1.2 / math.sqrt(w), w * w),
         r.normal(0, 0.1, w), r.normal(0, 1.0 / math.sqrt(w), w), r.normal(0, 0.1, 1)]
    norm = [r.uniform(-0.5, 1.5, d), r.uniform(0.8, 2.0, d), [-3.0], [2.5]]
    return np.concatenate(p + norm).astype(np.float32)


def _training_set(c, seed):
    gen = _gen(seed, 4)
    n, d = c["rows"], bs.MLP_FEATURES
    mix = torch.randn((d, d), device="cuda", generator=gen) / math.sqrt(d)
    x = torch.randn((n, d), device="cuda", generator=gen) @ mix + 0.5
    t = x[:, 0] - 0.5 * x[:, 1] * x[:, 2] + torch.sin(x[:, 3])
    t = t + 0.1 * torch.randn(n, device="cuda", generator=gen) - 3.0
    return x.contiguous(), t.contiguous()


# ---------------------------------------------------------------------------- prepare and run


def prepare(case, seed):
    c = case
    s = {"case": c, "seed": int(seed)}
    if c["kind"] == "estimate":
        s["plan"] = bs.Plan(c["nt"], c["nc"], _edges(c), precision=PRECISIONS[c["precision"]],
                            batch=c["batch"], multires=c["multires"], general=c["general"],
                            chan_sampling=bool(c["raw"]))
        s["flags"] = _flags(c) if c["flagged"] else None
        s["input"] = _raw(c, seed) if c["raw"] else _visibilities(c, seed)
    elif c["kind"] == "reduce":
        plan = bs.Plan(c["nt"], c["nc"], _edges(c), multires=True)
        vis = torch.zeros((1, c["nc"], c["nt"], c["nt"]), dtype=torch.complex64, device="cuda")
        plan.grid_load(vis, chan_flags=_flags(c))
        sums, nnu = _sums(c, seed)
        plan.delta_import(sums, nnu.cpu().numpy())
        torch.cuda.synchronize()  # the sums were copied into the plan
        del sums
        s["plan"], s["bins"] = plan, _binning(c, plan)
    elif c["kind"] == "mc":
        gs = _groups(c)
        s["groups"] = gs
        s["mc"] = bs.Ensemble([dict(nt=g["nt"], nchan=g["nc"], edges=list(_edges(g)), batch=g["batch"],
                                    multires=True, precision=PRECISIONS[c["precision"]]) for g in gs])
        s["sky"], s["buf"] = [], []
        for k, g in enumerate(gs):
            s["sky"].append(bs.SkyGenerator(g["nt"], g["nc"], max_batch=g["batch"]))
            s["buf"].append(torch.empty((g["batch"], g["nc"], g["nt"], g["nt"]), dtype=torch.complex64,
                                        device="cuda"))
            s["mc"].set_input(k, s["buf"][k])
            s["mc"].set_block(k, g["block"])
            if c["flagged"]:
                s["mc"].set_flags(k, _flags(g))
    elif c["kind"] == "infer":
        s["plan"] = bs.Plan(c["nt"], c["nc"], _edges(c), multires=True, torch_workspace=True)
        s["net"] = bs.Surrogate(width=WIDTH)
        s["net"].set_params(_network(seed))
        s["flags"] = _flags(c)
    else:
        s["net"] = bs.Surrogate(width=WIDTH)
        s["start"] = _network(seed)
        s["x"], s["t"] = _training_set(c, seed)
    return s


def _planes(plan, c):
    vt = torch.complex128 if c["general"] else torch.float64
    n2, ncl = 2 * c["nc"] - 1, plan.n_closable
    delta = torch.empty((plan.batch, ncl, n2, n2), dtype=vt, device="cuda")
    b3d = torch.empty((plan.batch, ncl, c["nc"], c["nc"]), dtype=vt, device="cuda")
    plan.mabs_delta_closable(delta)
    plan.bs3d_closable(b3d)
    return delta, b3d


def run(state):
    s, c = state, state["case"]
    if c["kind"] == "estimate":
        plan, out = s["plan"], {}
        if c["raw"]:
            uv, vis, flags = s["input"]
            grid, ng = plan.grid_visibilities(uv, vis, flags, mode=1)
            plan.grid_load(grid, ngrid=ng)
            out["grid"], out["ng"] = grid, ng
        else:
            plan.grid_load(s["input"], chan_flags=s["flags"])
        plan.mabs(symmetric=c["symmetric"])
        out["delta"], out["b3d"] = _planes(plan, c)
        if c["bound"]:
            out["bound"], out["relerr"] = plan.error_bound(out["delta"], closable=True)
        return out
    if c["kind"] == "reduce":
        plan, (kperp, kpar, k1, ke) = s["plan"], s["bins"]
        delta, b3d = _planes(plan, dict(c, general=False))
        mono, mono_n = plan.bs_monopole(b3d, kperp, kpar, k1, c["n_mu"], c["n_t"])
        multi, multi_n = plan.bs_multipoles(b3d, kperp, kpar, k1, c["n_mu"], c["n_t"], lmax=c["lmax"])
        cyl, cyl_n = plan.bs_cylindrical(b3d, kpar, ke)
        return {"delta": delta, "b3d": b3d, "mono": mono, "mono_n": mono_n, "multi": multi,
                "multi_n": multi_n, "cyl": cyl, "cyl_n": cyl_n}
    if c["kind"] == "mc":
        s["mc"].reset()
        for i in range(c["runs"]):
            for g, sky, buf in zip(s["groups"], s["sky"], s["buf"]):
                sky.generate(s["seed"], i * g["batch"], out=buf)
            s["mc"].run()
        return [list(s["mc"].stats(k, 1)) for k in range(len(s["groups"]))]
    if c["kind"] == "infer":
        feat = s["plan"].mlp_features(s["flags"])
        return {"features": feat, "log_var": s["net"].forward(feat)}
    net = s["net"]
    net.set_params(s["start"])
    net.fit_norm(s["x"], s["t"])
    loss, grad = net.grad(s["x"], s["t"])
    last = net.train(s["x"], s["t"], c["steps"], batch=c["batch"])
    p = net.params()
    return {"loss": loss, "grad": grad, "last_loss": last, "weights": p[:net.n_weights],
            "norm": p[net.n_weights:]}


# ---------------------------------------------------------------------------- FP64


def _fields(v, lab, m, M):
    """Image-plane fields [nc, M * M] of ring m at side M (complex128)."""
    nc, nt = v.shape[0], v.shape[1]
    grid = torch.zeros((nc, M, M), dtype=torch.complex128, device="cuda")
    iv, iu = torch.nonzero(lab == m, as_tuple=True)
    grid[:, (iv - nt // 2) % M, (iu - nt // 2) % M] = v[:, iv, iu]
    return torch.fft.ifft2(grid, norm="forward").reshape(nc, M * M)


def _collapse(c, v, blk, valid):
    """Sums over closed triangles collapsed to (nu1 - nu3, nu2 - nu3), and the number of closed
    triangles, per ring triple; v [nc, nt, nt] complex128."""
    nc, n2 = c["nc"], 2 * c["nc"] - 1
    lab = torch.from_numpy(_rings(c)[0]).cuda()
    unit = torch.ones((1, c["nt"], c["nt"]), dtype=torch.complex128, device="cuda")
    v = v * torch.from_numpy(np.asarray(valid, np.float64)).cuda()[:, None, None]
    n1, nn2, n3 = (torch.arange(blk[2 * k], blk[2 * k + 1], device="cuda") for k in range(3))
    at = ((n1[:, None, None] - n3 + nc - 1) * n2 + (nn2[None, :, None] - n3 + nc - 1)).reshape(-1)
    by_side = {}
    for t, ijl, _ in _closing(c):
        cm = sum(_rings_cmax(c)[m] for m in ijl)
        by_side.setdefault(_side(cm), []).append((t, ijl))
    sums, counts = {}, {}
    for M, todo in sorted(by_side.items()):
        F, I, pair = {}, {}, None
        for t, (i, j, l) in todo:
            for m in (i, j, l):
                if m not in F:
                    F[m] = _fields(v, lab, m, M)
                    I[m] = _fields(unit, lab, m, M).real
                    if _is_real(c):
                        F[m] = F[m].real.contiguous()
            T = int(round(float((I[i] * I[j] * I[l]).sum()) / (M * M)))
            if T <= 0:
                continue
            if pair != (i, j):
                pair = (i, j)
                P = (F[i][n1][:, None, :] * F[j][nn2][None, :, :]).reshape(-1, M * M)
            S = (P @ F[l][n3].T) / (M * M)
            plane = torch.zeros(n2 * n2, dtype=S.dtype, device="cuda")
            plane.index_add_(0, at, S.reshape(-1))
            sums[t], counts[t] = plane.view(n2, n2), T
        del F, I
        P = None
    return sums, counts


_CMAX = {}


def _rings_cmax(c):
    key = (c["nt"], c["nb"], c["spacing"])
    if key not in _CMAX:
        _CMAX[key] = _rings(c)[1]
    return _CMAX[key]


def _is_real(c):
    return not c.get("general")


def _block_sampling(c, blk, valid):
    nc = c["nc"]
    v = np.asarray(valid, np.int64)
    b = [torch.zeros(nc, dtype=torch.int64, device="cuda") for _ in range(3)]
    for k in range(3):
        b[k][blk[2 * k]:blk[2 * k + 1]] = torch.from_numpy(v[blk[2 * k]:blk[2 * k + 1]]).cuda()
    out = torch.zeros((2 * nc - 1, 2 * nc - 1), dtype=torch.int64, device="cuda")
    pair = b[0][:, None] * b[1][None, :]
    for n3 in range(nc):
        o = nc - 1 - n3
        out[o:o + nc, o:o + nc] += pair * b[2][n3]
    return out


def _fold(p):
    q = p + p.flip((-2, -1))
    mid = (p.shape[-1] - 1) // 2
    q[..., mid, mid] = p[..., mid, mid]
    return q


def _delay(planes, nc):
    """Eq. (dft), the real part of the sum over -nc/2 <= n, m < nc/2."""
    h = nc // 2
    n = torch.arange(-h, nc - h, device="cuda")
    sub = planes[..., (n + nc - 1)[:, None], (n + nc - 1)[None, :]]
    sub = torch.where(torch.isnan(sub), torch.zeros_like(sub), sub)
    a = torch.arange(-h, -h + nc, device="cuda")
    ang = -2 * math.pi * ((a[:, None] * n[None, :]) % nc).double() / nc
    ker = torch.complex(torch.cos(ang), torch.sin(ang))

    def one(x):
        return (ker @ x.to(torch.complex128) @ ker.T).real

    if sub.is_complex():
        return torch.complex(one(sub.real), one(sub.imag))
    return one(sub)


def _estimates(c, v, blk, valid, occupancy=None):
    """Folded planes and 3D bispectrum of the closable ring triples."""
    sums, T = _collapse(c, v, blk, valid)
    nnu = _fold(_block_sampling(c, blk, valid))
    den = _collapse(c, occupancy, blk, valid)[0] if occupancy is not None else None
    planes = []
    for t in sorted(sums):
        d = _fold(den[t]) if den is not None else (nnu * T[t]).double()
        x = _fold(sums[t]) / torch.where(nnu > 0, d, torch.ones_like(d))
        x[nnu == 0] = complex(math.nan, math.nan) if x.is_complex() else math.nan
        planes.append(x)
    delta = torch.stack(planes)
    return sorted(sums), delta, _delay(delta, c["nc"])


def _philox_normals(n, seed, realisation):
    """Unit normals of cells 0 .. n - 1: Philox4x32-10 and Box-Muller, four to a call."""
    mask = 0xFFFFFFFF
    q = torch.arange((n + 3) // 4, device="cuda", dtype=torch.int64)
    r = torch.full_like(q, int(realisation))
    w = [q & mask, q >> 32, r & mask, r >> 32]
    k0, k1 = seed & mask, (seed >> 32) & mask

    def mul(m, x):  # 32 x 32 -> (hi, lo), by halves so that int64 does not overflow
        xl, xh = x & 0xFFFF, x >> 16
        low, high = m * xl, m * xh
        s = (low >> 16) + (high & 0xFFFF)
        return (high >> 16) + (s >> 16), ((s & 0xFFFF) << 16) | (low & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, w[0])
        h1, l1 = mul(0xCD9E8D57, w[2])
        w = [h1 ^ w[1] ^ k0, l1, h0 ^ w[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    u = [(x.double() + 0.5) * 2.0 ** -32 for x in w]
    ra, rb = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
    z = torch.stack([ra * torch.cos(2 * math.pi * u[1]), ra * torch.sin(2 * math.pi * u[1]),
                     rb * torch.cos(2 * math.pi * u[3]), rb * torch.sin(2 * math.pi * u[3])], 1)
    return z.reshape(-1)[:n]


def _mc_exact(c, seed):
    out = []
    for g in _groups(c):
        nt, nc = g["nt"], g["nc"]
        valid, all_b = 1 - _flags(g), []
        for r in range(c["runs"] * g["batch"]):
            w = _philox_normals(nc * nt * nt, int(seed), r).view(nc, nt, nt)
            f = torch.fft.ifftn(torch.fft.fftn(w) * _root_power(nt, nc)).real
            v = torch.fft.fftshift(torch.fft.fft2(f + 0.5 * (f * f - 0.25)), dim=(1, 2))
            clos, _, b3d = _estimates(g, v, g["block"], valid)
            all_b.append(b3d)
        b = torch.stack(all_b)
        full = torch.full((2, len(_triples(g["nb"])), nc, nc), math.nan, dtype=torch.float64)
        at = torch.tensor(clos)
        full[0, at] = b.mean(0).cpu()
        if b.shape[0] > 1:
            full[1, at] = b.var(0).cpu()
        # a ring triple without closed triangles has estimate 0 in every realisation
        rest = torch.ones(full.shape[1], dtype=torch.bool)
        rest[at] = False
        full[0, rest] = 0.0
        full[1, rest] = 0.0 if b.shape[0] > 1 else math.nan
        out.append([full[0].numpy(), full[1].numpy(), None])
    return out


def _features(c):
    """The 45 features of every (ring triple, a, b); NaN rows where no triangle closes."""
    nc, nb = c["nc"], c["nb"]
    lab, _ = _rings(c)
    u = np.arange(c["nt"]) - c["nt"] // 2
    r = np.sqrt((u[:, None] ** 2 + u[None, :] ** 2).astype(np.float64))
    e = _edges(c)
    kperp = 2 * np.pi * np.array([r[lab == m].mean() if (lab == m).any() else 0.5 * (e[m] + e[m + 1])
                                  for m in range(nb)])
    flags = _flags(c)
    pos = np.arange(nc) % 32
    per = [flags[pos == q].mean() if (pos == q).any() else 0.0 for q in range(32)]
    nnu = _fold(_sampling(1 - flags))
    h = nc // 2
    sq = nnu[nc - 1 - h:2 * nc - 1 - h, nc - 1 - h:2 * nc - 1 - h]
    live = sq[sq > 0].double()
    tail = [float(torch.log((1 / live).sum())), len(live) / float(nc * nc), float(torch.log(live.sum() / len(live)))]
    out = torch.full((len(_triples(nb)), nc, nc, bs.MLP_FEATURES), math.nan, dtype=torch.float64, device="cuda")
    k = (torch.arange(nc, device="cuda") - h).double() * (2 * math.pi / nc)
    ka, kb = k[:, None].expand(nc, nc), k[None, :].expand(nc, nc)
    lab = torch.from_numpy(lab).cuda()
    unit = torch.ones((1, c["nt"], c["nt"]), dtype=torch.complex128, device="cuda")
    masks = {}
    for t, (i, j, l), M in _closing(c):
        for m in (i, j, l):
            if (m, M) not in masks:
                masks[m, M] = _fields(unit, lab, m, M).real
        T = int(round(float((masks[i, M] * masks[j, M] * masks[l, M]).sum()) / (M * M)))
        if T <= 0:
            continue
        ks = torch.stack([torch.sqrt(kperp[i] ** 2 + ka ** 2), torch.sqrt(kperp[j] ** 2 + kb ** 2),
                          torch.sqrt(kperp[l] ** 2 + (ka + kb) ** 2)]).sort(0, descending=True)[0]
        row = [torch.log(ks[0]), ks[1] / ks[0],
               (ks[0] ** 2 + ks[1] ** 2 - ks[2] ** 2) / (2 * ks[0] * ks[1]), flags.mean(), math.log(T),
               ka.abs(), kb.abs(), math.log(kperp[i]), math.log(kperp[j]), math.log(kperp[l])]
        for q, x in enumerate(row + per + tail):
            out[t, :, :, q] = x
    return out.reshape(-1, bs.MLP_FEATURES)


def _split(p):
    d, w = bs.MLP_FEATURES, WIDTH
    p = torch.from_numpy(p).cuda()
    parts = torch.split(p, [w * d, w, w * w, w, w, 1, d, d, 1, 1])
    W1, W2, w3 = (parts[k].to(torch.bfloat16).double() for k in (0, 2, 4))
    return [W1.view(w, d), parts[1].double(), W2.view(w, w), parts[3].double(), w3, parts[5].double(),
            parts[6].double(), parts[7].double(), parts[8].double(), parts[9].double()]


def exact(case, seed):
    c = case
    if c["kind"] == "estimate":
        real = 8.0 if c["general"] else 2.0 if c["raw"] else 1.0
        if real * c["batch"] * _contract_flops(c, c["nc"], c["nc"], c["nc"], False) > 4e12:
            return None
        blk, valid = (0, c["nc"]) * 3, 1 - _flags(c)
        out, delta, b3d = {}, [], []
        if c["raw"]:
            uv, vis, flags = _raw(c, seed)
            nt, h = c["nt"], c["nt"] // 2
            cell = torch.floor(uv + 0.5).to(torch.int64)
            ok = (cell.abs() < h).all(1)
            w = (flags == 0).double() * ok[:, None]
            x = vis.to(torch.complex128) * w
            grid = torch.zeros((nt * nt, c["nc"]), dtype=torch.complex128, device="cuda")
            n = torch.zeros((nt * nt, c["nc"]), dtype=torch.float64, device="cuda")
            for sign in (1, -1):
                at = torch.where(ok, (sign * cell[:, 1] + h) * nt + sign * cell[:, 0] + h, 0)
                grid.index_add_(0, at, x if sign > 0 else x.conj())
                n.index_add_(0, at, w)
            grid = torch.where(n > 0, grid / n.clamp(min=1.0), torch.zeros_like(grid))
            grid, n = grid.T.reshape(c["nc"], nt, nt), (n > 0).double().T.reshape(c["nc"], nt, nt)
            out["grid"], out["ng"] = grid, n
            _, d, b = _estimates(c, grid * n, blk, valid, n.to(torch.complex128))
            delta, b3d = [d], [b]
        else:
            vis = _visibilities(c, seed)
            for k in range(c["batch"]):
                _, d, b = _estimates(c, vis[k].to(torch.complex128), blk, valid)
                delta.append(d)
                b3d.append(b)
        out["delta"], out["b3d"] = torch.stack(delta), torch.stack(b3d)
        if c["bound"]:
            out["bound"] = out["relerr"] = None
        return out
    if c["kind"] == "reduce":
        sums, nnu = _sums(c, seed)
        folded = _fold(nnu)
        unit = torch.ones((1, c["nt"], c["nt"]), dtype=torch.complex128, device="cuda")
        lab = torch.from_numpy(_rings(c)[0]).cuda()
        planes = []
        for t, (i, j, l), M in _closing(c):
            I = [_fields(unit, lab, m, M).real for m in (i, j, l)]
            T = int(round(float((I[0] * I[1] * I[2]).sum()) / (M * M)))
            if T > 0:
                x = _fold(sums[0, t]) / (folded * (float(T) * M * M))
                x[folded == 0] = math.nan
                planes.append(x)
        del sums
        delta = torch.stack(planes)
        b3d = torch.stack([_delay(x, c["nc"]) for x in delta])
        kpar = (np.arange(c["nc"]) - c["nc"] // 2) * (2 * np.pi / c["nc"]) * 20.0
        ke, n = _cyl_edges(c, kpar), c["n_cyl"]
        q = np.searchsorted(ke, kpar, side="right") - 1
        one = torch.zeros((n, c["nc"]), dtype=torch.float64, device="cuda")
        for a, b in enumerate(q):
            if 0 <= b < n:
                one[b, a] = 1.0
        return {"delta": delta[None], "b3d": b3d[None], "mono": None, "mono_n": None, "multi": None,
                "multi_n": None, "cyl": (one @ b3d @ one.T)[None], "cyl_n": None}
    if c["kind"] == "mc":
        flops = sum(c["runs"] * g["batch"] * _contract_flops(g, g["block"][1], g["block"][3], g["block"][5], False)
                    for g in _groups(c))
        n = sum(c["runs"] * g["batch"] * (1 + len(_closing(g)) / 60.0) for g in _groups(c))
        return _mc_exact(c, seed) if flops < 6e12 and n < 1600 else None
    if c["kind"] == "infer":
        x = _features(c)
        W1, b1, W2, b2, w3, b3, mu, sd, my, sy = _split(_network(seed))
        y = torch.cat([torch.tanh(torch.tanh(((r - mu) / sd) @ W1.T + b1) @ W2.T + b2) @ w3
                       for r in x.split(1 << 18)]) + b3
        return {"features": x, "log_var": y * sy + my}
    x, t = _training_set(c, seed)
    x, t = x.double(), t.double()
    W1, b1, W2, b2, w3, b3 = _split(_network(seed))[:6]
    norm = [x.mean(0), x.std(0, unbiased=False), t.mean()[None], t.std(unbiased=False)[None]]
    xn, tn = (x - norm[0]) / norm[1], (t - norm[2]) / norm[3]
    h1 = torch.tanh(xn @ W1.T + b1)
    h2 = torch.tanh(h1 @ W2.T + b2)
    res = h2 @ w3 + b3 - tn
    dy = 2 * res / len(res)
    z2 = dy[:, None] * w3 * (1 - h2 * h2)
    z1 = (z2 @ W2) * (1 - h1 * h1)
    grad = torch.cat([(z1.T @ xn).reshape(-1), z1.sum(0), (z2.T @ h1).reshape(-1), z2.sum(0), h2.T @ dy,
                      dy.sum()[None]])
    return {"loss": float((res * res).mean()), "grad": grad.cpu().numpy(), "last_loss": None,
            "weights": None, "norm": torch.cat(norm).cpu().numpy()}
