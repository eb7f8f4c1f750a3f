"""The work a GW program has this library do, as cases to time and to check.

A case is one call (or the two or three calls that go together) of paper_2509_23018_gb300, with
sizes from the repository's configurations, tests and benchmark, cut where one pass would take
seconds.  listed() holds one or two of each kind of work; draw() gives more from the same ranges.
"split" is the mode the benchmark runs: two-float pair transforms and the split-precision
contraction on the BF16 tensor cores with seven slices; "fp64" is native double precision.
"""
import math

import numpy as np
import torch

from paper_2509_23018_gb300 import chi0 as gw

SLICES = 7
WP = 16.6  # plasma energy of the plasmon-pole inputs (eV), silicon's

# ------------------------------------------------------------------ the cases


def _chi(name, prec, grid, nv, nc, ngpsi, ng, nw=1, chunk=8192):
    return {"name": name, "kind": "chi", "prec": prec, "n0": grid[0], "n1": grid[1], "n2": grid[2], "nv": nv,
            "nc": nc, "ngpsi": ngpsi, "ng": ng, "nw": nw, "chunk": chunk}


def listed():
    return [
        # one q-point of a small cell in double precision: the smallest call, bound by latency
        _chi("chi_fp64_24", "fp64", (24, 24, 24), 16, 64, 600, 200),
        # a small non-cubic cell, odd band counts, several frequencies, ragged chunks and sphere
        _chi("chi_split_ragged", "split", (30, 36, 40), 13, 147, 1501, 517, nw=3, chunk=777),
        # double precision at an ordinary size: one chunk of pairs of the 48^3 system
        _chi("chi_fp64_48", "fp64", (48, 48, 48), 8, 1024, 6000, 2000),
        # the q-point loop of the 48^3 system: the next q's valence bands and sphere, then chi(0)
        _chi("chi_split_48", "split", (48, 48, 48), 128, 1024, 6000, 2000),
        # a chunk of the largest system (72^3, N_G = 6000)
        _chi("chi_split_72", "split", (72, 72, 72), 4, 2048, 20000, 6000),
        # many q-points of uneven spheres times imaginary frequencies, as one captured graph
        {"name": "batch_40", "kind": "batch", "prec": "split", "n0": 40, "n1": 40, "n2": 40, "nv": 32, "nc": 256,
         "ngpsi": 8000, "ng": 3000, "ng_lo": 300, "nq": 6, "nw": 4, "chunk": 8192},
        # sensitivities: forward and backward through the autograd function
        {"name": "grad_40", "kind": "grad", "prec": "split", "n0": 40, "n1": 40, "n2": 40, "nv": 48, "nc": 384,
         "ngpsi": 4500, "ng": 1500, "nw": 1, "chunk": 8192},
        # forward-mode derivative of chi along a perturbation of the bands
        {"name": "jvp_40", "kind": "jvp", "prec": "split", "n0": 40, "n1": 40, "n2": 40, "nv": 24, "nc": 384,
         "ngpsi": 4500, "ng": 1500, "nw": 1, "chunk": 8192},
        # full frequency dependence in the static subspace: chi(0), then chi_BB' at the frequencies
        {"name": "subspace_48", "kind": "subspace", "prec": "split", "n0": 48, "n1": 48, "n2": 48, "nv": 32,
         "nc": 512, "ngpsi": 6000, "ng": 2000, "neig": 400, "nw": 8, "chunk": 8192},
        # absorption: the real axis with broadening
        {"name": "real_48", "kind": "real", "prec": "split", "n0": 48, "n1": 48, "n2": 48, "nv": 32, "nc": 512,
         "ngpsi": 6000, "ng": 2000, "nw": 2, "chunk": 8192},
        # off-diagonal self-energy on an energy grid
        {"name": "sigma_6000", "kind": "sigma", "prec": "split", "nb": 3, "nocc": 1, "nsig": 384, "ng": 6000,
         "nw": 8},
        # the inverse dielectric matrix at a few frequencies
        {"name": "epsilon_2000", "kind": "epsilon", "prec": "split", "ng": 2000, "nw": 2},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sphere_count(radius):
    return 4.0 / 3.0 * math.pi * radius ** 3


def draw(rng):
    most = max(max(w["bytes"], w["flops"] / 50) for w in map(work, listed()))
    while True:
        case = _draw(rng)
        w = work(case)
        if max(w["bytes"], w["flops"] / 50) <= most and _fp64_flops(case) <= 0.15e12:
            return case


def _draw(rng):
    kind = rng.choice(["chi", "chi", "chi", "batch", "grad", "jvp", "subspace", "real", "sigma", "epsilon"])
    if kind == "epsilon":
        return {"kind": kind, "prec": "split", "ng": _log(rng, 150, 2000), "nw": rng.randint(1, 3)}
    if kind == "sigma":
        nb = rng.randint(1, 4)
        return {"kind": kind, "prec": "split", "nb": nb, "nocc": rng.randint(0, nb), "nsig": _log(rng, 24, 400),
                "ng": _log(rng, 300, 6000), "nw": _log(rng, 1, 10)}
    prec = "fp64" if kind == "chi" and rng.random() < 0.34 else "split"
    # cubic grids of the configurations, and non-cubic ones of the same range
    if rng.random() < 0.7:
        n = rng.choice([24, 40, 48, 72])
        grid = (n, n, n)
    else:
        grid = tuple(rng.choice([24, 30, 32, 36, 40, 45, 48, 54, 60]) for _ in range(3))
    n = min(grid)
    rpsi = n * rng.uniform(0.18, 0.27)           # radius of the wavefunction sphere
    rchi = rpsi * rng.uniform(0.6, 0.8)          # and of the dielectric one: no aliasing, 2 rpsi + rchi < n
    ngpsi, ng = int(_sphere_count(rpsi)), int(_sphere_count(rchi))
    nv, nc = _log(rng, 4, 128), _log(rng, 24, 1024)
    nb = nv + nc
    if nb > ngpsi // 3:                          # fewer bands than plane waves
        nv, nc = max(2, nv * ngpsi // (3 * nb)), max(4, nc * ngpsi // (3 * nb))
    nw = 1 if rng.random() < 0.5 else rng.randint(2, 6)
    case = {"kind": kind, "prec": prec, "n0": grid[0], "n1": grid[1], "n2": grid[2], "nv": nv, "nc": nc,
            "ngpsi": ngpsi, "ng": ng, "nw": nw, "chunk": rng.choice([8192, 8192, 4096, 1000])}
    if kind == "batch":
        case.update(nq=rng.randint(2, 8), ng_lo=max(40, ng // 10), nw=rng.randint(1, 6))
    if kind == "subspace":
        case.update(neig=max(8, ng // rng.randint(4, 10)), nw=rng.randint(2, 10))
    if kind == "grad":
        case.update(nw=1)
    return case


# ------------------------------------------------------------------ what a pass cannot do without


def _pair_flops(case):
    """Pair products and forward transforms, half of a full FFT's work (the output is a small sphere)."""
    n = case["n0"] * case["n1"] * case["n2"]
    return case["nv"] * case["nc"] * (2.5 * n * math.log2(n) + 6.0 * n)


def _batch_ng(case):
    """Sphere sizes of the q-points, spread over [ng_lo, ng]."""
    nq = case["nq"]
    return [case["ng_lo"] + (case["ng"] - case["ng_lo"]) * k // max(1, nq - 1) for k in range(nq)]


def work(case):
    k, ng, nw = case["kind"], case["ng"], case["nw"]
    if k == "epsilon":
        return {"bytes": nw * 2 * 16.0 * ng * ng, "flops": nw * 8.0 * ng ** 3}
    if k == "sigma":
        nb, ns = case["nb"], case["nsig"]
        return {"bytes": 16.0 * (nb * ns * ng + 2 * ng * ng + nw * ns * ns),
                "flops": nb * nw * (8.0 * (ns * ng * ng + ng * ns * ns) + 20.0 * ng * ng)}
    P = case["nv"] * case["nc"]
    coeff = 16.0 * case["ngpsi"] * (case["nv"] + case["nc"])
    herm = 4.0 * P                               # flops of a Hermitian contraction per ng^2
    out = 16.0 * nw * ng * ng
    if k == "batch":
        ngs = _batch_ng(case)
        sq = float(sum(g * g for g in ngs))
        return {"bytes": 16.0 * case["ngpsi"] * (case["nq"] * case["nv"] + case["nc"]) + 16.0 * nw * sq,
                "flops": case["nq"] * _pair_flops(case) + nw * herm * sq}
    if k == "grad":  # forward, then Y = M W, the back-transforms and the products
        return {"bytes": 2 * coeff + 2 * out, "flops": 3 * _pair_flops(case) + herm * ng * ng + 8.0 * P * ng * ng}
    if k == "jvp":   # three pair-element sets, two sums of products of which one is not Hermitian
        return {"bytes": 2 * coeff + out, "flops": 3 * _pair_flops(case) + nw * 3 * herm * ng * ng}
    if k == "subspace":
        ne = case["neig"]
        return {"bytes": coeff + 16.0 * (ng * ng + ng * ne + nw * ne * ne),
                "flops": _pair_flops(case) + herm * ng * ng + 8.0 * P * ng * ne + nw * herm * ne * ne}
    if k == "real":  # Hermitian and anti-Hermitian part
        return {"bytes": coeff + out, "flops": _pair_flops(case) + nw * 2 * herm * ng * ng}
    return {"bytes": coeff + out, "flops": _pair_flops(case) + nw * herm * ng * ng}


def _fp64_flops(case):
    """The double-precision pipes are far slower than the others: bounds the drawn fp64 cases."""
    return work(case)["flops"] if case["prec"] == "fp64" else 0.0


def tolerance(case):
    """About four times the distance to exact() that these inputs show; single entries, of a matrix
    whose diagonal outweighs the rest, up to a hundred times that."""
    if case["prec"] == "fp64":
        rel = 1e-14
    else:
        rel = {"real": 1e-10, "sigma": 3e-10, "epsilon": 1e-10}.get(case["kind"], 4e-11)
    return {"rel": rel, "max": 100 * rel}


# ------------------------------------------------------------------ inputs


def gsphere(n, q=(0.0, 0.0, 0.0), head=True):
    """The first n plane waves by |q + G|^2 (ties in lexicographic order); head=False leaves G = 0 out."""
    r = int(math.ceil((3.0 * n / (4.0 * math.pi)) ** (1.0 / 3.0))) + 3
    ax = np.arange(-r, r + 1)
    g = np.stack(np.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    if not head:
        g = g[np.any(g != 0, axis=1)]
    k2 = ((g + np.asarray(q)) ** 2).sum(1)
    return np.ascontiguousarray(g[np.lexsort((g[:, 2], g[:, 1], g[:, 0], k2))[:n]].astype(np.int32))


def _normal(gen, *shape):
    re, im = (torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64) for _ in range(2))
    return torch.complex(re, im)


def _bands(gen, nb, ngpsi):
    """nb orthonormal random coefficient rows: a Cholesky factor of the overlaps, applied once."""
    a = _normal(gen, nb, ngpsi)
    low = torch.linalg.cholesky(a @ a.mH)
    return torch.linalg.solve_triangular(low, a, upper=False).contiguous()


def _uniform(gen, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)


def _hermitian(gen, n):
    a = _normal(gen, n, n)
    return (0.5 * (a + a.mH)).contiguous()


def _omegas(case):
    """One frequency is the static limit; more are spread over [0, 100) eV."""
    return [100.0 * (k / case["nw"]) ** 2 for k in range(case["nw"])]


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _system(case, seed):
    """Bands, energies and sphere of one q-point, and what else the case's calls take."""
    gen = _gen(seed)
    dev = "cuda"
    s = {"gpsi": torch.as_tensor(gsphere(case["ngpsi"]), device=dev)}
    b = _bands(gen, case["nv"] + case["nc"], case["ngpsi"])
    s["cv"], s["cc"] = b[:case["nv"]].contiguous(), b[case["nv"]:].contiguous()
    s["ev"], s["ec"] = _uniform(gen, case["nv"], -10.0, -1.0), _uniform(gen, case["nc"], 1.0, 30.0)
    s["gchi"] = torch.as_tensor(gsphere(case["ng"], head=False), device=dev)
    k = case["kind"]
    if k == "grad":
        s["W"] = _hermitian(gen, case["ng"])
    if k == "jvp":
        s["dcv"], s["dcc"] = (_normal(gen, *s[x].shape) / math.sqrt(2.0 * case["ngpsi"]) for x in ("cv", "cc"))
        s["dev"], s["dec"] = (torch.randn(s[x].shape, generator=gen, device=dev, dtype=torch.float64)
                              for x in ("ev", "ec"))
    if k == "subspace":
        a = _normal(gen, case["neig"], case["ng"])
        low = torch.linalg.cholesky(a @ a.mH)
        s["basis"] = torch.linalg.solve_triangular(low, a, upper=False).mH.resolve_conj().contiguous()
    if k == "batch":
        s["cvs"] = [_bands(gen, case["nv"], case["ngpsi"]) for _ in range(case["nq"])]
        s["evs"] = [_uniform(gen, case["nv"], -10.0, -1.0) for _ in range(case["nq"])]
        m = 4
        qs = [((i % m) / m, (i // m % m) / m, 0.25 * (i // (m * m))) for i in range(case["nq"])]
        s["gchis"] = [torch.as_tensor(gsphere(n, q=q, head=any(q)), device=dev) for n, q in zip(_batch_ng(case), qs)]
    return s


def _coulomb(gchi):
    return 4.0 * math.pi / (gchi.double() ** 2).sum(1)


def _pole_inputs(case, seed):
    """Plasmon-pole parameters: strengths that decay with |G - G'|, mode energies with a damping."""
    gen = _gen(seed)
    ng, nb = case["ng"], case["nb"]
    g = torch.as_tensor(gsphere(ng, head=False), device="cuda")
    gd = g.double()
    g2 = (gd * gd).sum(1)
    d2 = g2[:, None] + g2[None, :] - 2.0 * (gd @ gd.T)
    t, u = _uniform(gen, ng, 0.0, 2.0 * math.pi), _uniform(gen, ng, 0.0, 1.0)
    ph = torch.polar(torch.ones_like(t), t)
    strength = WP * WP * torch.exp(-d2 / 8.0)
    wt = WP * (1.0 + 0.5 * (u[:, None] + u[None, :]))
    occ, emp = _uniform(gen, case["nocc"], -10.0, -1.0), _uniform(gen, nb - case["nocc"], 1.0, 30.0)
    return {"M": _normal(gen, nb, case["nsig"], ng) / math.sqrt(2.0 * ng), "En": torch.cat([occ, emp]).tolist(),
            "omega2": strength * (ph[:, None] * ph.conj()[None, :]), "wt": torch.complex(wt, torch.full_like(wt, -0.25)),
            "v": _coulomb(g), "E": [-6.0 + 12.0 * (k + 0.5) / case["nw"] for k in range(case["nw"])]}


def _chi_inputs(case, seed):
    """Negative semidefinite Hermitian blocks of full rank, scaled as the plane-wave sphere's Coulomb term asks."""
    gen = _gen(seed)
    ng = case["ng"]
    blocks = []
    for _ in range(case["nw"]):
        a = _normal(gen, ng, ng) / math.sqrt(2.0 * ng)
        blocks.append(-0.2 * (a @ a.mH))
    chi = torch.stack(blocks)
    return {"chi": 0.5 * (chi + chi.mH), "v": _coulomb(torch.as_tensor(gsphere(ng, head=False), device="cuda"))}


def _handle(case, nq=1):
    grid = (case.get("n0", 24), case.get("n1", 24), case.get("n2", 24))
    prec = {"fp64": dict(prec="fp64", mtxel="fp64"), "split": dict(prec="ozaki", nslices=SLICES, mtxel="twofloat")}
    return gw.Chi0(grid, nq=nq, pair_chunk=case.get("chunk", 8192), **prec[case["prec"]])


def prepare(case, seed):
    k = case["kind"]
    st = {"kind": k, "omega": _omegas(case)}
    if k == "sigma":
        st.update(_pole_inputs(case, seed), nocc=case["nocc"], h=_handle(case))
        return st
    if k == "epsilon":
        st.update(_chi_inputs(case, seed), h=_handle(case))
        return st
    st.update(_system(case, seed))
    h = st["h"] = _handle(case, nq=case.get("nq", 1))
    if k == "grad":
        for x in ("cv", "ev", "cc", "ec"):
            st[x].requires_grad_(True)
        return st
    h.set_bands(0, 1, st["gpsi"], st["cc"], st["ec"])
    if k == "batch":
        for i in range(case["nq"]):
            h.set_bands(i, 0, st["gpsi"], st["cvs"][i], st["evs"][i])
            h.set_gsphere(i, st["gchis"][i])
        tot = sum(case["nw"] * n * n for n in _batch_ng(case))
        st["out"] = torch.empty(tot, dtype=torch.complex128, device="cuda")
        return st
    h.set_bands(0, 0, st["gpsi"], st["cv"], st["ev"])
    h.set_gsphere(0, st["gchi"])
    if k == "subspace":
        h.keep_pair_elements(True)
    return st


# ------------------------------------------------------------------ one pass


def run(st):
    k, h = st["kind"], st["h"]
    if k == "chi":  # the next q-point: its valence bands and sphere, then chi
        h.set_bands(0, 0, st["gpsi"], st["cv"], st["ev"])
        h.set_gsphere(0, st["gchi"])
        return h.compute(0, st["omega"])[0]
    if k == "batch":
        return h.compute_batch(range(len(st["cvs"])), st["omega"], out=st["out"])
    if k == "grad":
        leaves = [st["cv"], st["ev"], st["cc"], st["ec"]]
        chi = gw.Chi0Fn.apply(h, st["gpsi"], *leaves, st["gchi"], 0.0)
        return [chi.detach(), *torch.autograd.grad(chi, leaves, st["W"])]
    if k == "jvp":
        return h.jvp(0, st["omega"], st["dcv"], st["dcc"], st["dev"], st["dec"])
    if k == "subspace":
        return [h.compute(0, [0.0])[0], h.compute_subspace(0, st["basis"], st["omega"])]
    if k == "real":
        return h.compute_real(0, [2.0 + 15.0 * i for i in range(len(st["omega"]))], 0.1)
    if k == "sigma":
        return h.sigma_gpp(st["M"], st["En"], st["nocc"], st["omega2"], st["wt"], st["v"], st["E"])
    return h.epsilon_inverse(st["chi"], st["v"])


# ------------------------------------------------------------------ the same in plain double precision


def _grid(case, gpsi, c):
    """psi(r) = sum_K c(K) e^{iKr} on the case's grid."""
    n = (case["n0"], case["n1"], case["n2"])
    box = torch.zeros((c.shape[0], n[0] * n[1] * n[2]), dtype=torch.complex128, device=c.device)
    box = box.index_copy(1, _cells(case, gpsi), c)
    return torch.fft.ifftn(box.view(-1, *n), dim=(1, 2, 3), norm="forward")


def _cells(case, g):
    g = g.long()
    return ((g[:, 0] % case["n0"]) * case["n1"] + g[:, 1] % case["n1"]) * case["n2"] + g[:, 2] % case["n2"]


def _elements(case, psi_v, psi_c, cells):
    """M_vc(G) = (1/N) sum_r conj(psi_v) psi_c e^{iGr} for one valence band and some conduction bands."""
    f = torch.fft.ifftn(psi_v.conj()[None] * psi_c, dim=(1, 2, 3))
    return f.reshape(f.shape[0], -1)[:, cells]


def _weights(x, w, eta=None):
    if eta is None:
        return 4.0 * x / (x * x + w * w)
    z = torch.full_like(x, w) + 1j * eta
    return 2.0 / (x - z) + 2.0 / (x + z)


def _blocks(case, psi_c):
    step = max(1, int(3e9 / (16.0 * psi_c[0].numel())))
    return [(a, min(a + step, psi_c.shape[0])) for a in range(0, psi_c.shape[0], step)]


def _chi_exact(case, s, cv, ev, gchi, weights, basis=None):
    """chi at each of the weights (functions of x = E_v - E_c), pair block by pair block."""
    cells = _cells(case, gchi)
    psi_v, psi_c = _grid(case, s["gpsi"], cv), s["psi_c"]
    n = gchi.shape[0] if basis is None else basis.shape[1]
    out = torch.zeros((len(weights), n, n), dtype=torch.complex128, device="cuda")
    for v in range(cv.shape[0]):
        for a, b in _blocks(case, psi_c):
            m = _elements(case, psi_v[v], psi_c[a:b], cells)
            if basis is not None:
                m = m @ basis
            for i, f in enumerate(weights):
                out[i].addmm_(m.mH, f(ev[v] - s["ec"][a:b])[:, None] * m)
    return out


def _grad_exact(case, s):
    leaves = [s[x].requires_grad_(True) for x in ("cv", "ev", "cc", "ec")]
    cells = _cells(case, s["gchi"])
    psi = [_grid(case, s["gpsi"], s[x]).detach().requires_grad_(True) for x in ("cv", "cc")]
    e = [s[x].detach().requires_grad_(True) for x in ("ev", "ec")]
    chi = torch.zeros((case["ng"], case["ng"]), dtype=torch.complex128, device="cuda")
    for v in range(case["nv"]):
        m = _elements(case, psi[0][v], psi[1], cells)
        d = _weights(e[0][v] - e[1], 0.0)
        chi.addmm_(m.detach().mH, d.detach()[:, None] * m.detach())
        (d * ((m.conj() @ s["W"].conj()) * m).sum(1).real).sum().backward()
    out = []
    for x, p in (("cv", psi[0]), ("cc", psi[1])):
        out += torch.autograd.grad(_grid(case, s["gpsi"], s[x]), [s[x]], p.grad)
    del leaves
    return [chi, out[0], e[0].grad, out[1], e[1].grad]


def _jvp_exact(case, s, omegas):
    cells = _cells(case, s["gchi"])
    pv, pc, dpv, dpc = (_grid(case, s["gpsi"], s[x]) for x in ("cv", "cc", "dcv", "dcc"))
    out = torch.zeros((len(omegas), case["ng"], case["ng"]), dtype=torch.complex128, device="cuda")
    for v in range(case["nv"]):
        m = _elements(case, pv[v], pc, cells)
        dm = _elements(case, dpv[v], pc, cells) + _elements(case, pv[v], dpc, cells)
        x, dx = s["ev"][v] - s["ec"], s["dev"][v] - s["dec"]
        for i, w in enumerate(omegas):
            d, q = _weights(x, w), x * x + w * w
            dd = dx * 4.0 * (w * w - x * x) / (q * q)
            half = dm.mH @ (d[:, None] * m)
            out[i] += half + half.mH + m.mH @ (dd[:, None] * m)
    return out


def _sigma_exact(case, p):
    out = torch.zeros((case["nw"], case["nsig"], case["nsig"]), dtype=torch.complex128, device="cuda")
    a = p["v"][None, :] * p["omega2"] / (2.0 * p["wt"])
    for n in range(case["nb"]):
        sgn = -1.0 if n < case["nocc"] else 1.0
        for i, e in enumerate(p["E"]):
            pole = a / (e - p["En"][n] - sgn * p["wt"])
            out[i] += (p["M"][n].conj() @ pole) @ p["M"][n].T
    return out


def exact(case, seed):
    k, om = case["kind"], _omegas(case)
    if k == "sigma":
        return _sigma_exact(case, _pole_inputs(case, seed))
    if k == "epsilon":
        p = _chi_inputs(case, seed)
        eye = torch.eye(case["ng"], dtype=torch.complex128, device="cuda")
        return torch.linalg.inv(eye - p["v"][:, None] * p["chi"])
    s = _system(case, seed)
    if k == "grad":
        return _grad_exact(case, s)
    if k == "jvp":
        return _jvp_exact(case, s, om)
    s["psi_c"] = _grid(case, s["gpsi"], s["cc"])
    static = [lambda x: _weights(x, 0.0)]
    axis = [lambda x, w=w: _weights(x, w) for w in om]
    if k == "batch":
        return [_chi_exact(case, s, cv, ev, g, axis) for cv, ev, g in zip(s["cvs"], s["evs"], s["gchis"])]
    if k == "subspace":
        return [_chi_exact(case, s, s["cv"], s["ev"], s["gchi"], static),
                _chi_exact(case, s, s["cv"], s["ev"], s["gchi"], axis, basis=s["basis"])]
    if k == "real":
        return _chi_exact(case, s, s["cv"], s["ev"], s["gchi"],
                          [lambda x, w=2.0 + 15.0 * i: _weights(x, w, 0.1) for i in range(case["nw"])])
    return _chi_exact(case, s, s["cv"], s["ev"], s["gchi"], axis)
