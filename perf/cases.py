"""What a user of the library has it compute, as cases to time and to compare.

Each case is one call sequence through the public entry points (the C-ABI's ctypes binding in
``paper_1407_3444_gb300.chi0``) on seeded tight-binding eigen-data of the kinds in
``workloads.py``: the free-electron sphere, the 9-orbital Cr-like and 10-orbital FeSe-like
models and random 4- to 80-band models.  Eigen-data are diagonalised on the GPU.

Precision follows use: FP64 is the library's default and is what small meshes run in; the
mixed form is there for the production meshes (the repository's mixed workloads: 32^3 and up
at 9 bands, the 40- and 80-band models).

``exact`` is a plain 64-bit torch evaluation of the same integrals (both carvings, fourth
divided differences of x^3 ln|x|, cubic B-splines, Kramers-Kronig sums) that uses none of the
library's code.
"""
import ctypes as ct
import math

import numpy as np
import torch

from paper_1407_3444_gb300 import chi0, workloads

PI = math.pi

# bonds of the simple-cubic models (half of each shell; H(k) = t0 + sum 2 cos(2 pi k.R) t_R)
SC1 = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
SC2 = [(1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)]


def _case(kind, model, n, nb, nq, prec, nw=0, overlap="fp32", kq="shift", c64=False, windows=False, name=None):
    c = {"kind": kind, "model": model, "n0": n[0], "n1": n[1], "n2": n[2], "nb": nb, "nq": nq, "prec": prec,
         "nw": nw, "overlap": overlap, "kq": kq, "c64": c64, "windows": windows}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a first look at a model on a coarse mesh, default precision
        _case("static", "random", (6, 6, 6), 4, 2, "fp64", kq="explicit", name="tiny_static_fp64"),
        # the validation run every user starts with: free-electron Lindhard curve, CMA, 32 q
        _case("static", "free", (16, 16, 16), 1, 32, "fp64", kq="explicit", name="free_electron_32q_fp64"),
        # a q-path segment of the Cr-like model in the default precision
        _case("static", "cr", (24, 24, 24), 9, 4, "fp64", kq="explicit", name="cr_static_24_fp64"),
        # the Cr-like production run (a stretch of its 256 q on Gamma-X-M-Gamma)
        _case("static", "cr", (48, 48, 48), 9, 4, "mixed", kq="explicit", name="cr_static_48_mixed"),
        # the same from page-locked host memory, as a band-structure code hands it over
        _case("host_static", "cr", (32, 32, 32), 9, 4, "mixed", kq="explicit", name="cr_static_32_host_mixed"),
        # band-truncation sweep: 40 bands, every q with its own window, tensor-core overlaps
        _case("static", "random", (32, 32, 32), 40, 16, "mixed", overlap="bf16x3", windows=True,
              name="sweep_static_40b_bf16x3"),
        # band-pair histogram on an odd, anisotropic mesh, Gamma among the q points
        _case("pairs", "random", (15, 14, 13), 7, 3, "fp64", name="pairs_ragged_7b_fp64"),
        # the FeSe-like spectrum, 512 frequencies
        _case("dynamic", "fese", (64, 64, 16), 10, 1, "mixed", nw=512, kq="explicit", name="fese_dynamic_512w_mixed"),
        # a spectrum of the same model on a coarse mesh in the default precision
        _case("dynamic", "fese", (16, 16, 8), 10, 2, "fp64", nw=128, kq="explicit", name="fese_dynamic_128w_fp64"),
        # the 80-band run (the largest mesh whose pass stays well below two seconds)
        _case("dynamic", "random", (32, 32, 32), 80, 1, "mixed", nw=256, overlap="bf16x6", c64=True,
              name="large_dynamic_80b_bf16x6"),
        # Im on a uniform grid and Re by Kramers-Kronig
        _case("kk", "random", (32, 32, 32), 12, 1, "mixed", nw=400, name="kk_12b_400w_mixed"),
        # a q that is not on the mesh: interpolated k+q data, then the static value
        _case("offgrid", "cr", (33, 32, 31), 9, 1, "mixed", name="offgrid_static_9b_mixed"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed families' ranges: odd and anisotropic meshes among them."""
    kind = rng.choice(["small", "free", "cr64", "cr", "host", "sweep", "pairs", "fese", "dyn64", "large", "kk", "offgrid"])
    r = rng.randint
    if kind == "small":
        return _case("static", "random", (r(4, 12), r(4, 12), r(4, 12)), r(2, 8), r(1, 4), "fp64",
                     kq=rng.choice(["explicit", "shift"]), c64=rng.random() < 0.3)
    if kind == "free":
        n = r(10, 20)
        return _case("static", "free", (n, n, n), 1, _logint(rng, 2, 32), "fp64", kq="explicit")
    if kind == "cr64":
        return _case("static", "cr", (r(12, 26), r(12, 26), r(12, 26)), 9, r(1, 4), "fp64",
                     kq=rng.choice(["explicit", "shift"]))
    if kind == "cr":
        return _case("static", "cr", (r(34, 48), r(34, 48), r(34, 48)), 9, r(1, 4), "mixed",
                     kq=rng.choice(["explicit", "shift"]), c64=rng.random() < 0.3)
    if kind == "host":
        return _case("host_static", "cr", (r(32, 36), r(32, 36), r(32, 36)), 9, r(1, 4), "mixed", kq="explicit")
    if kind == "sweep":
        return _case("static", "random", (r(24, 32), r(24, 32), r(24, 32)), rng.choice([20, 25, 30, 32, 35, 36, 40]), r(1, 16), "mixed",
                     overlap=rng.choice(["fp32", "bf16x3", "bf16x6"]), windows=rng.random() < 0.7)
    if kind == "pairs":
        return _case("pairs", "random", (r(8, 17), r(8, 17), r(8, 17)), r(4, 9), r(1, 4), "fp64")
    if kind == "fese":
        return _case("dynamic", "fese", (r(40, 64), r(40, 64), r(14, 18)), 10, 1, "mixed", nw=_logint(rng, 48, 512),
                     kq=rng.choice(["explicit", "shift"]))
    if kind == "dyn64":
        return _case("dynamic", "fese", (r(8, 17), r(8, 17), r(6, 9)), 10, r(1, 2), "fp64", nw=_logint(rng, 12, 160),
                     kq=rng.choice(["explicit", "shift"]))
    if kind == "large":
        return _case("dynamic", "random", (r(20, 32), r(20, 32), r(20, 32)), rng.choice([32, 36, 42, 49, 56, 63, 72, 80]), 1, "mixed", nw=r(64, 256),
                     overlap=rng.choice(["bf16x3", "bf16x6"]), c64=True)
    if kind == "kk":
        return _case("kk", "random", (r(28, 34), r(28, 34), r(28, 34)), r(8, 14), 1, "mixed", nw=r(200, 512))
    return _case("offgrid", "cr", (r(32, 36), r(32, 36), r(32, 36)), 9, 1, "mixed", c64=rng.random() < 0.3)


# ------------------------------------------------------------------------------ inputs
def _herm(rng, n, sigma):
    g = rng.normal(0.0, sigma, (n, n)) + 1j * rng.normal(0.0, sigma, (n, n))
    return 0.5 * (g + g.conj().T)


def _model(case, rng):
    """(t0, bonds) of the case's tight-binding model (the recipes of workloads.py, seeded)."""
    nb = case["nb"]
    if case["model"] == "cr":
        t0 = np.diag(rng.uniform(-2.0, 2.0, nb)).astype(np.complex128)
        return t0, [(R, _herm(rng, nb, 0.8)) for R in SC1] + [(R, _herm(rng, nb, 0.3)) for R in SC2]
    if case["model"] == "fese":
        h = nb // 2
        t0 = np.diag(rng.uniform(-1.0, 1.0, nb)).astype(np.complex128)
        g = rng.normal(0.0, 0.5, (h, nb - h)) + 1j * rng.normal(0.0, 0.5, (h, nb - h))
        t0[:h, h:] = g
        t0[h:, :h] = g.conj().T
        return t0, [(SC1[0], _herm(rng, nb, 0.5)), (SC1[1], _herm(rng, nb, 0.5)), (SC1[2], _herm(rng, nb, 0.05))]
    return _random(rng, nb, 8.0)


def _random(rng, nb, spread):
    """Random onsite and nearest-neighbour model, about ``spread`` from the lowest to the highest band."""
    s = spread / (8.0 + 11.0 * math.sqrt(nb))
    t0 = _herm(rng, nb, 1.0)
    return t0 * s, [(R, _herm(rng, nb, 1.0) * s) for R in SC1]


def _eig(model, frac, c64):
    """Energies [N, nb] (float64, ascending) and eigenvectors [N, norb, nb] at fractional k."""
    t0, bonds = model
    dt = torch.complex64 if c64 else torch.complex128
    t0 = torch.from_numpy(t0).to("cuda", dt)
    E, C = [], []
    chunk = min(1 << 15, max(1, (1 << 24) // (t0.shape[0] ** 2)))
    for f in frac.split(chunk):
        H = t0.expand(f.shape[0], -1, -1).clone()
        for R, t in bonds:
            # the phase reduced to [0, 1/2]: k and -k get the same Hamiltonian to the last bit
            p = (f @ torch.tensor(R, dtype=torch.float64, device="cuda")) % 1.0
            p = torch.round(torch.minimum(p, 1.0 - p) * 2.0 ** 40) / 2.0 ** 40
            H += (2.0 * torch.cos(2.0 * PI * p)).to(H.real.dtype)[:, None, None] * torch.from_numpy(t).to("cuda", dt)
        w, v = torch.linalg.eigh(H)
        E.append(w.double())
        C.append(v)
    E = torch.sort(torch.cat(E), dim=1).values  # (32-bit solvers may leave ties a rounding apart)
    return E.contiguous(), torch.cat(C).contiguous()


def _mesh(n):
    ax = [torch.arange(m, dtype=torch.float64, device="cuda") / m for m in n]
    return torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 3)


def _eig_mesh(case, rng, n):
    """(model, E, C) of the case on the mesh.  Random models past 32 bands are the sum of two
    independent random models on a product of orbital spaces, H = H_1 x 1 + 1 x H_2 (batched
    diagonalisation on the GPU is only quick for small matrices)."""
    nb, mesh = case["nb"], _mesh(n)
    if case["model"] != "random" or nb <= 32:
        model = _model(case, rng)
        return (model, *_eig(model, mesh, case["c64"]))
    p = max(x for x in range(1, int(math.sqrt(nb)) + 1) if nb % x == 0)
    (Ea, Ca), (Eb, Cb) = (_eig(_random(rng, m, 4.0), mesh, False) for m in (p, nb // p))
    E, order = (Ea[:, :, None] + Eb[:, None, :]).reshape(-1, nb).sort(dim=1, stable=True)
    C = torch.empty(E.shape[0], nb, nb, dtype=torch.complex64 if case["c64"] else torch.complex128, device="cuda")
    for a in range(0, E.shape[0], 8192):
        x = torch.einsum("kai,kbj->kabij", Ca[a:a + 8192].to(C.dtype), Cb[a:a + 8192].to(C.dtype)).reshape(-1, nb, nb)
        C[a:a + 8192] = torch.gather(x, 2, order[a:a + 8192, None, :].expand(-1, nb, -1))
    return None, E.contiguous(), C


def _fermi(E, nocc):
    """Midpoint between the last occupied and the first empty level at this filling, moved to
    the nearest gap between distinct levels."""
    flat = E.reshape(-1).sort().values
    k = min(max(int(round(nocc * E.shape[0])), 1), flat.numel() - 1)
    gaps = torch.nonzero(flat[1:] - flat[:-1] > 1e-9 * max(1.0, float(flat.abs().max())))[:, 0] + 1
    k = int(gaps[(gaps - k).abs().argmin()])
    return float(0.5 * (flat[k - 1] + flat[k]))


def _inputs(case, seed):
    """Everything the call reads, made from the seed: a dict of device tensors and numbers."""
    rng = np.random.default_rng(1407344400 + 7919 * (int(seed) % (1 << 31)))
    n = (case["n0"], case["n1"], case["n2"])
    nb, nq = case["nb"], case["nq"]
    d = {"n": n, "nb": nb, "periodic": 1, "cma": 0, "C": None, "windows": [(0, nb)] * nq, "gamma": [0] * nq,
         "shift": [(0, 0, 0)] * nq, "Eq": [None] * nq, "Cq": [None] * nq}
    if case["model"] == "free":
        kf = (rng.uniform(0.35, 0.45) * (2 * PI) ** 3 * 3.0 / (4.0 * PI)) ** (1.0 / 3.0)
        ax = [-PI + 2.0 * PI * torch.arange(m + 1, dtype=torch.float64, device="cuda") / m for m in n]
        K = torch.stack(torch.meshgrid(*ax, indexing="ij"), dim=-1).reshape(-1, 3)
        d.update(periodic=0, cma=1, ef=0.5 * kf * kf, E=(0.5 * (K * K).sum(1))[:, None].contiguous())
        for j in range(nq):  # (100), 0 .. 2 kF
            x = 2.0 * kf * j / max(1, nq - 1)
            Kq = K + torch.tensor([x, 0.0, 0.0], dtype=torch.float64, device="cuda")
            d["Eq"][j] = (0.5 * (Kq * Kq).sum(1))[:, None].contiguous()
            d["gamma"][j] = int(x == 0.0)
        return d
    model, d["E"], d["C"] = _eig_mesh(case, rng, n)
    nocc = {"cr": 2 * nb // 3, "fese": 6 * nb // 10}.get(case["model"], nb / 2)
    d["ef"] = _fermi(d["E"], nocc)
    d["qfrac"] = tuple(float(x) for x in rng.uniform(0.05, 0.45, 3))
    for j in range(nq):
        if case["kind"] == "pairs" and j == 0:
            d["gamma"][j] = 1  # on-grid Gamma
        elif case["kq"] == "explicit":
            q = torch.from_numpy(rng.uniform(0.02, 0.5, 3)).to("cuda")
            if case["model"] == "fese":  # on Gamma-M
                q[1], q[2] = q[0], 0.0
            d["Eq"][j], d["Cq"][j] = _eig(model, _mesh(n) + q, case["c64"])
        else:
            while d["shift"][j] == (0, 0, 0):
                d["shift"][j] = tuple(int(rng.integers(0, m)) for m in n)
        if case["windows"]:  # centred on the Fermi level, 4 bands and up
            w = int(rng.integers(4, nb + 1))
            lo = min(max(int(nocc) - w // 2, 0), nb - w)
            d["windows"][j] = (lo, lo + w)
    return d


# ------------------------------------------------------------------------------ the calls
class _State:
    """What a program keeps: the inputs, the plan and the q descriptors."""

    def __init__(self, case, d):
        self.case, self.d = case, d
        o = chi0.chi0_opts_default()
        o.precision = chi0.CHI0_PREC_FP64 if case["prec"] == "fp64" else chi0.CHI0_PREC_MIXED
        o.overlap = chi0.OVERLAP_MODES[case["overlap"]]
        o.cma = d["cma"]
        o.inputs_on_device = o.outputs_on_device = 1
        o.stream = ct.c_void_p(torch.cuda.current_stream().cuda_stream)
        g = chi0.chi0_kgrid_t()
        g.n[:] = list(d["n"])
        g.periodic, g.nbands, g.norb, g.e_fermi = d["periodic"], d["nb"], d["nb"], d["ef"]
        g.evec_dtype = chi0.CHI0_C64 if case["c64"] else chi0.CHI0_C128
        g.energies = d["E"].data_ptr()
        g.evecs = None if d["cma"] else d["C"].data_ptr()
        self.h = chi0.chi0_plan(g, None, chi0.chi0_band_window_t(0, d["nb"]), o)
        self.q = (chi0.chi0_q_t * case["nq"])()
        for j in range(case["nq"]):
            self.q[j].shift[:] = list(d["shift"][j])
            self.q[j].e_kq = d["Eq"][j].data_ptr() if d["Eq"][j] is not None else None
            self.q[j].c_kq = d["Cq"][j].data_ptr() if d["Cq"][j] is not None else None
            self.q[j].win = chi0.chi0_band_window_t(*d["windows"][j])
            self.q[j].gamma = d["gamma"][j]

    def __del__(self):
        if getattr(self, "h", None):
            chi0.chi0_destroy(self.h)
            self.h = None


def _omega(case):
    """w in [0, 2] eV, as the dynamic workloads have it."""
    return torch.linspace(0.0, 2.0, case["nw"], dtype=torch.float64, device="cuda")


def _wmax(d):
    """A grid end past the largest band-pair energy (the transform needs the whole spectrum)."""
    return 1.01 * float(d["E"].max() - d["E"].min())


def prepare(case, seed):
    d = _inputs(case, seed)
    if case["kind"] == "host_static":
        W = workloads.Workload("host", d["n"], True, d["nb"], d["nb"], d["E"].cpu().numpy(), d["C"].cpu().numpy(),
                               d["ef"], (0, d["nb"]), False,
                               [workloads.QPoint(Eq=e.cpu().numpy(), Cq=c.cpu().numpy()) for e, c in zip(d["Eq"], d["Cq"])])
        del d
        return {"case": case, "plan": chi0.Plan(W, precision=case["prec"], device=False,
                                                staged=chi0.HostInputs(W, pinned=True))}
    s = {"case": case, "plan": _State(case, d)}
    if case["kind"] == "dynamic":
        s["omega"] = _omega(case)
    elif case["kind"] == "kk":
        s["wmax"] = _wmax(d)
    elif case["kind"] == "offgrid":
        s["q"] = (ct.c_double * 3)(*d["qfrac"])
    return s


def run(state):
    case, P = state["case"], state["plan"]
    kind, nq, nw = case["kind"], case["nq"], case["nw"]
    if kind == "host_static":
        return P.static()
    f64 = dict(dtype=torch.float64, device="cuda")
    chi = torch.empty(nq, **f64)
    if kind == "static":
        chi0.chi0_static(P.h, P.q, nq, chi.data_ptr())
        return chi
    if kind == "pairs":
        pairs = torch.empty(sum((hi - lo) ** 2 for lo, hi in P.d["windows"]), **f64)
        chi0.chi0_static_pairs(P.h, P.q, nq, chi.data_ptr(), pairs.data_ptr())
        return {"chi": chi, "pairs": pairs}
    if kind == "offgrid":
        E, C = torch.empty_like(P.d["E"]), torch.empty_like(P.d["C"])
        chi0.chi0_interpolate_kq(P.h, state["q"], E.data_ptr(), C.data_ptr())
        q = (chi0.chi0_q_t * 1)()
        q[0].e_kq, q[0].c_kq, q[0].win = E.data_ptr(), C.data_ptr(), chi0.chi0_band_window_t(-1, -1)
        chi0.chi0_static(P.h, q, 1, chi.data_ptr())
        return {"chi": chi, "e_kq": E, "c_kq": C}
    re, im = torch.empty(nq, nw, **f64), torch.empty(nq, nw, **f64)
    if kind == "dynamic":
        chi0.chi0_dynamic(P.h, P.q, nq, state["omega"].data_ptr(), nw, re.data_ptr(), im.data_ptr())
    else:
        chi0.chi0_dynamic_kk(P.h, P.q, nq, state["wmax"], nw, re.data_ptr(), im.data_ptr())
    return {"re": re, "im": im}


def work(case):
    """Bytes: energies and eigenvectors at k once, explicit k+q data once per q, results once.
    Flops: the overlaps (8 w^2 norb per corner and q) and, per tetrahedron and (occupied, empty)
    pair, a closed form of about 100 (static), or moments and near frequencies of about 500."""
    n, nb, nq = (case["n0"], case["n1"], case["n2"]), case["nb"], case["nq"]
    free = case["model"] == "free"
    nc = math.prod(m + 1 for m in n) if free else math.prod(n)
    vec = 0 if free else nb * nb * (8 if case["c64"] else 16)
    kq = nq if (case["kq"] == "explicit" or case["kind"] == "offgrid") else 0
    out = nq * max(1, case["nw"]) * (16 if case["nw"] else 8)
    if case["kind"] == "offgrid":
        out += nc * (8 * nb + vec)
    w = 0.6 * nb if case["windows"] else nb  # mean window width
    occ = w * {"cr": 2 / 3, "fese": 0.6, "free": 0.4}.get(case["model"], 0.5)
    pairs = 0.25 if free else occ * (w - occ)
    per = 100 if not case["nw"] else 500
    return {"bytes": nc * (8 * nb + vec) * (1 + kq) + out,
            "flops": nq * ((0 if free else 8 * w * w * nb * nc) + 6 * math.prod(n) * pairs * per)}


# ------------------------------------------------------------------------------ 64-bit values
def _mix(P, Q, t):
    return (1.0 - t)[:, None] * P + t[:, None] * Q


def _cut(V, r, ids, second):
    """Keeps the part of every tetrahedron where the key is negative: key a (the first carving)
    or -(a + D) (the second).  V [M, 4 vertices, (a, D, f)]; returns pieces with their volume
    ratios and parents."""
    key = -(V[..., 0] + V[..., 1]) if second else V[..., 0]
    key, p = key.sort(dim=1)
    V = torch.gather(V, 1, p[..., None].expand(-1, -1, 3))
    neg = (key < 0).sum(1)
    out = []

    def cutter(m):
        S, k = V[m], key[m]

        def c(i, j):
            t = k[:, i] / (k[:, i] - k[:, j])
            X = _mix(S[:, i], S[:, j], t)
            if not second:
                X[:, 0] = 0.0
            return X, t
        return S, c, r[m], ids[m]

    m = neg == 4
    out.append((V[m], r[m], ids[m]))
    S, c, rr, ii = cutter(neg == 1)
    (A, t1), (B, t2), (D, t3) = c(0, 1), c(0, 2), c(0, 3)
    out.append((torch.stack([S[:, 0], A, B, D], 1), rr * t1 * t2 * t3, ii))
    S, c, rr, ii = cutter(neg == 2)
    (P02, u0), (P03, v0), (P12, u1), (P13, v1) = c(0, 2), c(0, 3), c(1, 2), c(1, 3)
    out.append((torch.stack([S[:, 0], P02, P03, S[:, 1]], 1), rr * u0 * v0, ii))
    out.append((torch.stack([P02, P03, S[:, 1], P12], 1), rr * v0 * (1 - u0) * u1, ii))
    out.append((torch.stack([P03, S[:, 1], P12, P13], 1), rr * (1 - v0) * u1 * v1, ii))
    S, c, rr, ii = cutter(neg == 3)
    (P03, s0), (P13, s1), (P23, s2) = c(0, 3), c(1, 3), c(2, 3)
    out.append((torch.stack([S[:, 0], S[:, 1], S[:, 2], P03], 1), rr * s0, ii))
    out.append((torch.stack([S[:, 1], S[:, 2], P03, P13], 1), rr * (1 - s0) * s1, ii))
    out.append((torch.stack([S[:, 2], P03, P13, P23], 1), rr * (1 - s0) * (1 - s1) * s2, ii))
    V, r, ids = (torch.cat(x) for x in zip(*out))
    ok = r > 0
    return V[ok], r[ok], ids[ok]


def _g0(t):
    return torch.where(t == 0, torch.zeros_like(t), t ** 3 * torch.log(t.abs().clamp_min(1e-300)))


def _taylor(t):
    """Divided difference of x^3 ln|x| over n + 1 knots [M, n + 1] that lie together, from the
    Taylor series about their mean."""
    n = t.shape[1] - 1
    c = t.mean(1)
    e = (t - c[:, None]) / c[:, None]
    L = torch.log(c.abs())
    h = [torch.ones_like(c) for _ in range(n + 1)]
    low = torch.zeros_like(c)
    high = torch.zeros_like(c)
    der = {1: 3 * c * c * L + c * c, 2: 3 * c * L + 2.5 * c, 3: L + 11.0 / 6.0}
    for k in range(n, n + 36):
        if k > n:
            h[0] = e[:, 0] * h[0]
            for i in range(1, n + 1):
                h[i] = h[i - 1] + e[:, i] * h[i]
        if k < 4:
            low = low + der[k] * c ** (k - n) * h[n]
        else:
            high = high + (6.0 * (-1) ** k / (k * (k - 1) * (k - 2) * (k - 3))) * h[n]
    return low + c ** (3 - n) * high


def _dd5(t):
    """g[t_0 .. t_4], g = x^3 ln|x|, sorted knots [M, 5]."""
    v = [_g0(t[:, i]) for i in range(5)]
    for n in range(1, 5):
        for i in range(0, 5 - n):
            a, b = t[:, i], t[:, i + n]
            d = b - a
            near = ((a > 0) & (d <= 0.25 * a)) | ((b < 0) & (d <= -0.25 * b))
            r = torch.where(d > 0, (v[i + 1] - v[i]) / torch.where(d > 0, d, torch.ones_like(d)), torch.zeros_like(d))
            at = torch.nonzero(near)[:, 0]
            if at.numel():
                r[at] = _taylor(t[at, i:i + n + 1])
            v[i] = r
    return v[0]


def _inv(x, f):
    """sum_j f_j (1/V) int lambda_j / X over a tetrahedron with X = x at its vertices (sorted;
    principal value across X = 0)."""
    out = torch.zeros_like(x[:, 0])
    near = ((x[:, 0] > 0) | (x[:, 3] < 0)) & (x[:, 3] - x[:, 0] <= 0.5 * (x[:, 0] + x[:, 3]).abs())
    at = torch.nonzero(near)[:, 0]
    if at.numel():
        y, ff = x[at], f[at]
        c = 0.5 * (y[:, 0] + y[:, 3])
        e = (y - c[:, None]) / c[:, None]
        H = [torch.ones_like(c) for _ in range(4)]
        P = [torch.ones_like(c) for _ in range(4)]
        s = 0.25 * ff.sum(1)
        for k in range(1, 56):
            H[0] = e[:, 0] * H[0]
            for i in range(1, 4):
                H[i] = H[i - 1] + e[:, i] * H[i]
            P = [H[3] + e[:, j] * P[j] for j in range(4)]
            s = s + ((-1) ** k * 6.0 / ((k + 1) * (k + 2) * (k + 3) * (k + 4))) * sum(ff[:, j] * P[j] for j in range(4))
        out[at] = s / c
    at = torch.nonzero(~near)[:, 0]
    if at.numel():
        y, ff = x[at], f[at]
        s = y.abs().amax(1).clamp_min(1e-300)
        u = y / s[:, None]
        out[at] = sum(ff[:, j] * _dd5(torch.cat([u[:, :j + 1], u[:, j:]], 1)) for j in range(4)) / s
    return out


def _bspline(t, order):
    """M-spline M(0; t) of the sorted knots t (integral 1) by the de Boor-Cox recursion."""
    M = [torch.where((t[:, i] <= 0) & (t[:, i + 1] > 0), 1.0 / (t[:, i + 1] - t[:, i]).clamp_min(1e-300),
                     torch.zeros_like(t[:, 0])) for i in range(order)]
    for k in range(2, order + 1):
        for i in range(order + 1 - k):
            d = t[:, i + k] - t[:, i]
            v = k * (-t[:, i] * M[i] + t[:, i + k] * M[i + 1]) / ((k - 1) * torch.where(d > 0, d, torch.ones_like(d)))
            M[i] = torch.where(d > 0, v, torch.zeros_like(d))
    return M[0]


def _delta(x, f):
    """sum_j f_j (1/V) int lambda_j delta(X), sorted vertex values x."""
    return 0.25 * sum(f[:, j] * _bspline(torch.cat([x[:, :j + 1], x[:, j:]], 1), 4) for j in range(4))


def _tets(d):
    """Corner indices [6 cubes, 4] of the mesh split around the cubes' (000)-(111) diagonals."""
    n = d["n"]
    N = [m if d["periodic"] else m + 1 for m in n]
    i = torch.stack(torch.meshgrid(*[torch.arange(m, device="cuda") for m in n], indexing="ij"), -1).reshape(-1, 1, 1, 3)
    off = []
    for a in range(3):
        for b in range(3):
            if a != b:
                o = np.zeros((4, 3), dtype=np.int64)
                o[1:, a] = 1
                o[2:, b] = 1
                o[3] = 1
                off.append(o)
    x = i + torch.from_numpy(np.stack(off)).to("cuda")[None]

    def index(shift):
        y = x + torch.tensor(shift, device="cuda")
        if d["periodic"]:
            y = y % torch.tensor(N, device="cuda")
        return ((y[..., 0] * N[1] + y[..., 1]) * N[2] + y[..., 2]).reshape(-1, 4)
    return index


def _pieces(d, j, chunk):
    """The final tetrahedra of q point j: sorted D and f at their vertices, volumes, band pairs,
    a chunk of items at a time."""
    lo, hi = d["windows"][j]
    w = hi - lo
    index = _tets(d)
    ck = index((0, 0, 0))
    cq = ck if d["Eq"][j] is not None else index(d["shift"][j])
    A = d["E"][:, lo:hi] - d["ef"]
    B = (d["E"] if d["Eq"][j] is None else d["Eq"][j])[:, lo:hi] - d["ef"]
    occ, emp = A[ck].amin(1) < 0, B[cq].amax(1) > 0  # [T, w]
    W2 = None
    if not d["cma"]:
        Ck = d["C"][:, :, lo:hi].to(torch.complex128)
        if d["Eq"][j] is not None:
            Cq = d["Cq"][j][:, :, lo:hi].to(torch.complex128)
        else:
            n = d["n"]
            Cq = torch.roll(d["C"].reshape(*n, -1), [-s for s in d["shift"][j]], (0, 1, 2)).reshape(d["C"].shape)
            Cq = Cq[:, :, lo:hi].to(torch.complex128)
        W2 = torch.matmul(Ck.conj().transpose(1, 2), Cq).abs() ** 2
    gamma = d["gamma"][j] or (d["Eq"][j] is None and not any(d["shift"][j]))
    vol = 1.0 / (6.0 * math.prod(d["n"]))
    step = max(1, chunk // (w * w))
    for t0 in range(0, ck.shape[0], step):
        m = occ[t0:t0 + step, :, None] & emp[t0:t0 + step, None, :]
        if gamma:
            m &= ~torch.eye(w, dtype=torch.bool, device="cuda")
        t, bm, bn = torch.nonzero(m, as_tuple=True)
        if not t.numel():
            continue
        k4, q4 = ck[t0 + t], cq[t0 + t]
        a, b = A[k4, bm[:, None]], B[q4, bn[:, None]]
        f = torch.ones_like(a) if W2 is None else W2[k4, bm[:, None], bn[:, None]]
        V, r, ids = _cut(torch.stack([a, b - a, f], -1), torch.full_like(a[:, 0], vol), torch.arange(t.numel(), device="cuda"), False)
        V, r, ids = _cut(V, r, ids, True)
        x, p = V[..., 1].clamp_min(0.0).sort(dim=1)
        yield x, torch.gather(V[..., 2], 1, p), r, (bm * w + bn)[ids]


def _dos(d, j):
    """Tetrahedron density of states at the Fermi level per band of q point j's window (one spin)."""
    lo, hi = d["windows"][j]
    a = (d["E"][:, lo:hi] - d["ef"])[_tets(d)((0, 0, 0))]
    return torch.stack([_bspline(a[:, :, b].sort(dim=1).values, 3).sum() for b in range(hi - lo)]) / (6.0 * math.prod(d["n"]))


def exact(case, seed):
    d = _inputs(case, seed)
    nq, nw, kind = case["nq"], case["nw"], case["kind"]
    tets = 6 * math.prod(d["n"])
    if kind == "dynamic" and tets * case["nb"] ** 2 * nw > 4e8:
        return None  # more than some seconds of closed forms
    if kind != "dynamic" and tets * sum((hi - lo) ** 2 for lo, hi in d["windows"]) > 4e8:
        return None
    if kind == "offgrid":
        E, C = _interpolate(d, d["qfrac"])
        d["Eq"], d["Cq"] = [E], [C.to(d["C"].dtype)]
    chi, pairs, re, im = [], [], [], []
    w = _omega(case) if kind == "dynamic" else torch.arange(nw, dtype=torch.float64, device="cuda") * ((_wmax(d) if kind == "kk" else 0.0) / max(1, nw - 1))
    for j in range(nq):
        wj = d["windows"][j][1] - d["windows"][j][0]
        gamma = d["gamma"][j] or (d["Eq"][j] is None and not any(d["shift"][j]))
        dos = _dos(d, j) if gamma else torch.zeros(wj, dtype=torch.float64, device="cuda")
        P = torch.diag(dos).reshape(-1)
        R, I = torch.zeros_like(w), torch.zeros_like(w)
        for x, f, r, pair in _pieces(d, j, 1 << 21):
            if kind in ("dynamic", "kk"):
                _spectrum(x, f, r, w, R if kind == "dynamic" else None, I)
            else:
                P = P.index_add(0, pair, 2.0 * r * _inv(x, f))
        if kind == "dynamic":
            R = R + torch.where(w == 0, dos.sum(), torch.zeros_like(w))
        if kind == "kk":
            R = _kramers_kronig(I, w) + torch.where(w == 0, dos.sum(), torch.zeros_like(w))
        chi.append(2.0 * P.sum())
        pairs.append(2.0 * P)
        re.append(2.0 * R)
        im.append(2.0 * I)
    if kind in ("dynamic", "kk"):
        return {"re": torch.stack(re), "im": torch.stack(im)}
    if kind == "pairs":
        return {"chi": torch.stack(chi), "pairs": torch.cat(pairs)}
    if kind == "offgrid":
        return {"chi": torch.stack(chi), "e_kq": E, "c_kq": C}
    return torch.stack(chi)


def _spectrum(x, f, r, w, R, I):
    """Adds the pieces' Re (both terms, if R is given) and Im at the frequencies w >= 0."""
    if R is not None:
        step = max(1, (1 << 21) // w.numel())
        for a in range(0, x.shape[0], step):
            y, g, v = x[a:a + step], f[a:a + step], r[a:a + step]
            shape = (y.shape[0], w.numel(), 4)
            g = g[:, None, :].expand(shape).reshape(-1, 4)
            for s in (-1.0, 1.0):
                z = (y[:, None, :] + s * w[None, :, None]).reshape(-1, 4)
                R += (v[:, None] * _inv(z, g).reshape(shape[:2])).sum(0)
    lo, hi = torch.searchsorted(w, x[:, 0].contiguous(), right=True), torch.searchsorted(w, x[:, 3].contiguous())
    cnt = (hi - lo).clamp_min(0)
    ends = cnt.cumsum(0)
    total = int(ends[-1]) if cnt.numel() else 0
    for a in range(0, total, 1 << 22):
        e = torch.arange(a, min(total, a + (1 << 22)), device="cuda")
        p = torch.searchsorted(ends, e, right=True)
        iw = lo[p] + (e - (ends[p] - cnt[p]))
        v = PI * r[p] * _delta(x[p] - w[iw, None], f[p])
        I += torch.where(w > 0, torch.zeros_like(w).index_add(0, iw, v), torch.zeros_like(w))


def _kramers_kronig(I, w):
    """(1/pi) PV int Im(u) [1/(u - w) + 1/(u + w)] du, Im piecewise linear on the nodes, 0 past them."""
    m, du = w.numel(), float(w[1])
    pad = torch.zeros(m + 3, dtype=torch.float64, device="cuda")
    pad[2:m + 1] = I[1:]
    d2 = pad[:-2] - 2.0 * pad[1:-1] + pad[2:]  # nodes 0 .. m
    u = torch.arange(m + 1, dtype=torch.float64, device="cuda") * du

    def G(x):
        return x * torch.log(x.abs().clamp_min(1e-300))
    return ((G(u[None, :] - w[:, None]) + G(u[None, :] + w[:, None])) * d2[None, :]).sum(1) / (PI * du)


def _interpolate(d, q):
    """Energies and eigenvectors at k + q, linear in the mesh tetrahedron that holds k + q, each
    band's corner vectors turned onto the first one's phase, the sum normalised."""
    n = torch.tensor(d["n"], device="cuda")
    i = (_mesh(d["n"]) * n).round()
    x = i + torch.tensor(q, dtype=torch.float64, device="cuda") * n
    base = torch.floor(x)
    t, p = (x - base).sort(dim=1, descending=True, stable=True)
    wt = torch.stack([1 - t[:, 0], t[:, 0] - t[:, 1], t[:, 1] - t[:, 2], t[:, 2]], 1)
    at = base.long()
    E, C = 0.0, 0.0
    first = None
    for v in range(4):
        if v:
            at = at.scatter_add(1, p[:, v - 1:v], torch.ones_like(p[:, :1]))
        y = at % n
        c = (y[:, 0] * d["n"][1] + y[:, 1]) * d["n"][2] + y[:, 2]
        z = d["C"][c].to(torch.complex128)
        if v == 0:
            first = z
        else:
            s = (first.conj() * z).sum(1, keepdim=True)
            z = z * torch.where(s.abs() > 0, s.conj() / s.abs().clamp_min(1e-300), torch.ones_like(s))
        E = E + wt[:, v, None] * d["E"][c]
        C = C + wt[:, v, None, None] * z
    return E, C / C.abs().square().sum(1, keepdim=True).sqrt().clamp_min(1e-300)
