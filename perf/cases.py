"""Performance cases: what a program built on this framework has it do.

Kinds of case (one pass = one call chain a user's program makes):
  layers   two brickwork layers (even bonds left to right, odd bonds right to
           left) on a saturated state the program already holds, then the
           one- and two-site Pauli expectation values: the unit a long
           emulation repeats.  Options: complex64 / complex128, exact
           truncation or subspace iteration (sketch of k columns, q power
           iterations).
  emulate  a whole circuit from the product state at several noise levels and
           the fit to the target level, through runner.emulate: superoperator
           build, state creation, every layer from bond dimension 1 up, the
           sweep, the fit.
  serve    a burst of such jobs submitted to a Server and collected.
  expect   the expectation sweep of a state at hand (long chains, wide bonds).
  entropy  the MPO entropy of every bond.
  fit      the noise extrapolation of a table of expectation values.
  gemm     the batched complex64 GEMM entry point (the gate step's routine).

States of the layers / expect / entropy cases are random right-canonical
chains with a graded Schmidt spectrum and a dominant identity component, as a
noisy mixed state has; observables are all one- and neighbouring two-site Pauli
strings.  Results of complex64 states are handed back in single
precision (the precision they were computed in), those of complex128 states
in double; the emulation fidelity as F itself, which is what the fits weight
with and what single precision determines well (log F near 0 it does not).
"""
import math
import types

import numpy as np
import torch

from paper_2501_13237_gb300 import nne, runner

DEV = "cuda:0"
_PAULI = (np.eye(2, dtype=complex), np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]]),
          np.diag([1.0, -1.0]).astype(complex))


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the last step of every run: 199 observables at 5 levels, weighted log-linear fit with its fallback
        {"name": "fit_obs199_l5", "kind": "fit", "levels": 5, "obs": 199},
        # the smallest whole job of a request stream: 8 qubits, bonds of 16, 4 levels
        {"name": "emulate_n8_chi16_l4", "kind": "emulate", "n": 8, "depth": 5, "chi": 16, "levels": 4,
         "dtype": "c64", "noise": 0.02},
        # a validation run: double precision, nothing cut (8 qubits, bonds up to 256)
        {"name": "emulate_n8_chi256_l4_c128", "kind": "emulate", "n": 8, "depth": 8, "chi": 256, "levels": 4,
         "dtype": "c128", "noise": 0.001},
        # an ordinary circuit of a batch: 16 qubits, 7 layers, bonds of 64, 5 levels
        {"name": "emulate_n16_chi64_l5", "kind": "emulate", "n": 16, "depth": 7, "chi": 64, "levels": 5,
         "dtype": "c64", "noise": 0.02},
        # a burst of small jobs to the server
        {"name": "serve_jobs8", "kind": "serve", "jobs": 8, "n": 12, "depth": 6, "chi": 32, "levels": 4,
         "noise": 0.02},
        # saturated layers at an odd length and bond, 5 levels
        {"name": "layers_n15_chi45_l5", "kind": "layers", "n": 15, "chi": 45, "levels": 5, "dtype": "c64", "k": 0,
         "q": 0, "noise": 0.01},
        # saturated layers of the 128-bond workload at its 6 levels
        {"name": "layers_n16_chi128_l6", "kind": "layers", "n": 16, "chi": 128, "levels": 6, "dtype": "c64", "k": 0,
         "q": 0, "noise": 0.01},
        # the double-precision path at a moderate bond
        {"name": "layers_n12_chi64_l2_c128", "kind": "layers", "n": 12, "chi": 64, "levels": 2, "dtype": "c128",
         "k": 0, "q": 0, "noise": 0.01},
        # the flagship: bonds of 512, 8 levels, subspace iteration with 640 columns and 4 power iterations
        {"name": "layers_n16_chi512_l8_k640", "kind": "layers", "n": 16, "chi": 512, "levels": 8, "dtype": "c64",
         "k": 640, "q": 4, "noise": 0.01},
        # observables of a long wide chain at 4 levels
        {"name": "expect_n40_chi512_l4", "kind": "expect", "n": 40, "chi": 512, "levels": 4, "dtype": "c64"},
        # the entropy profile of a moderate chain
        {"name": "entropy_n24_chi128_l4", "kind": "entropy", "n": 24, "chi": 128, "levels": 4, "dtype": "c64"},
        # the two-site product of bonds of 512 at 8 levels through the GEMM entry point
        {"name": "gemm_2048x2048x512_b8", "kind": "gemm", "m": 2048, "nn": 2048, "kk": 512, "batch": 8, "ca": 0,
         "cb": 0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("fit", "emulate", "emulate", "serve", "layers", "layers", "layers", "expect", "entropy", "gemm"))
    if kind == "fit":
        return {"kind": "fit", "levels": rng.randint(4, 16), "obs": _log_int(rng, 8, 1000)}
    if kind == "emulate":
        if rng.random() < 0.25:
            return {"kind": "emulate", "n": rng.randint(4, 8), "depth": rng.randint(4, 8), "chi": 256,
                    "levels": rng.randint(3, 5), "dtype": "c128", "noise": 0.001}
        return {"kind": "emulate", "n": rng.randint(6, 20), "depth": rng.randint(4, 7), "chi": _log_int(rng, 12, 72),
                "levels": rng.randint(3, 8), "dtype": "c64", "noise": 0.02}
    if kind == "serve":
        return {"kind": "serve", "jobs": rng.randint(4, 12), "n": rng.randint(8, 14), "depth": rng.randint(4, 7),
                "chi": _log_int(rng, 12, 40), "levels": rng.randint(3, 6), "noise": 0.02}
    if kind == "layers":
        mode = rng.choice(("exact", "exact", "rsvd", "c128"))
        if mode == "rsvd":
            chi = _log_int(rng, 160, 512)
            return {"kind": "layers", "n": rng.randint(11, 16), "chi": chi, "levels": rng.randint(2, 8), "dtype": "c64",
                    "k": chi + chi // 4, "q": 4, "noise": 0.01}
        if mode == "c128":
            return {"kind": "layers", "n": rng.randint(8, 14), "chi": _log_int(rng, 20, 72),
                    "levels": rng.randint(1, 4), "dtype": "c128", "k": 0, "q": 0, "noise": 0.01}
        return {"kind": "layers", "n": rng.randint(8, 18), "chi": _log_int(rng, 16, 150), "levels": rng.randint(2, 8),
                "dtype": "c64", "k": 0, "q": 0, "noise": 0.01}
    if kind == "expect":
        return {"kind": "expect", "n": rng.randint(10, 48), "chi": _log_int(rng, 32, 512), "levels": rng.randint(1, 5),
                "dtype": "c64"}
    if kind == "entropy":
        return {"kind": "entropy", "n": rng.randint(10, 24), "chi": _log_int(rng, 24, 140),
                "levels": rng.randint(1, 5), "dtype": "c64"}
    return {"kind": "gemm", "m": _log_int(rng, 160, 2048), "nn": _log_int(rng, 96, 2048), "kk": _log_int(rng, 80, 640),
            "batch": rng.randint(1, 8), "ca": rng.randint(0, 1), "cb": rng.randint(0, 1)}


# ---------------------------------------------------------------- inputs
def _haar(rng, count):
    z = (rng.standard_normal((count, 4, 4)) + 1j * rng.standard_normal((count, 4, 4))) / math.sqrt(2.0)
    q, r = np.linalg.qr(z)
    d = np.diagonal(r, axis1=1, axis2=2)
    return q * (d / np.abs(d))[:, None, :]


def _circuit(n, depth, rng):
    layers = [list(range(t % 2, n - 1, 2)) for t in range(depth)]
    return types.SimpleNamespace(n=n, layers=layers, unitaries=[_haar(rng, len(qs)) for qs in layers])


def _levels(case):
    return np.arange(1, case["levels"] + 1, dtype=np.float64)


def _rates(case):
    # depolarizing, amplitude damping and dephasing, scaled per level (no single-qubit depolarizing)
    return _levels(case)[:, None] * case["noise"] * np.array([[1.0, 0.5, 0.5, 0.0]])


def _strings(n):
    """Every Pauli on one site and on two neighbouring sites: the reduced states of all neighbouring pairs."""
    p = np.zeros((12 * n - 9, n), np.uint8)
    for i in range(n):
        for a in range(3):
            p[3 * i + a, i] = a + 1
    for i in range(n - 1):
        for a in range(9):
            p[3 * n + 9 * i + a, i:i + 2] = a // 3 + 1, a % 3 + 1
    return p


def _caps(n, chi):
    return [1] + [min(chi, 4 ** k, 4 ** (n - k)) for k in range(1, n)] + [1]


def _chain(case, seed):
    """Right-canonical site tensors (levels, dl, 4, dr) on the GPU, centre on site 0, norm 1."""
    n, z, caps = case["n"], case["levels"], _caps(case["n"], case["chi"])
    dt = torch.complex64 if case["dtype"] == "c64" else torch.complex128
    gen = torch.Generator(DEV)
    gen.manual_seed(1000003 * int(seed) + 17)
    grade = [torch.exp(-1.5 * torch.arange(d, device=DEV) / d) for d in caps]
    out, carry = [None] * n, None
    for k in range(n - 1, -1, -1):
        dl, dr = caps[k], caps[k + 1]
        m = torch.randn((z, dl, 4, dr), dtype=dt, device=DEV, generator=gen)
        m *= (1.5 / math.sqrt(dl + dr)) * (grade[k][:, None, None] * grade[k + 1])
        m[:, 0, 0, 0] += 0.7
        m[:, 0, 3, 0] += 0.7
        if carry is not None:
            m = torch.matmul(m, carry[:, None])
        if k == 0:
            out[0] = m / torch.linalg.vector_norm(m, dim=(1, 2, 3), keepdim=True)
            break
        q, r = torch.linalg.qr(m.reshape(z, dl, 4 * dr).mH)       # m^H = q r
        out[k] = q.mH.resolve_conj().reshape(z, dl, 4, dr)
        carry = r.mH.resolve_conj()
        carry = carry / torch.linalg.vector_norm(carry, dim=(1, 2), keepdim=True)
    return out


def _state(ctx, case, seed, trunc=nne.TRUNC_EXACT):
    st = nne.State(ctx, case["n"], case["chi"], case["levels"], nne.C64 if case["dtype"] == "c64" else nne.C128, trunc)
    for k, m in enumerate(_chain(case, seed)):
        host = m.cpu().numpy()
        for i in range(case["levels"]):
            st.write_site(i, k, host[i])
    st.set_centre(0)
    return st


def _sketch(case, seed):
    rng = np.random.default_rng(int(seed) + 1234)
    shape = (4 * case["chi"], case["k"])
    return ((rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / math.sqrt(2.0)).astype(np.complex64)


def _fit_table(case, seed):
    """Decaying expectation values with a noise floor: some change sign or never rise above it."""
    rng = np.random.default_rng(int(seed) + 77)
    lam = _levels(case)
    a = rng.uniform(-1, 1, case["obs"]) * 10.0 ** rng.uniform(-6, 0, case["obs"])
    b = rng.uniform(0.02, 0.4, case["obs"])
    y = a[None, :] * np.exp(-np.outer(lam, b)) + 1e-4 * rng.standard_normal((case["levels"], case["obs"]))
    return lam, y, -rng.uniform(0.5, 1.5) * 0.8 ** lam


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng(int(seed))
    s = {"case": case}
    if kind == "gemm":
        m, n, k, z = case["m"], case["nn"], case["kk"], case["batch"]
        gen = torch.Generator(DEV)
        gen.manual_seed(int(seed) + 5)
        s["A"] = torch.randn((z, k, m) if case["ca"] else (z, m, k), dtype=torch.complex64, device=DEV, generator=gen)
        s["B"] = torch.randn((z, n, k) if case["cb"] else (z, k, n), dtype=torch.complex64, device=DEV, generator=gen)
        s["C"] = torch.empty((z, m, n), dtype=torch.complex64, device=DEV)
    s["ctx"] = ctx = nne.Context(0)
    if kind == "fit":
        s["lam"], s["y"], s["lf"] = _fit_table(case, seed)
    elif kind == "emulate":
        s["circuit"], s["rates"], s["paulis"] = _circuit(case["n"], case["depth"], rng), _rates(case), _strings(case["n"])
    elif kind == "serve":
        s["srv"] = nne.Server(0, hbm_budget_bytes=64 << 30, workers=4)
        s["jobs"] = [nne.Job(case["n"], runner.layer_plan(_circuit(case["n"], case["depth"], rng)), _levels(case),
                             _rates(case), case["chi"], _strings(case["n"]), fit_method=nne.FIT_POLY, fit_degree=2)
                     for _ in range(case["jobs"])]
    elif kind == "layers":
        s["st"] = _state(ctx, case, seed, nne.TRUNC_RSVD if case["k"] else nne.TRUNC_EXACT)
        if case["k"]:
            s["st"].set_sketch(_sketch(case, seed), case["q"])
        s["layers"] = runner.build_layer_superops(ctx, _circuit(case["n"], 2, rng), _rates(case))
        s["paulis"] = _strings(case["n"])
    elif kind in ("expect", "entropy"):
        s["st"], s["paulis"] = _state(ctx, case, seed), _strings(case["n"])
    return s


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "fit":
        return ctx.extrapolate(s["lam"], s["y"], s["lf"], method=nne.FIT_EXP_LOGLIN, lambda_star=1.0)
    if kind == "gemm":
        ctx.cgemm(case["ca"], case["cb"], s["A"], s["B"], s["C"])
        return s["C"]
    if kind == "serve":
        tickets = [s["srv"].submit(j) for j in s["jobs"]]
        got = [s["srv"].poll(t) for t in tickets]
        return [{"values": np.float32(r["values"]), "fidelity": np.float32(np.exp(r["log_fid"])),
                 "estimate": np.float32(r["estimate"]), "status": r["status"]} for r in got]
    if kind == "entropy":
        return np.float32(s["st"].entropy())
    single = case["dtype"] == "c64"
    if kind == "emulate":
        st, vals, lf = runner.emulate(ctx, s["circuit"], s["rates"], case["chi"], s["paulis"],
                                      nne.C64 if single else nne.C128)
        est, status = ctx.extrapolate(_levels(case), vals.real, lf, method=nne.FIT_POLY, degree=2, lambda_star=1.0)
        st.close()
        out = (vals, np.exp(lf), est, status)
    else:
        if kind == "layers":
            runner.evolve(s["st"], s["layers"])
        vals, lf = s["st"].expect(s["paulis"])
        out = (vals, np.exp(lf))
    if single:
        out = (np.complex64(out[0]), np.float32(out[1])) + ((np.float32(out[2]), out[3]) if kind == "emulate" else ())
    return out


# ---------------------------------------------------------------- work a pass cannot do without
def _gates(layers):
    """(left bond, middle bond, right bond, rank kept) of every gate, for bond dimensions that start at dims."""
    dims, chi, plan = layers
    for t, qs in enumerate(plan):
        for q in qs if t % 2 == 0 else qs[::-1]:
            r = min(chi, 4 * dims[q], 4 * dims[q + 2])
            yield dims[q], dims[q + 1], dims[q + 2], r
            dims[q + 1] = r


def _circuit_work(case, dims, depth):
    w = 8 if case.get("dtype", "c64") == "c64" else 16
    plan = [list(range(t % 2, case["n"] - 1, 2)) for t in range(depth)]
    by = fl = 0.0
    for dl, dm, dr, r in _gates((dims, case["chi"], plan)):
        rows, cols = 4.0 * dl, 4.0 * dr
        # two sites read, two written; the two-site product, the superoperator, and (where the rank is cut)
        # at least one product that finds the kept subspace and one that projects on it
        by += w * (rows * dm + dm * cols + rows * r + r * cols) + 4096
        fl += 8 * rows * cols * dm + 128 * rows * cols + (16 * rows * cols * r if r < min(rows, cols) else 0)
    site = sum(4.0 * a * b * w for a, b in zip(dims[:-1], dims[1:]))
    return {"bytes": (by + 2 * site) * case["levels"], "flops": (fl + 2 * site) * case["levels"]}


def work(case):
    kind = case["kind"]
    if kind == "fit":
        # every level and observable read, every estimate written; a few exponentials and logarithms per value
        return {"bytes": 8.0 * case["obs"] * (case["levels"] + 2), "flops": 100.0 * case["obs"] * case["levels"]}
    if kind == "gemm":
        m, n, k, z = (float(case[x]) for x in ("m", "nn", "kk", "batch"))
        return {"bytes": 8 * z * (m * k + k * n + m * n), "flops": 8 * z * m * n * k}
    if kind == "emulate":
        return _circuit_work(case, [1] * (case["n"] + 1), case["depth"])
    if kind == "serve":
        w = _circuit_work(case, [1] * (case["n"] + 1), case["depth"])
        return {k: v * case["jobs"] for k, v in w.items()}
    caps = _caps(case["n"], case["chi"])
    if kind == "layers":
        return _circuit_work(case, caps, 2)
    size = sum(4.0 * a * b for a, b in zip(caps[:-1], caps[1:])) * case["levels"]
    if kind == "expect":
        return {"bytes": 8 * size, "flops": 16 * size}
    # the Gram matrix of every bond and its reduction to tridiagonal form, one centre move each
    fl = sum(32.0 * a * b * b + 16.0 / 3.0 * b ** 3 + 32.0 * a * b * b for a, b in zip(caps[:-2], caps[1:-1]))
    return {"bytes": 16 * size, "flops": fl * case["levels"]}


# ---------------------------------------------------------------- the same results in 64 bits
def _superop(ops):
    s = np.zeros((2, 2, 2, 2, 2, 2, 2, 2), complex)       # i1 j1 i2 j2, k1 l1 k2 l2
    for k in ops:
        k4 = np.asarray(k).reshape(2, 2, 2, 2)            # i1 i2 k1 k2
        s += np.einsum("acik,bdjl->abcdijkl", k4, k4.conj())
    return s.reshape(16, 16)


def _noise_superop(rates):
    p, g, d, _ = rates
    pairs = [np.kron(a, b) for a in _PAULI for b in _PAULI]
    depol = [math.sqrt(1 - 15 * p / 16) * pairs[0]] + [math.sqrt(p / 16) * x for x in pairs[1:]]
    damp = [np.diag([1.0, math.sqrt(1 - g)]), np.array([[0, math.sqrt(g)], [0, 0]])]
    phase = [math.sqrt(1 - d) * _PAULI[0], math.sqrt(d) * _PAULI[3]]
    s = _superop(depol)
    for one in (damp, phase):
        s = _superop([np.kron(a, b) for a in one for b in one]) @ s
    return s


def _svd(x):
    try:
        return np.linalg.svd(x, full_matrices=False)
    except np.linalg.LinAlgError:
        w, v = np.linalg.eigh(x.conj().T @ x)
        w, v = np.sqrt(np.maximum(w[::-1], 1e-300)), v[:, ::-1]
        return (x @ v) / w, w, v.conj().T


def _move(sites, centre, target):
    while centre < target:
        a, s, b = sites[centre].shape
        q, r = np.linalg.qr(sites[centre].reshape(a * s, b))
        sites[centre] = q.reshape(a, s, -1)
        sites[centre + 1] = np.tensordot(r, sites[centre + 1], 1)
        centre += 1
    while centre > target:
        a, s, b = sites[centre].shape
        q, r = np.linalg.qr(sites[centre].reshape(a, s * b).conj().T)
        sites[centre] = q.conj().T.reshape(-1, s, b)
        sites[centre - 1] = np.tensordot(sites[centre - 1], r.conj().T, 1)
        centre -= 1
    return centre


def _evolve64(sites, circuit, rates, chi):
    """Every gate, truncated by the SVD of the two-site tensor in mixed canonical form; returns log F."""
    noise, centre, lf = _noise_superop(rates), 0, 0.0
    for t, (qs, us) in enumerate(zip(circuit.layers, circuit.unitaries)):
        right = t % 2 == 0
        for q, u in list(zip(qs, us))[::1 if right else -1]:
            centre = _move(sites, centre, q if right else q + 1)
            th = np.tensordot(sites[q], sites[q + 1], 1)                     # a s1 s2 b
            g = (noise @ _superop([u])).reshape(4, 4, 4, 4)
            th = np.einsum("uvst,astb->auvb", g, th, optimize=True)
            a, b = th.shape[0], th.shape[3]
            x = th.reshape(4 * a, 4 * b)
            r = min(chi, *x.shape)
            if r < min(x.shape):
                p, w, v = _svd(x)
                lf += math.log(np.sum(w[:r] ** 2) / np.sum(w ** 2))
                p, v = (p[:, :r], w[:r, None] * v[:r]) if right else (p[:, :r] * w[:r], v[:r])
            elif right:
                p, v = np.linalg.qr(x)
            else:
                p, v = np.linalg.qr(x.conj().T)
                p, v = v.conj().T, p.conj().T
            sites[q], sites[q + 1] = p.reshape(a, 4, -1), v.reshape(-1, 4, b)
            centre = q + 1 if right else q
            sites[centre] = sites[centre] / np.linalg.norm(sites[centre])
    return lf


def _expect64(sites, paulis):
    n = len(sites)
    vec = [p.T.reshape(4) for p in _PAULI]                                   # v[2 i + j] = P[j][i]
    t = [[np.tensordot(v, m, (0, 1)) for v in vec] for m in sites]
    left, right = [np.ones((1, 1), complex)], [np.ones((1, 1), complex)]
    for k in range(n):
        e = left[-1] @ t[k][0]
        left.append(e / np.abs(e).max())
    for k in range(n - 1, -1, -1):
        e = t[k][0] @ right[-1]
        right.append(e / np.abs(e).max())
    right = right[::-1]
    out = np.zeros(len(paulis), complex)
    for i, codes in enumerate(paulis):
        at = np.flatnonzero(codes)
        e = ref = left[at[0]]
        for k in range(at[0], at[-1] + 1):
            e, ref = e @ t[k][codes[k]], ref @ t[k][0]
        out[i] = (e @ right[at[-1] + 1])[0, 0] / (ref @ right[at[-1] + 1])[0, 0]
    return out


def _product(n):
    m = np.zeros((1, 4, 1), complex)
    m[0, 0, 0] = 1.0
    return [m.copy() for _ in range(n)]


def _poly2(lam, y):
    """Value at lambda = 1 of the least-squares parabola, and the status of a fit made."""
    t = (lam - 1.0) / max(np.abs(lam - 1.0).max(), 1e-300)
    return np.linalg.lstsq(np.stack([t ** 0, t, t * t], 1), y, rcond=None)[0][0]


def _exp3(lam, y):
    """a e^(-b lam) + c at lambda = 1: b on a grid of [-50, 50] / span, then golden section."""
    lim = 50.0 / (lam.max() - lam.min())

    def loss(b):
        e = np.exp(-np.multiply.outer(b, lam))
        de, dy = e - e.mean(-1, keepdims=True), y - y.mean()
        see = (de * de).sum(-1)
        a = np.where(see > 0, (de * dy).sum(-1) / np.where(see > 0, see, 1.0), 0.0)
        c = y.mean() - a * e.mean(-1)
        return np.where(b == 0, 1e300, ((a[..., None] * e + c[..., None] - y) ** 2).sum(-1)), a, c

    grid = np.linspace(-lim, lim, 4001)
    i = int(np.argmin(loss(grid)[0]))
    lo, hi = grid[max(i - 1, 0)], grid[min(i + 1, 4000)]
    g = (math.sqrt(5.0) - 1) / 2
    while hi - lo > 1e-12 * lim:
        x1, x2 = hi - g * (hi - lo), lo + g * (hi - lo)
        lo, hi = (lo, x2) if loss(np.float64(x1))[0] <= loss(np.float64(x2))[0] else (x1, hi)
    b = np.float64(0.5 * (lo + hi))
    _, a, c = loss(b)
    return float(a * math.exp(-b) + c)


def _loglin(lam, y, lf):
    keep = (np.abs(y) >= 1e-10) & (np.sign(y) == (1.0 if y[0] >= 0 else -1.0))
    if keep.sum() < 2:
        return _exp3(lam, y)
    good = [v for v, f in zip(lam, np.exp(lf)) if f > 0.99]
    d = min(good) if good else lam.max() - lam.min()
    w = (4.0 * lf - 40.0 * np.abs(1.0 - lam) / d)[keep]
    w, x, z = np.exp(w - w.max()), lam[keep], np.log(np.abs(y[keep]))
    i, j = np.triu_indices(x.size, 1)
    lp = (4.0 * lf - 40.0 * np.abs(1.0 - lam) / d)[keep]
    lp = lp[i] + lp[j] + 2 * np.log(np.abs(x[i] - x[j]))
    c = np.exp(lp - lp.max())
    slope = np.sum(c * (z[i] - z[j]) / (x[i] - x[j])) / c.sum()
    return math.copysign(math.exp(np.sum(w * (z - slope * x)) / w.sum() + slope), y[0])


def _exact_circuit(case, circuit, rates, start):
    vals, lfs = [], []
    for i in range(case["levels"]):
        sites = start(i)
        lfs.append(_evolve64(sites, circuit, rates[i], case["chi"]))
        vals.append(_expect64(sites, _strings(case["n"])))
    return np.array(vals), np.exp(lfs)


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        s = prepare(case, seed)
        a, b = s["A"].to(torch.complex128), s["B"].to(torch.complex128)
        return torch.matmul(a.mH if case["ca"] else a, b.mH if case["cb"] else b)
    if kind == "fit":
        if case["obs"] > 250:
            return None
        lam, y, lf = _fit_table(case, seed)
        return np.array([_loglin(lam, y[:, o], lf) for o in range(case["obs"])]), None
    # work of one gate's SVD on the host is about 30 (4 chi)^3 multiply-adds
    gates = {"emulate": 1, "serve": case.get("jobs", 1)}.get(kind, 0) * case.get("depth", 0) * case["n"] / 2
    gates = (gates if kind != "layers" else case["n"]) * case["levels"]
    if case["chi"] <= 128 and gates * (4.0 * min(case["chi"], 4 ** (case["n"] // 2 - 1))) ** 3 > 3e9:
        return None
    if kind in ("layers", "emulate", "serve") and case["chi"] > 128 and case["dtype"] == "c64":
        return None
    rng = np.random.default_rng(int(seed))
    if kind in ("emulate", "serve"):
        out = []
        for _ in range(case.get("jobs", 1)):
            vals, fid = _exact_circuit(case, _circuit(case["n"], case["depth"], rng), _rates(case),
                                      lambda i: _product(case["n"]))
            est = _poly2(_levels(case), vals.real)
            out.append((vals, fid, est, None) if kind == "emulate" else
                       {"values": vals.real, "fidelity": fid, "estimate": est, "status": None})
        return out[0] if kind == "emulate" else out
    chain = [m.to(torch.complex128).cpu().numpy() for m in _chain(case, seed)]
    if kind == "layers":
        return _exact_circuit(case, _circuit(case["n"], 2, rng), _rates(case), lambda i: [m[i] for m in chain])
    if kind == "expect":
        vals = np.array([_expect64([m[i] for m in chain], _strings(case["n"])) for i in range(case["levels"])])
        return vals, np.ones(case["levels"])
    ent = np.zeros((case["levels"], case["n"] - 1))
    for i in range(case["levels"]):
        sites = [m[i] for m in chain]
        for k in range(case["n"] - 1):
            w = np.linalg.svd(sites[k].reshape(-1, sites[k].shape[2]), compute_uv=False) ** 2
            w = w[w > 0] / w.sum()
            ent[i, k] = -np.sum(w * np.log(w))
            _move(sites, k, k + 1)
    return ent
