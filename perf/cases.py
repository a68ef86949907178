"""Cases to time: what a program that simulates circuits with this library asks of it.

Every case goes through the package's public entry points (Context, dmrgc_batch_run) with
host buffers in and out, as a user's program calls them.  Inputs are seeded: gates of the random-circuit and
QAOA families of the paper's Sec. V.A on a rows x cols grid, states obtained from a dense statevector of such a
circuit (so their spectra are the ones the sweep meets), uniform bit strings.

Kinds:
  run      a whole open-mode run from |0..0>: create, (apply_layer, sweep) per layer; the partial fidelity after
           every update, and, where the bond dimension holds every state of the circuit, all amplitudes.
  step     one compression step of a resumed run: load a state (a checkpoint), apply_layer, sweep.  The tensors of
           the new state are defined up to a unitary on every bond, so what is returned is what the step
           defines: the partial fidelity after every update.
  grouped  one step of the single-site variant over grouped qubits from its seeded random guess.
  batch    independent instances on worker streams.
  amplitude, sample   read-outs of a loaded state.

A heavily truncated step at 54 qubits has no value to compare: there the sweep amplifies rounding (two precisions
differ by 1e-3 in f), so the saturated updates of the benchmark stand here at 24 qubits, at its bond dimension.
The complex64 modes store single precision, so their results are returned in single precision.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2207_05612_gb300 as dm
from paper_2207_05612_gb300 import binding

PRECISION = {"fp64": binding.DMRGC_FP64, "bf16x3": binding.DMRGC_BF16X3, "tf32x3": binding.DMRGC_TF32X3,
             "fp32": binding.DMRGC_FP32}
DEVICE = torch.device("cuda")


def listed():
    return [
        # one amplitude of a small state: the smallest call there is, one site after the other
        {"name": "amplitude_1_4x6", "kind": "amplitude", "rows": 4, "cols": 6, "chi": 128, "precision": "bf16x3", "count": 1},
        # the exact FP64 run of 12 qubits, chi = 64 (small matrices, launches and host round trips), all amplitudes read
        {"name": "run_3x4_fp64", "kind": "run", "rows": 3, "cols": 4, "chi": 64, "cycles": 8, "family": "random", "precision": "fp64"},
        # an exact FP64 QAOA run, odd grid: rank-2 gates, strongly graded spectra
        {"name": "run_qaoa_3x5_fp64", "kind": "run", "rows": 3, "cols": 5, "chi": 128, "cycles": 4, "family": "qaoa", "precision": "fp64"},
        # the first layers of the 54-qubit run, bonds still growing: many small truncated SVDs and the layer MPOs
        {"name": "run_6x9_chi256_tf32x3", "kind": "run", "rows": 6, "cols": 9, "chi": 256, "cycles": 4, "family": "random", "precision": "tf32x3"},
        # one step resumed from a checkpoint, a small odd bond dimension
        {"name": "step_4x5_chi100_tf32x3", "kind": "step", "rows": 4, "cols": 5, "chi": 100, "cycles": 8, "family": "random", "precision": "tf32x3", "compress": 0},
        # one step at a bond dimension that just begins to truncate
        {"name": "step_4x5_chi512_bf16x3", "kind": "step", "rows": 4, "cols": 5, "chi": 512, "cycles": 8, "family": "random", "precision": "bf16x3", "compress": 1},
        # one step of the 24-qubit run at the benchmark's bond dimension and precision: saturated two-site updates
        {"name": "step_4x6_chi512_bf16x3", "kind": "step", "rows": 4, "cols": 6, "chi": 512, "cycles": 8, "family": "random", "precision": "bf16x3", "compress": 1},
        # independent instances on worker streams
        {"name": "batch_8_tf32x3", "kind": "batch", "count": 8, "workers": 8, "chi": 64, "cycles": 8, "precision": "tf32x3"},
        # one step of the single-site variant, a column of the grid per tensor
        {"name": "grouped_4x5_chi24_fp64", "kind": "grouped", "rows": 4, "cols": 5, "chi": 24, "cycles": 6, "family": "random", "precision": "fp64"},
        # read-outs of a 54-qubit state: amplitudes of many strings, samples
        {"name": "amplitude_6x9_chi512_bf16x3", "kind": "amplitude", "rows": 6, "cols": 9, "chi": 512, "precision": "bf16x3", "count": 16384},
        {"name": "sample_6x9_chi256_tf32x3", "kind": "sample", "rows": 6, "cols": 9, "chi": 256, "precision": "tf32x3", "count": 4096},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 8 + ["run"] * 4 + ["batch", "grouped"] * 2 + ["amplitude"] * 2 + ["sample"])
    if kind == "step":
        rows, cols = rng.choice([(4, 4), (3, 6), (2, 9), (4, 5), (3, 7), (4, 6)])
        precision = rng.choice(["bf16x3", "bf16x3", "tf32x3", "tf32x3", "fp32"])
        low = 200 if precision == "bf16x3" else 48
        return {"kind": kind, "rows": rows, "cols": cols, "chi": log(low, max(low + 1, min(512, 2 ** (rows * cols // 2)))),
                "cycles": rng.choice([6, 8]), "family": "random", "precision": precision, "compress": rng.randint(0, 1)}
    if kind == "run" and rng.random() < 0.5:
        rows, cols = rng.choice([(2, 5), (3, 4), (2, 7), (3, 5)])
        return {"kind": kind, "rows": rows, "cols": cols, "chi": 2 ** (rows * cols // 2) + rng.randint(0, 9),
                "cycles": rng.choice([4, 6]), "family": rng.choice(["random", "qaoa"]), "precision": "fp64"}
    if kind == "run":
        rows, cols = rng.choice([(5, 5), (5, 6), (6, 6), (6, 7), (6, 9)])
        return {"kind": kind, "rows": rows, "cols": cols, "chi": log(64, 256), "cycles": 4, "family": "random", "precision": "tf32x3"}
    if kind == "batch":
        return {"kind": kind, "count": rng.randint(3, 8), "workers": rng.randint(2, 8), "chi": log(32, 64), "cycles": rng.choice([6, 8]),
                "precision": "tf32x3"}
    if kind == "grouped":
        rows, cols = rng.choice([(2, 6), (3, 5), (4, 4), (4, 5)])
        return {"kind": kind, "rows": rows, "cols": cols, "chi": log(6, 40), "cycles": rng.choice([4, 6]), "family": "random", "precision": "fp64"}
    rows, cols = rng.choice([(4, 5), (5, 5), (5, 7), (6, 9)])
    if kind == "sample":
        return {"kind": kind, "rows": rows, "cols": cols, "chi": log(50, 256), "precision": "tf32x3", "count": log(200, 4096)}
    precision = rng.choice(["bf16x3", "tf32x3", "fp32", "fp64"])
    return {"kind": kind, "rows": rows, "cols": cols, "chi": log(50, 100 if precision == "fp64" else 512), "precision": precision,
            "count": log(1, 2000 if precision == "fp64" else 16384)}


# ---------------------------------------------------------------- circuits

def _gates_random(rows, cols, first_cycle, cycles, rng):
    """Cycles of the Sycamore-like family: sqrt(X|Y|W) on every qubit, then fSim(pi/2, pi/6) on one coupler
    pattern of ABCDCDAB."""
    x, y = np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]], complex)
    one = [(np.eye(2) - 1j * p) / math.sqrt(2) for p in (x, y, (x + y) / math.sqrt(2))]
    two = np.eye(4, dtype=complex)
    two[1:3, 1:3] = [[0, -1j], [-1j, 0]]
    two[3, 3] = np.exp(-1j * math.pi / 6)
    prev, out = [-1] * (rows * cols), []
    for cyc in range(first_cycle, first_cycle + cycles):
        for q in range(rows * cols):
            prev[q] = int(rng.choice([k for k in range(3) if k != prev[q]]))
            out.append((q, -1, one[prev[q]]))
        pat = "ABCDCDAB"[cyc % 8]
        for r in range(rows):
            for c in range(cols):
                if (r + c) % 2 != (pat in "CD"):
                    continue
                if pat in "AC" and c + 1 < cols:
                    out.append((r * cols + c, r * cols + c + 1, two))
                if pat in "BD" and r + 1 < rows:
                    out.append((r * cols + c, (r + 1) * cols + c, two))
    return out


def _gates_qaoa(rows, cols, level, rng):
    """One QAOA level on the grid graph: exp(-i gamma Z Z) on every edge, exp(-i beta X) on every qubit."""
    ga, be = rng.uniform(0, math.pi), rng.uniform(0, math.pi / 2)
    out = []
    if level == 0:
        out += [(q, -1, np.array([[1, 1], [1, -1]], complex) / math.sqrt(2)) for q in range(rows * cols)]
    e = np.exp(-1j * ga)
    zz = np.diag([e, e.conjugate(), e.conjugate(), e])
    for r in range(rows):
        for c in range(cols):
            if c + 1 < cols:
                out.append((r * cols + c, r * cols + c + 1, zz))
            if r + 1 < rows:
                out.append((r * cols + c, (r + 1) * cols + c, zz))
    xr = np.array([[math.cos(be), -1j * math.sin(be)], [-1j * math.sin(be), math.cos(be)]])
    return out + [(q, -1, xr) for q in range(rows * cols)]


def _layers(case, seed, cycles, extra=0):
    """Layers of two cycles (or of one QAOA level) covering `cycles` cycles and `extra` more layers."""
    rng = np.random.default_rng(seed)
    if case["family"] == "qaoa":
        return [_gates_qaoa(case["rows"], case["cols"], k, rng) for k in range(cycles // 2 + extra)]
    return [_gates_random(case["rows"], case["cols"], 2 * k, 2, rng) for k in range(cycles // 2 + extra)]


def _statevector(n, layers, dtype):
    """Dense state of the circuit from |0..0>, axis q = qubit q."""
    psi = torch.zeros((2,) * n, dtype=dtype, device=DEVICE)
    psi[(0,) * n] = 1
    for q0, q1, u in (g for layer in layers for g in layer):
        qs = [q0] if q1 < 0 else [q0, q1]
        k = len(qs)
        g = torch.from_numpy(np.ascontiguousarray(u, dtype=np.complex128)).to(DEVICE, dtype).reshape((2,) * (2 * k))
        psi = torch.movedim(torch.tensordot(g, psi, dims=(list(range(k, 2 * k)), qs)), list(range(k)), qs)
    return psi


def _snake(rows, cols):
    return [(r if c % 2 == 0 else rows - 1 - r) * cols + c for c in range(cols) for r in range(rows)]


def _mps_of(psi, rows, cols, chi, group=1):
    """Mixed-canonical MPS (centre on tensor nt // 2 of nt, bonds <= chi) of a dense state, along the column snake,
    `group` sites per tensor."""
    p = 2 ** group
    nt = rows * cols // group
    m = nt // 2
    t = psi.permute(_snake(rows, cols)).reshape(1, -1).to(torch.complex128)

    def split(mat):   # rows of mat: the kept left singular vectors and the rest
        h = mat @ mat.mH
        lam, u = torch.linalg.eigh(h)
        k = max(1, min(chi, int((lam > 1e-12 * lam[-1]).sum())))
        u = u[:, -k:].flip(1)
        return u, u.mH @ mat

    left, right = [], []
    for _ in range(m):
        u, rest = split(t.reshape(t.shape[0] * p, -1))
        left.append(u.reshape(-1, p, u.shape[1]))
        t = rest
    cl = t.shape[0]
    t = t.reshape(-1, 1)
    for _ in range(nt - 1 - m):
        cr = t.shape[1]
        mat = t.reshape(-1, p * cr)
        u, rest = split(mat.mT)
        right.append(u.mT.reshape(-1, p, cr))
        t = rest.mT
    c = t.reshape(cl, p, -1)
    mps = left + [c / torch.linalg.norm(c)] + right[::-1]
    return [a.cpu().numpy() for a in mps]


def _single(case, v):
    v = np.asarray(v)
    if case["precision"] == "fp64":
        return v
    return v.astype(np.complex64 if v.dtype.kind == "c" else np.float32)


def _holds(case):
    """Whether a run's bond dimension holds every state of the circuit."""
    return case["chi"] >= 2 ** (case["rows"] * case["cols"] // 2)


def _all_bits(n):
    return ((np.arange(2 ** n)[:, None] >> (n - 1 - np.arange(n))) & 1).astype(np.uint8)


# ---------------------------------------------------------------- prepare / run

def _context(case, **more):
    return dm.Context(case["rows"], case["cols"], case["chi"], precision=PRECISION[case["precision"]], **more)


def _random_state(case, seed):
    """Random right-canonical MPS, bonds min(2^i, 2^(n-i), chi), entries of the storage precision."""
    g = torch.Generator(device=DEVICE).manual_seed(seed)
    n, chi = case["rows"] * case["cols"], case["chi"]
    dtype = torch.complex128 if case["precision"] == "fp64" else torch.complex64
    bond = [min(2 ** i, 2 ** (n - i), chi) for i in range(n + 1)]
    mps = []
    for i in range(n):
        z = torch.randn(2 * bond[i + 1], bond[i], dtype=torch.complex64, device=DEVICE, generator=g)
        q = torch.linalg.qr(z.to(dtype))[0] if i else z.to(dtype) / torch.linalg.norm(z)
        mps.append(q.mH.reshape(bond[i], 2, bond[i + 1]).contiguous())
    return mps


def prepare(case, seed):
    kind = case["kind"]
    rng = np.random.default_rng([seed, 7])
    if kind == "run":
        return {"case": case, "layers": _layers(case, seed, case["cycles"]), "bits": _all_bits(case["rows"] * case["cols"]) if _holds(case) else None}
    if kind in ("step", "grouped"):
        layers = _layers(case, seed, case["cycles"], 1)
        n = case["rows"] * case["cols"]
        group = case["rows"] if kind == "grouped" else 1   # one column of the grid per tensor
        mps = _mps_of(_statevector(n, layers[:-1], torch.complex64), case["rows"], case["cols"], case["chi"], group)
        more = {"groups": [group] * (n // group)} if kind == "grouped" else {"mpo_compress": case["compress"]}
        return {"case": case, "ctx": _context(case, **more), "mps": mps, "layer": layers[-1]}
    if kind == "batch":
        # instances of uneven size, depth and bond dimension
        todo = []
        for k in range(case["count"]):
            rows, cols = ((4, 4), (3, 5), (4, 5))[int(rng.integers(3))]
            c = {"rows": rows, "cols": cols, "family": "random"}
            chi = int(case["chi"] * (1 + k % 2))
            todo.append((rows, cols, chi, _layers(c, int(rng.integers(1 << 30)), case["cycles"] + 2 * (k % 2)), 2))
        return {"case": case, "todo": todo}
    if kind in ("amplitude", "sample"):
        ctx = _context(case)
        ctx.set_mps([a.cpu().numpy() for a in _random_state(case, seed)])
        return {"case": case, "ctx": ctx, "seed": seed, "bits": _read_bits(case, seed)}
    raise ValueError(kind)


def _read_bits(case, seed):
    return np.random.default_rng([seed, 7]).integers(0, 2, size=(case["count"], case["rows"] * case["cols"]), dtype=np.uint8)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "run":
        ctx = _context(case)
        f = []
        for layer in state["layers"]:
            ctx.apply_layer(layer)
            ctx.sweep(2)
            f += ctx.history()
        out = {"f": _single(case, f)}
        if state["bits"] is not None:
            out["amplitudes"] = _single(case, ctx.amplitude(state["bits"]))
        ctx.close()
        return out
    if kind in ("step", "grouped"):
        ctx = state["ctx"]
        ctx.set_mps(state["mps"])
        ctx.apply_layer(state["layer"])
        ctx.sweep(2 if kind == "step" else 4)
        return {"f": _single(case, ctx.history())}
    if kind == "batch":
        items, keep = binding.pack_batch(state["todo"])
        opt = binding.dmrgc_default_options()
        opt.precision = PRECISION[case["precision"]]
        binding.dmrgc_batch_run(items, case["count"], case["workers"], opt)
        return {"F": _single(case, np.exp([it.log_F_tilde for it in items])),
                "updates": np.array([it.updates for it in items])}
    if kind == "amplitude":
        return _single(case, state["ctx"].amplitude(state["bits"]))
    if kind == "sample":
        return state["ctx"].sample(case["count"], state["seed"])
    raise ValueError(kind)


# ---------------------------------------------------------------- work / exact

def _bonds(case):
    n = case["rows"] * case["cols"]
    return [min(2 ** i, 2 ** (n - i), case["chi"]) for i in range(n + 1)]


def _site_values(case):
    b = _bonds(case)
    return sum(2 * b[i] * b[i + 1] for i in range(len(b) - 1))


def _step_work(case, itemsize):
    """One compression step: per two-site update the contraction with the layer operator, theta, its truncated SVD
    through one Gram matrix and the new environment; the old state read, the new one written."""
    n, b = case["rows"] * case["cols"], _bonds(case)
    where = {q: i for i, q in enumerate(_snake(case["rows"], case["cols"]))}
    rng = np.random.default_rng(0)
    gates = (_gates_qaoa if case["family"] == "qaoa" else _gates_random)(
        case["rows"], case["cols"], *((0, rng) if case["family"] == "qaoa" else (case["cycles"], 2, rng)))
    rank = 2 if case["family"] == "qaoa" else 4
    d = [1] * (n + 1)
    for cut in range(1, n):
        for q0, q1, _ in gates:
            if q1 >= 0 and (where[q0] < cut) != (where[q1] < cut):
                d[cut] = min(d[cut] * rank, 4 ** min(cut, n - cut), 256)
    flops = 0.0
    for i in range(n - 1):
        a, c, m, k = b[i], b[i + 2], b[i + 1], min(2 * b[i], 2 * b[i + 2])
        one = 2 * a * b[i] * d[i] * m + 4 * a * m * d[i] * d[i + 1]      # X (Y alike)
        one += 4 * a * c * d[i + 1] * m + 2 * a * m * d[i + 1] * m       # theta, environment
        one += k * k * 2 * max(a, c) + k ** 3 // 2 + m * 4 * a * c       # truncated SVD, the other tensor
        flops += 2 * 8.0 * one                                           # two updates per bond
    return {"bytes": 2.0 * itemsize * _site_values(case), "flops": flops}


def work(case):
    kind = case["kind"]
    item = 16 if case["precision"] == "fp64" else 8
    if kind == "run":
        one = _step_work(case, item)
        return {k: v * case["cycles"] / 2 for k, v in one.items()}
    if kind == "step":
        return _step_work(case, item)
    if kind == "batch":
        one = _step_work({"rows": 4, "cols": 4, "chi": int(1.5 * case["chi"]), "cycles": 2, "family": "random"}, item)
        return {k: v * case["count"] * (case["cycles"] + 1) / 2 for k, v in one.items()}
    if kind == "grouped":
        # per tensor and sweep: L B, the layer operator site by site, F and the environment
        chi, p, nt = case["chi"], 2 ** case["rows"], case["cols"]
        return {"bytes": 2.0 * item * nt * chi * p * chi, "flops": 4 * nt * 8.0 * (3 * p * 4 * chi ** 3 + case["rows"] * 32 * p * chi ** 2)}
    if kind in ("amplitude", "sample"):
        values = _site_values(case)
        n = case["rows"] * case["cols"]
        return {"bytes": float(item * values + case["count"] * (n + 16)), "flops": 8.0 * case["count"] * values / (2 if kind == "amplitude" else 1)}
    raise ValueError(kind)


def exact(case, seed):
    kind = case["kind"]
    if kind == "run" and _holds(case):
        layers = _layers(case, seed, case["cycles"])
        n = case["rows"] * case["cols"]
        psi = _statevector(n, layers, torch.complex128).reshape(-1).cpu().numpy()
        return {"f": np.ones(2 * (n - 1) * len(layers)), "amplitudes": psi}
    if kind == "amplitude":
        bits = _read_bits(case, seed)
        order = _snake(case["rows"], case["cols"])
        mps = [a.to(torch.complex128) for a in _random_state(case, seed)]
        out = []
        for part in np.array_split(bits, -(-len(bits) // 4096)):
            x = torch.from_numpy(part).to(DEVICE).long()
            v = torch.ones(len(part), 1, dtype=torch.complex128, device=DEVICE)
            for q, a in zip(order, mps):
                v = torch.where(x[:, q, None] == 1, v @ a[:, 1], v @ a[:, 0])
            out.append(v[:, 0])
        return torch.cat(out).cpu().numpy()
    return None
