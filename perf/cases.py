"""Performance cases of the fused-gate state-vector simulator.

Each case is one piece of work that a program using the package has it do, through the public
bindings: running a fused circuit on a state, a batch of small circuits, Pauli expectation values,
importing / sampling / exporting a state.  ``listed`` names the cases, ``draw`` makes further ones of
the same ranges, ``prepare`` makes what a program holds before the call, ``run`` is one pass,
``work`` what a pass cannot do without, ``exact`` the same result in 64 bits from plain torch.

States are returned as they lie in their buffers: blocks of 32 amplitudes, 32 real parts then 32
imaginary parts (the documented device layout).
"""
import math
import os

import numpy as np
import torch

import paper_2602_09604_gb300
from paper_2602_09604_gb300 import binding as B
from paper_2602_09604_gb300 import workloads as wl
from paper_2602_09604_gb300.batch import Batch
from paper_2602_09604_gb300.state import DeviceState

COST_MODEL = os.path.join(os.path.dirname(paper_2602_09604_gb300.__file__), "cost_model_gb300.bin")
PRECISION = {"fp32": B.PREC_FP32, "tf32": B.PREC_TF32, "bf16x3": B.PREC_BF16X3}

# the batch options that the batch autotuner starts from (circuits kept unfused, staged tiles of
# 14 local qubits with register phases); a program that runs one batch many times keeps them
BATCH_OPTS = {"threads": 512, "smem_max_n": 0, "split_min_n": 8, "tile_log2": 12, "wave_mb": 48, "stage_log2": 14,
              "stage_k": 2, "stage_layers": 1, "ctas_per_sm": 1}


def listed():
    return [
        # the smallest circuit: 4x4 grid, 14 cycles, gates fused to two qubits; a few microseconds
        # of work per gate, so launches and latency count
        {"name": "grid16_k2", "kind": "circuit", "circuit": "grid", "n": 16, "depth": 14, "fuse": "greedy", "max_k": 2,
         "precision": "fp32", "start": "init"},
        # a circuit seen for the first time (quantum volume, 18 qubits): fused with the default
        # options, started and applied, and its plan freed, as a program with new gates each time does
        {"name": "qv18_new", "kind": "circuit", "circuit": "qv", "n": 18, "depth": 18, "fuse": "greedy", "max_k": 4,
         "precision": "fp32", "start": "lazy", "fresh": True},
        # a mid-size circuit in plain fp32 (256 MB of state), fusion size 3 as in the paper's runs
        {"name": "grid25_k3", "kind": "circuit", "circuit": "grid", "n": 25, "depth": 20, "fuse": "greedy", "max_k": 3,
         "precision": "fp32", "start": "init"},
        # the default options (greedy, at most four qubits, fp32) on a 2 GiB state
        {"name": "grid28_k4", "kind": "circuit", "circuit": "grid", "n": 28, "depth": 20, "fuse": "greedy", "max_k": 4,
         "precision": "fp32", "start": "init"},
        # tensor-core fusion at a size that stays near the L2 cache
        {"name": "grid24_k6_bf16x3", "kind": "circuit", "circuit": "grid", "n": 24, "depth": 20, "fuse": "greedy",
         "max_k": 6, "precision": "bf16x3", "start": "init"},
        # the fast mode (tf32 products) with five-qubit gates
        {"name": "grid28_k5_tf32", "kind": "circuit", "circuit": "grid", "n": 28, "depth": 20, "fuse": "greedy",
         "max_k": 5, "precision": "tf32", "start": "init"},
        # the headline circuit: 5x6 grid, 20 cycles, learned fusion, split-bf16 tensor cores, lazy start
        {"name": "grid30_learned", "kind": "circuit", "circuit": "grid", "n": 30, "depth": 20, "fuse": "learned",
         "max_k": 6, "precision": "bf16x3", "start": "lazy"},
        # the 30-qubit QFT of a basis state: post-phase gates and the swap network
        {"name": "qft30_learned", "kind": "circuit", "circuit": "qft", "n": 30, "depth": 1, "fuse": "learned",
         "max_k": 6, "precision": "bf16x3", "start": "init"},
        # Grover rounds on an odd size: many-control gates between dense layers
        {"name": "grover23_k4", "kind": "circuit", "circuit": "grover", "n": 23, "depth": 3, "fuse": "greedy", "max_k": 4,
         "precision": "fp32", "start": "init"},
        # a double-precision reference run
        {"name": "grid24_c128_k3", "kind": "circuit", "circuit": "grid", "n": 24, "depth": 14, "fuse": "greedy",
         "max_k": 3, "precision": "c128", "start": "init"},
        # 256 uneven hardware-efficient-ansatz circuits in one launch
        {"name": "hea256", "kind": "batch", "count": 256, "n_lo": 10, "n_hi": 20, "layers": 8},
        # the energy of a nearest-neighbour chain (XX, YY, ZZ couplings and a Z field) in a
        # variational state, then the state's readout: both read a state that is there
        {"name": "energy26_readout", "kind": "readout", "n": 26, "terms": "xyz", "samples": 1024},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("fp32", "fp32", "tensor", "learned", "qft", "grover", "new", "c128", "batch", "readout", "readout"))
    c = {"kind": "circuit", "fuse": "greedy", "precision": "fp32", "start": rng.choice(("init", "lazy"))}
    if kind == "fp32":
        c.update(circuit=rng.choice(("grid", "grid", "qv")), n=rng.randint(10, 27), depth=rng.randint(8, 20), max_k=rng.randint(2, 6))
        if c["circuit"] == "qv":
            c["depth"] = min(c["depth"], 10)
        if c["n"] > 25:
            c["depth"] = min(c["depth"], 14)
    elif kind == "tensor":
        c.update(circuit="grid", n=rng.randint(14, 28), depth=rng.randint(8, 20), max_k=rng.randint(4, 6),
                 precision=rng.choice(("tf32", "bf16x3", "bf16x3")))
    elif kind == "learned":
        c.update(circuit="grid", n=rng.randint(16, 29), depth=rng.randint(8, 20), max_k=6, fuse="learned", precision="bf16x3")
    elif kind == "qft":
        c.update(circuit="qft", n=rng.randint(12, 30), depth=1, max_k=6, fuse="learned", precision="bf16x3", start="init")
    elif kind == "grover":
        c.update(circuit="grover", n=rng.randint(10, 26), depth=rng.randint(1, 4), max_k=rng.randint(3, 5))
    elif kind == "new":
        c.update(circuit=rng.choice(("qv", "grid")), n=rng.randint(7, 20), depth=rng.randint(6, 16), max_k=rng.randint(3, 5),
                 fresh=True)
    elif kind == "c128":
        c.update(circuit="grid", n=rng.randint(10, 23), depth=rng.randint(6, 14), max_k=rng.randint(1, 4), precision="c128")
    elif kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 12, 240), "n_lo": rng.randint(8, 12), "n_hi": rng.randint(14, 20),
                "layers": rng.randint(4, 8)}
    else:
        return {"kind": "readout", "n": rng.randint(16, 28), "terms": rng.choice(("xyz", "x_zz", "z")),
                "samples": _log_int(rng, 1, 4096)}
    return c


# --------------------------------------------------------------------------------------- inputs
def _grid(n):
    """The most square grid that holds n sites, the surplus dropped from the end of the last row."""
    rows = max(2, int(math.isqrt(n)))
    cols = -(-n // rows)
    full = rows * cols
    return wl.Grid(rows, cols, dropped=tuple((rows - 1, cols - 1 - i) for i in range(full - n)))


def _gates(case, seed):
    """(gates, basis index the circuit starts from)"""
    n, kind = case["n"], case["circuit"]
    if kind == "grid":
        return wl.random_grid_circuit(_grid(n), case["depth"], seed=seed), 0
    if kind == "qv":
        return wl.qv_circuit(n, case["depth"], seed=seed), 0
    if kind == "qft":
        return wl.qft_circuit(n), wl.qft_basis_index(n, seed)
    marked = int(np.random.default_rng(seed).integers(0, 1 << n))
    return wl.grover_circuit(n, marked, case["depth"]), 0


def _batch(case, seed):
    """The batch's circuits: uneven sizes that belong to the case, angles from the seed."""
    ns = np.random.default_rng(5).integers(case["n_lo"], case["n_hi"] + 1, size=case["count"])
    rng = np.random.default_rng(seed)
    return [(int(n), wl.hea_circuit(int(n), case["layers"], rng)) for n in ns]


def _ansatz_state(n, seed, device):
    """Amplitudes (complex64) as an ansatz leaves them: single-qubit rotations by seeded angles and a
    sign per neighbouring pair of ones, then a random part in every amplitude (an entangled state's
    follow no product form).  Pauli terms on it are of order one."""
    rng = np.random.default_rng(seed)
    th, ph = rng.normal(1.45, 0.25, n), rng.uniform(0, 2 * math.pi, n)
    psi = torch.ones(1, dtype=torch.complex128, device=device)
    for q in range(n):
        lo, hi = psi * math.cos(th[q] / 2), psi * (np.exp(1j * ph[q]) * math.sin(th[q] / 2))
        if q:
            hi[hi.numel() // 2:] *= -1.0   # CZ(q - 1, q)
        psi = torch.cat((lo, hi))
    gen = torch.Generator(device=device).manual_seed(seed)
    psi *= 1 + 0.3 * torch.randn(psi.shape, dtype=torch.complex128, device=device, generator=gen)
    return (psi / torch.linalg.vector_norm(psi)).to(torch.complex64)


def _strings(case):
    """(x_masks, z_masks) of a nearest-neighbour chain's terms."""
    n, xs, zs = case["n"], [], []
    for q in range(n - 1):
        pair = 3 << q
        if case["terms"] == "xyz":
            xs += [pair, pair]
            zs += [0, pair]
        xs.append(0)
        zs.append(pair)
    for q in range(n):
        xs.append(1 << q if case["terms"] == "x_zz" else 0)
        zs.append(0 if case["terms"] == "x_zz" else 1 << q)
    return np.array(xs, dtype=np.uint64), np.array(zs, dtype=np.uint64)


class _Kept:
    """A fused circuit or batch that is freed with the state that holds it."""

    def __init__(self, obj, free):
        self.obj, self._free = obj, free

    def __del__(self):
        self._free(self.obj)


def _fuse(case, gates):
    kw = dict(max_k=case["max_k"])
    if case["precision"] in ("tf32", "bf16x3"):
        kw.update(precision=PRECISION[case["precision"]], tc_min_k=4)
    if case["fuse"] != "learned":
        return B.sv_fuse_circuit(gates, case["n"], **kw)
    model = B.sv_mlp_load(COST_MODEL)
    try:
        start = 28 if case["start"] == "lazy" else 0
        return B.sv_fuse_circuit(gates, case["n"], mode=B.FUSE_LEARNED, model=model, start_qubits=start, **kw)
    finally:
        B.sv_mlp_free(model)


def prepare(case, seed):
    if case["kind"] == "circuit":
        gates, basis = _gates(case, seed)
        st = DeviceState(case["n"], c128=case["precision"] == "c128")
        fused = None if case.get("fresh") else _Kept(_fuse(case, gates), B.sv_fused_free)
        return {"case": case, "gates": gates, "basis": basis, "st": st, "fused": fused}
    if case["kind"] == "batch":
        b = Batch(_batch(case, seed), 0)
        b.set(ctas=torch.cuda.get_device_properties(0).multi_processor_count, **BATCH_OPTS)
        return {"case": case, "batch": _Kept(b, Batch.free)}
    amps = _ansatz_state(case["n"], seed, "cuda")
    xs, zs = _strings(case)
    uniforms = np.random.default_rng(seed + 1).random(case["samples"])
    return {"case": case, "amps": amps, "out": torch.empty_like(amps), "st": DeviceState(case["n"]), "xs": xs, "zs": zs,
            "uniforms": uniforms}


# ----------------------------------------------------------------------------------------- pass
def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"].obj
        b.run()
        return b.arena
    st = state["st"]
    if case["kind"] == "readout":
        # a state made elsewhere on the device is imported, measured, sampled and handed back
        B.sv_load(st.h, state["amps"].data_ptr(), False)
        energy = B.sv_expval_pauli(st.h, state["xs"], state["zs"])
        samples, norm = B.sv_sample_norm(st.h, state["uniforms"])
        B.sv_store(st.h, state["out"].data_ptr(), False)
        return {"terms": energy, "samples": samples.view(np.int64), "norm": norm, "amps": state["out"]}
    fused = _fuse(case, state["gates"]) if state["fused"] is None else state["fused"].obj
    if case["start"] == "lazy":
        B.sv_init_apply(st.h, state["basis"], fused)
    else:
        st.init(state["basis"])
        st.apply(fused)
    if state["fused"] is None:
        B.sv_fused_free(fused)
    return st.buf


# ----------------------------------------------------------------------------------------- work
def _gate_flops(g):
    """Flops per amplitude of the whole state that gate g needs by itself (its zeros left out)."""
    m = np.asarray(g.matrix)
    k, off = len(g.targets), m[~np.eye(len(m), dtype=bool)]
    if not off.any():
        each = 6.0 * np.count_nonzero(np.abs(np.diag(m) - 1) > 0) / len(m)
    else:
        per_row = np.count_nonzero(m, axis=1)
        each = float(np.mean(np.where(per_row > 1, 8.0 * per_row - 2, 6.0)))
    return each / 2 ** len(g.controls)


def work(case):
    if case["kind"] == "batch":
        ns = np.array([float(n) for n, _ in _batch(dict(case, layers=0), 0)])
        amps = 2.0 ** ns
        # RZ: 6 flops an amplitude, RY (real): 6, CZ: a sign
        return {"bytes": float((8 * amps).sum()), "flops": float((amps * case["layers"] * (12 * ns + ns)).sum())}
    n = case["n"]
    amps = 2.0 ** n
    if case["kind"] == "readout":
        # read the given amplitudes, write them back out; 4 flops a term and amplitude
        return {"bytes": 16 * amps, "flops": amps * (4.0 * len(_strings(case)[0]) + 4)}
    per_amp = 16 if case["precision"] == "c128" else 8
    gates, _ = _gates(case, 5)
    return {"bytes": per_amp * amps, "flops": float(amps * sum(_gate_flops(g) for g in gates))}


# ---------------------------------------------------------------------------------------- exact
def _apply64(psi, n, g):
    """psi (complex128, bit q <-> qubit q) under one gate, in place."""
    kind = {q: "t" for q in g.targets}
    kind.update({q: "c" for q in g.controls})
    shape, idx, tdim = [], [], {}
    q = n - 1
    while q >= 0:   # dimensions from the top qubit down: runs of free or control qubits, single targets
        kd, lo = kind.get(q, "f"), q
        if kd != "t":
            while lo > 0 and kind.get(lo - 1, "f") == kd:
                lo -= 1
        size = 1 << (q - lo + 1)
        if kd == "t":
            tdim[q] = len(shape)
        shape.append(size)
        idx.append(size - 1 if kd == "c" else slice(None))
        q = lo - 1
    v = psi.view(shape)

    def part(j):
        at = list(idx)
        for b, t in enumerate(g.targets):
            at[tdim[t]] = (j >> b) & 1
        return v[tuple(at)]

    u = np.asarray(g.matrix, dtype=np.complex128)
    d = len(u)
    if not u[~np.eye(d, dtype=bool)].any():
        for j in range(d):
            if u[j, j] != 1:
                part(j).mul_(complex(u[j, j]))
        return
    used = [j for j in range(d) if np.count_nonzero(u[j]) != 1 or np.count_nonzero(u[:, j]) != 1 or u[j, j] == 0]
    x = {j: part(j).clone() for j in used}
    for r in range(d):
        if r not in x:
            if u[r, r] != 1:
                part(r).mul_(complex(u[r, r]))
            continue
        cols = [j for j in used if u[r, j] != 0]
        y = x[cols[0]] * complex(u[r, cols[0]])
        for j in cols[1:]:
            y.add_(x[j], alpha=complex(u[r, j]))
        part(r).copy_(y)


def _blocked(psi):
    """The device layout of psi: blocks of 32 real parts, then 32 imaginary parts."""
    pad = (-psi.numel()) % 32
    if pad:
        psi = torch.cat((psi, psi.new_zeros(pad)))
    v = torch.view_as_real(psi).view(-1, 32, 2)
    return v.transpose(1, 2).reshape(-1)


def _circuit64(n, gates, basis):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[basis] = 1
    for g in gates:
        _apply64(psi, n, g)
    return psi


def _signs(z, n, device):
    """(-1)^popcount(j & z) for every j"""
    s = torch.ones(1, dtype=torch.float64, device=device)
    for q in range(n):
        s = torch.cat((s, -s if (z >> q) & 1 else s))
    return s


def exact(case, seed):
    if case["kind"] == "batch":
        return torch.cat([_blocked(_circuit64(n, gates, 0)) for n, gates in _batch(case, seed)])
    n = case["n"]
    if case["kind"] == "readout":
        amps = _ansatz_state(n, seed, "cuda")
        psi = amps.to(torch.complex128)
        out, products = [], {}
        for x, z in zip(*(m.tolist() for m in _strings(case))):
            if x not in products:   # conj(c_(j^x)) c_j
                j = torch.arange(1 << n, device="cuda") ^ x
                products = {x: psi[j].conj_physical_() * psi}
            p = products[x]
            c = bin(x & z).count("1") & 3
            s = _signs(z, n, "cuda")
            out.append(float((p.real * s).sum()) * (1, 0, -1, 0)[c] + float((p.imag * s).sum()) * (0, -1, 0, 1)[c])
        return {"terms": np.array(out), "samples": None, "norm": float(torch.view_as_real(psi).square().sum()), "amps": psi}
    if case["circuit"] == "qft":   # 2^(-n/2) exp(2 pi i x y / 2^n)
        basis = wl.qft_basis_index(n, seed)
        out = torch.empty(2 << n, dtype=torch.float64, device="cuda")
        step = 1 << min(n, 26)
        for y0 in range(0, 1 << n, step):
            y = torch.arange(y0, y0 + step, device="cuda")
            angle = ((y * basis) & ((1 << n) - 1)).double() * (2 * math.pi / (1 << n))
            out[2 * y0:2 * (y0 + step)] = _blocked(torch.polar(torch.full_like(angle, 2.0 ** (-n / 2)), angle))
        return out
    if n > 28:
        return None   # tens of seconds of 64-bit passes
    gates, basis = _gates(case, seed)
    return _blocked(_circuit64(n, gates, basis))
