"""Staged passes on the CPU: the plan's geometry and gate descriptors, read as the kernel reads them.
Every address a thread forms lies in its tile (or in the state), the groups of a gate are disjoint
and complete, tiles are copied whole and once, and a numpy run of the passes gives the oracle's state."""
import struct
import time

import numpy as np
import pytest

import oracle
from paper_2602_09604_gb300 import build as libbuild
from paper_2602_09604_gb300 import workloads as wl


@pytest.fixture(scope="module")
def B():
    libbuild.build()
    from paper_2602_09604_gb300 import binding
    return binding


SWZ = [1, 2, 4, 8, 16, 20, 24, 12, 28]   # position XOR of tile block bit i


def xor_sum(vectors, index):
    """XOR of vectors[b] over the set bits b of every entry of index."""
    out = np.zeros_like(index)
    for b, v in enumerate(vectors):
        out ^= np.where((index >> b) & 1, v, 0)
    return out


def swz(c):
    return xor_sum(SWZ, c)


def tile_address(t):
    """float offset in the tile of tile-local amplitude t's real part"""
    c = t >> 5
    return 64 * c + ((t & 31) ^ swz(c))


class Pass:
    def __init__(self, block, n):
        head = struct.unpack("<8i16qii", block[:168])
        self.fb, self.fpos, self.ioff, self.n_gates, units = head[0], head[1:8], head[8:24], head[24], head[25]
        assert len(block) == 168 + 16 * units
        self.image = np.frombuffer(block, dtype=np.float32, offset=168)
        self.n, self.tiles = n, 1 << (n - 5 - self.fb)
        self.gates = []
        for i in range(self.n_gates):
            w = struct.unpack("<5I7HH5HHHBB4xQ", block[168 + 64 * i:168 + 64 * i + 64])
            self.gates.append(dict(lane=w[:5], step=w[5:12], tv=w[13:18], cset=w[18], moff=w[19], k=w[20], nb=w[21], cm_out=w[22]))

    def base(self, t):
        for b in range(self.fb):
            low = t & ((1 << self.fpos[b]) - 1)
            t = ((t >> self.fpos[b]) << (self.fpos[b] + 1)) | low
        return t

    def moves(self, threads):
        """(float offset from the tile's first block, float offset in the tile, order of the four floats)
        of every 16-byte chunk that the threads copy."""
        sh = 3 if threads == 128 else 5
        tid = np.arange(threads)
        lane, warp = tid & 31, tid >> 5
        cthr = (warp & 3) | ((lane >> 4) << 2) | ((warp >> 2) << 3)
        goff = (lane & 15) * 4
        for b in range(min(self.fb, sh)):
            goff = goff + np.where((cthr >> b) & 1, 64 << self.fpos[b], 0)
        soff = cthr * 64 + (lane & 8) * 4 + (((lane & 7) ^ (swz(cthr) >> 2)) << 2)
        out = []
        for i in range(1 << (7 - sh)):
            has = cthr + (i << sh) < (1 << self.fb)
            iv = (i << sh) * 64 ^ (int(swz(np.array(i << sh))) >> 2) << 2
            assert (i << (sh - 3)) < 16
            out += list(zip((goff + self.ioff[i << (sh - 3)])[has], (soff ^ iv)[has], (warp & 3)[has]))
        return out

    def groups(self, g, threads):
        """Base address of every group that a thread takes: (thread, trip, v) -> address."""
        fast = threads == 512
        per = 1 if fast else {1: 4, 2: 4, 3: 4, 4: 2, 5: 1}[g["k"]]
        lt, lv = (9 if fast else 7), {4: 2, 2: 1, 1: 0}[per]
        nb, tid = g["nb"], np.arange(threads)
        active = tid if nb >= lt else tid[(tid >> nb) == 0]
        bt = np.zeros_like(active) ^ g["cset"]
        for b in range(5):
            bt ^= np.where((active >> b) & 1, g["lane"][b] & 0xffff, 0)
            bt ^= np.where((active >> (b + 5)) & 1, g["lane"][b] >> 16, 0)
        rows = []
        for it in range(1 << max(0, nb - lt - lv)):
            base = bt.copy()
            for b in range(lt + lv, nb):
                if (it >> (b - lt - lv)) & 1:
                    base ^= g["step"][b - 5]
            for v in range(per):
                pv = 0
                for b in range(lv):
                    if (v >> b) & 1:
                        pv ^= g["step"][lt - 5 + b]
                rows.append(base ^ pv)
        return np.array(rows)   # rows of threads

    def check(self):
        size = 64 << self.fb
        every = tile_address(np.arange(32 << self.fb))
        assert np.array_equal(np.sort(every), np.flatnonzero(np.arange(size) & 32 == 0))
        used = []
        for threads in (128, 512):
            got = self.moves(threads)
            assert len(got) == 16 << self.fb
            where = sorted(int(s) for _, s, _ in got)
            assert where == list(range(0, size, 4))
            top = (self.base(self.tiles - 1) << 6) + max(int(g) for g, _, _ in got) + 4
            assert top == 2 << self.n   # the last tile's last chunk ends the state
            assert min(int(g) for g, _, _ in got) == 0
            for g, s, p in got[:: max(1, len(got) // 64)]:   # chunk float e lands at s + (e ^ p)
                block = int(g) >> 6
                tb = sum(((block >> f) & 1) << b for b, f in enumerate(self.fpos[:self.fb]))
                for e in range(4):
                    at = (int(g) & 63) + e
                    want = tile_address(np.array(32 * tb + (at & 31))) + (at & 32)
                    assert s + (e ^ p) == want
        end = 64 * self.n_gates // 4
        for g in self.gates:
            assert 1 <= g["k"] <= 5 and 4 * g["moff"] >= end and 4 * g["moff"] + (2 << 2 * g["k"]) <= self.image.size
            used.append((4 * g["moff"], 4 * g["moff"] + (2 << 2 * g["k"])))
            rows = xor_sum(g["tv"][:g["k"]], np.arange(1 << g["k"]))
            for threads in (128, 512):
                base = self.groups(g, threads)
                addr = base[..., None] ^ rows
                assert addr.min() >= 0 and addr.max() + 32 < size and not (addr & 32).any()
                distinct = np.unique(base)
                assert len(distinct) == 1 << g["nb"]
                assert len(np.unique(distinct[:, None] ^ rows)) == len(distinct) << g["k"]
                # copies of a group are one thread's
                assert len(distinct) == sum(len(np.unique(base[:, t])) for t in range(base.shape[1]))
        assert all(a[1] <= b[0] for a, b in zip(sorted(used), sorted(used)[1:]))

    def run(self, psi):
        """psi (complex128, 2^n) under the pass."""
        t = np.arange(32 << self.fb)
        addr = tile_address(t)
        for tile in range(self.tiles):
            b0 = self.base(tile)
            block = b0 + sum((((t >> (5 + b)) & 1) << self.fpos[b]) for b in range(self.fb))
            idx = 32 * block + (t & 31)
            mem = np.zeros(64 << self.fb, dtype=np.complex128)
            mem[addr] = psi[idx]
            for g in self.gates:
                if ((b0 << 5) & g["cm_out"]) != g["cm_out"]:
                    continue
                d = 1 << g["k"]
                m = self.image[4 * g["moff"]:4 * g["moff"] + 2 * d * d].reshape(d, d // 2, 4)
                u = np.empty((d, d), dtype=np.complex128)
                u[0::2] = (m[:, :, 0] + 1j * m[:, :, 2]).T
                u[1::2] = (m[:, :, 1] + 1j * m[:, :, 3]).T
                a = np.unique(self.groups(g, 128))[:, None] ^ xor_sum(g["tv"][:g["k"]], np.arange(d))
                mem[a] = mem[a] @ u.T
            psi[idx] = mem[addr]


def circuit(n, max_k, seed, count=60):
    rng = np.random.default_rng(seed)
    gates = []
    for _ in range(count):
        k = int(rng.integers(1, min(max_k, n) + 1))
        g = wl.random_gate(n, k, rng)
        free = [q for q in range(n) if q not in g.targets]
        if k <= 2 and free and rng.random() < 0.25:
            c = int(rng.integers(1, len(free) + 1))
            g = wl.Gate(g.targets, g.matrix, tuple(int(q) for q in rng.choice(free, c, replace=False)), "c")
        gates.append(g)
    return gates


@pytest.mark.parametrize("n", [5, 6, 9, 11, 12, 14, 16])
@pytest.mark.parametrize("max_k", [1, 2, 3, 4, 5])
def test_passes_run_as_the_kernel_reads_them(B, n, max_k):
    gates = circuit(n, max_k, seed=100 * n + max_k, count=24)
    f = B.sv_fuse_circuit(gates, n, max_k=max_k)
    plan = B.sv_fused_plan_passes(f)
    assert sorted(g for s in plan for g in s["gates"]) == list(range(B.sv_fused_count(f)))
    psi = wl.random_state(n, np.random.default_rng(n)).astype(np.complex128)
    ref = psi.copy()
    threads = oracle.default_threads()
    passes = 0
    for s in plan:
        if s["tile"]:
            p = Pass(s["block"], n)
            p.check()
            p.run(psi)
            passes += 1
        else:
            assert len(s["gates"]) == 1
            info = B.sv_fused_get_info(f, s["gates"][0])
            oracle.apply_gate(psi, n, wl.Gate(info["targets"], B.sv_fused_get_matrix(f, s["gates"][0]), info["controls"], "f"), threads)
    assert passes or B.sv_fused_count(f) == 1
    for g in gates:
        oracle.apply_gate(ref, n, g, threads)
    # the images hold the matrices in fp32: 2^-24 a component, at most 2^(k+1) of them a row
    assert oracle.l2_error(ref, psi) <= B.sv_fused_count(f) * 2 ** (max_k + 1) * 2.0 ** -24
    B.sv_fused_free(f)


@pytest.mark.parametrize("n", [17, 19, 22, 35])
def test_addresses_on_large_states(B, n):
    for max_k in (1, 2, 3, 4, 5):
        gates = circuit(n, max_k, seed=n + max_k, count=40)
        # pieces near each other at the top and the bottom, so that passes form at every size
        rng = np.random.default_rng(n)
        gates += [wl.random_gate(n, min(2, max_k), rng, targets=tuple(range(q, q + min(2, max_k)))) for q in (0, 3, 4, n - 2, n - 4, n - 3, 5, n - 2)]
        f = B.sv_fuse_circuit(gates, n, max_k=max_k)
        plans = [B.sv_fused_plan_passes(f), B.sv_fused_plan_passes(f, from_basis=True)]
        for plan in plans:
            assert sorted(g for s in plan for g in s["gates"]) == list(range(B.sv_fused_count(f)))
            for s in plan:
                if s["tile"] and not s["on_small"]:
                    Pass(s["block"], n).check()
        assert any(s["tile"] for s in plans[0])
        B.sv_fused_free(f)


@pytest.mark.parametrize("from_basis", [False, True])
def test_order_is_kept_around_tensor_core_gates(B, from_basis):
    n, rng = 20, np.random.default_rng(2)
    pick = lambda k, hi: tuple(int(q) for q in rng.choice(hi, k, replace=False))
    gates = [wl.random_gate(n, 2, rng, targets=pick(2, n - 4)) for _ in range(50)]
    gates += [wl.random_gate(n, 5, rng, targets=(1, n - 4, n - 3, n - 2, n - 1))]
    gates += [wl.random_gate(n, 2, rng, targets=pick(2, n)) for _ in range(30)]
    f = B.sv_fuse_circuit(gates, n, mode=B.FUSE_NONE, precision=B.PREC_BF16X3, tc_min_k=4)
    plan = B.sv_fused_plan_passes(f, from_basis)
    for small in (True, False):
        order = [g for s in plan if s["on_small"] == small for g in s["gates"]]
        assert order == sorted(order)
    assert any(len(s["gates"]) > 1 for s in plan)
    B.sv_fused_free(f)
    f = B.sv_fuse_circuit(gates, n, mode=B.FUSE_NONE)   # without tensor cores gates do move
    order = [g for s in B.sv_fused_plan_passes(f) for g in s["gates"]]
    assert order != sorted(order)
    B.sv_fused_free(f)


def scan_plan(B, f, n, keep_order):
    """The passes by scans of all gates left: a gate joins when none left out before it shares a qubit
    with it and it fits (states below 21 qubits, where every run of two or more is a pass)."""
    infos = [B.sv_fused_get_info(f, i) for i in range(B.sv_fused_count(f))]
    masks = [sum(1 << q for q in i["targets"]) for i in infos]
    named = [m | sum(1 << q for q in i["controls"]) for m, i in zip(masks, infos)]
    fits = [i["path"] == B.PATH_CONTROLLED or (i["path"] in (B.PATH_LOW, B.PATH_HIGH, B.PATH_MIXED) and i["k"] <= 5) for i in infos]
    tile = min(n, 12 if n >= 19 else 10 if n <= 17 and max(i["k"] for i in infos) <= 2 else 11)
    left, out = list(range(len(infos))), []
    while left:
        lam, blocked, floats, took, rest = 31, 0, 0, [], []
        for s, g in enumerate(left):
            if (fits[g] and not named[g] & blocked and bin(lam | masks[g]).count("1") <= tile and len(took) < 48
                    and floats + 2 * 4 ** infos[g]["k"] <= 4096):
                lam |= masks[g]
                floats += 2 * 4 ** infos[g]["k"]
                took.append(g)
                continue
            if not took:
                took.append(g)
                rest += left[s + 1:]
                break
            blocked |= named[g]
            rest.append(g)
            if keep_order:
                rest += left[s + 1:]
                break
        out.append(took)
        left = rest
    return out


@pytest.mark.parametrize("n", [6, 13, 17, 20])
@pytest.mark.parametrize("max_k,precision", [(1, 0), (2, 0), (4, 0), (6, 0), (6, 2)])
def test_plan_is_the_first_fit_by_scans(B, n, max_k, precision):
    gates = circuit(n, min(max_k, 3), seed=n * max_k, count=150)
    f = B.sv_fuse_circuit(gates, n, max_k=min(max_k, n), precision=precision, tc_min_k=4)
    paths = {B.sv_fused_get_info(f, i)["path"] for i in range(B.sv_fused_count(f))}
    want = scan_plan(B, f, n, bool(paths & {B.PATH_TC_TF32, B.PATH_TC_BF16X3}))
    assert [s["gates"] for s in B.sv_fused_plan_passes(f)] == want
    B.sv_fused_free(f)


def test_planning_time_grows_with_the_gates(B):
    """200,000 unfused gates: 0.26 s with their images; scans of all gates left took 21 s."""
    n, rng = 20, np.random.default_rng(0)
    u = [wl.random_unitary(4, rng) for _ in range(8)]
    pairs = rng.integers(0, n, (200000, 2))
    gates = [wl.Gate((int(a), int(b)), u[i % 8], (), "g") for i, (a, b) in enumerate(pairs) if a != b]
    f = B.sv_fuse_circuit(gates, n, mode=B.FUSE_NONE)
    began = time.monotonic()
    assert B.lib.sv_fused_plan_passes(f, 0, 0, None, None, None, None, None, None, 0) > 1000
    assert time.monotonic() - began < 5.0
    B.sv_fused_free(f)
