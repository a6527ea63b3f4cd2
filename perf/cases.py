"""Measured cases: amplitude sweeps as users of the library run them.

A case names a circuit shape (n qubits, d entangling layers), how many
bitstrings are evaluated and the public entry point that evaluates them. The
circuits are the ones the library is built for: brickwork CZ, a uniform random
Clifford in every one-qubit slot, T gates at density 0.095 per qubit-layer and
uniform output bitstrings; one kind replaces both by Haar-random one-qubit
gates and random controlled phases. The boundary width is ceil(d/2).

Kinds:
  host    Plan.amplitudes: host bitstrings in, host amplitudes out, workspace kept
  device  Plan.amplitudes_device (device-resident inputs, asynchronous)
  xeb     device sweep, then the log-XEB estimate of its amplitudes on the device
  dense   device sweep of a circuit with Haar gates and controlled phases
  open    Plan(open_k=k).amplitudes: all 2^k amplitudes of every prefix
  split   device sweeps of one circuit in both split-precision forms
  batch   Batch.launch: uneven circuits recorded into one CUDA graph
  serve   Server.submit / wait: a burst of requests of uneven size
"""
import cmath
import math
import random

import numpy as np
import torch

import paper_2608_13110_gb300 as tb

T_DENSITY = 0.095
MAX_WORK = 70 * 31 * 2.0 ** 31  # row-steps x boundary entries of the largest listed case


def listed():
    return [
        # the smallest configuration: every amplitude of a 12-qubit check, one call
        dict(name="tiny_12x8", kind="host", n=12, d=8, nb=64),
        # a narrow serving request, the most bitstrings a request brings
        dict(name="narrow_45x22", kind="device", n=45, d=22, nb=256),
        # one amplitude of a mid-size circuit of odd depth: latency of the whole call
        dict(name="single_33x35", kind="host", n=33, d=35, nb=1),
        # a mid-width serving request with many bitstrings
        dict(name="request_61x32", kind="host", n=61, d=32, nb=200),
        # the oracle-sized slice of the n=70, d=56 circuit and its log-XEB
        dict(name="slice_30x40", kind="xeb", n=30, d=40, nb=32),
        # general gates: Haar one-qubit gates and controlled phases
        dict(name="dense_28x42", kind="dense", n=28, d=42, nb=16),
        # the method at scale: width 28, 2 GiB boundary
        dict(name="scale_70x56", kind="device", n=70, d=56, nb=2),
        # near the widest plain sweeps: width 31, 16 GiB boundary
        dict(name="wide_70x62", kind="device", n=70, d=62, nb=1),
        # batched sampling: 256 amplitudes per prefix from one sweep (width 26)
        dict(name="open_40x52_k8", kind="open", n=40, d=52, nb=2, k=8),
        # the precision comparison's oracle-sized slice, 3xTF32 and 3xBF16
        dict(name="split_32x48", kind="split", n=32, d=48, nb=4),
        # uneven circuits (n in 20..70, widths 8..24) in one graph launch
        dict(name="batch_24", kind="batch", circuits=24, max_width=24, nb=32, mix=11),
        # a burst of serving requests (n in 16..70, widths 4..20, 1..128 bitstrings)
        dict(name="serve_24", kind="serve", circuits=24, max_width=20, nb=128, mix=12),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["host", "device", "device", "xeb", "dense", "open", "split", "batch", "serve"])
    if kind in ("batch", "serve"):
        wide = kind == "batch"
        return dict(kind=kind, circuits=_log_int(rng, 4, 32), max_width=rng.randint(10, 23 if wide else 20),
                    nb=_log_int(rng, 4, 32 if wide else 128), mix=rng.randrange(1 << 30))
    n = rng.randint(12, 70)
    if kind == "open":
        h = rng.randint(13, 26)
        d = 2 * h - rng.randint(0, 1)
        return dict(kind=kind, n=n, d=d, nb=rng.randint(1, 4), k=rng.randint(1, min(10, d // 4, n - 1)))
    lo, hi = {"host": (2, 22), "device": (4, 31), "xeb": (4, 24), "dense": (4, 24), "split": (14, 26)}[kind]
    h = rng.randint(lo, hi)
    nb = _log_int(rng, 1, 256)
    nb = max(1, min(nb, int(MAX_WORK / 4 / _steps_work(n, 2 * h))))
    return dict(kind=kind, n=n, d=max(2, 2 * h - rng.randint(0, 1)), nb=nb)


# ---- inputs ---------------------------------------------------------------

def _shapes(case):
    """(n, d, bitstrings) of every circuit of a case."""
    if case["kind"] not in ("batch", "serve"):
        return [(case["n"], case["d"], case["nb"])]
    rng = random.Random(case["mix"])
    out = []
    lo_n, lo_h = (20, 8) if case["kind"] == "batch" else (16, 4)
    for _ in range(case["circuits"]):
        n, h = rng.randint(lo_n, 70), rng.randint(lo_h, case["max_width"])
        out.append((n, 2 * h, case["nb"] if case["kind"] == "batch" else rng.randint(1, case["nb"])))
    return out


def _circuit(case, seed, i):
    """Gate indices, bitstrings and (kind "dense") gates of circuit i."""
    n, d, nb = _shapes(case)[i]
    g = np.random.default_rng([seed, i, n, d])
    cliff = g.integers(0, 24, size=(d + 1, n), dtype=np.uint8)
    tmask = np.zeros(d * n, np.uint8)
    tmask[g.choice(d * n, size=int(round(T_DENSITY * n * d)), replace=False)] = 1
    bits = g.integers(0, 2, size=(nb, n - case.get("k", 0)), dtype=np.uint8)
    c = dict(n=n, d=d, nb=nb, cliff=cliff, tmask=tmask.reshape(d, n), bits=bits, extra=None, phases=None)
    if case["kind"] == "dense":
        z = g.standard_normal((d + 1, n, 2, 2)) + 1j * g.standard_normal((d + 1, n, 2, 2))
        q, r = np.linalg.qr(z)
        ph = np.diagonal(r, axis1=-2, axis2=-1)
        c["extra"] = q * (ph / np.abs(ph))[..., None, :]
        c["phases"] = g.uniform(0.0, 2.0 * np.pi, size=(d, n - 1))
    return c


def _plan(c, **opts):
    extra = None
    if c["extra"] is not None:
        extra = [(q, t, c["extra"][t, q]) for t in range(c["d"] + 1) for q in range(c["n"])]
    return tb.Plan(c["n"], c["d"], c["cliff"], c["tmask"], extra, cphase=c["phases"], **opts)


def _resident(plan, c):
    """Device buffers of one evaluation: (plan, bits, workspace with tables, out)."""
    d_bits = torch.from_numpy(c["bits"]).cuda()
    ws = plan.alloc_workspace(c["nb"])
    plan.upload(ws)
    return plan, d_bits, ws, torch.zeros((c["nb"], 2), dtype=torch.float64, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    cs = [_circuit(case, seed, i) for i in range(len(_shapes(case)))]
    st = dict(kind=kind, n=cs[0]["n"])
    if kind in ("host", "open"):
        st["plan"] = _plan(cs[0], open_k=case.get("k", 0))
        st["bits"] = cs[0]["bits"]
        st["ws"] = st["plan"].alloc_workspace(cs[0]["nb"])
    elif kind in ("device", "xeb", "dense"):
        st["evals"] = [_resident(_plan(cs[0]), cs[0])]
        st["f"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    elif kind == "split":
        st["evals"] = [_resident(_plan(cs[0], precision=p), cs[0]) for p in ("tf32x3", "bf16x3")]
    elif kind == "batch":
        items = [(_plan(c), torch.from_numpy(c["bits"]).cuda(),
                  torch.zeros((c["nb"], 2), dtype=torch.float64, device="cuda")) for c in cs]
        st["batch"] = tb.Batch(items)
        st["outs"] = [it[2] for it in items]
    else:
        st["server"] = tb.Server(hbm_budget_bytes=8 << 30, slots=4)
        st["requests"] = [(_plan(c), c["bits"]) for c in cs]
    return st


# ---- one pass -------------------------------------------------------------

def run(st):
    kind = st["kind"]
    if kind in ("host", "open"):
        return st["plan"].amplitudes(st["bits"], ws=st["ws"])
    if kind == "batch":
        st["batch"].launch()
        return st["outs"]
    if kind == "serve":
        tickets = [st["server"].submit(plan, bits) for plan, bits in st["requests"]]
        return [st["server"].wait(t)[0] for t in tickets]
    for plan, d_bits, ws, d_out in st["evals"]:
        plan.amplitudes_device(d_bits, ws, d_out)
    if kind == "xeb":
        tb.log_xeb_device(st["evals"][0][3], st["n"], st["f"])
        return [st["evals"][0][3], st["f"]]
    return [e[3] for e in st["evals"]]


# ---- work -----------------------------------------------------------------

def _steps_work(n, d):
    h = (d + 1) // 2
    return float(n) * h * 2.0 ** h


def work(case):
    """Inputs (bitstrings, two gate indices per slot) and amplitudes once; the
    paired steps of the dense method, one controlled 2x2 complex gate per
    boundary bit and absorbed row: 16 flops per boundary entry and step."""
    b = f = 0.0
    reps = 2 if case["kind"] == "split" else 1
    for n, d, nb in _shapes(case):
        k = case.get("k", 0)
        h = (d + 1) // 2
        b += reps * (nb * (n - k) + 2.0 * n * (d + 1) + 16.0 * nb * 2.0 ** k)
        f += reps * nb * max(1, n - 2 - max(0, k - 1)) * h * 2.0 ** h * 16.0
        if k:  # early region joined over its k crossing bits
            f += nb * 2.0 ** h * 2.0 ** k * 8.0
    return {"bytes": b, "flops": f}


# ---- the same amplitudes in 64 bits ---------------------------------------

def _gates(c):
    """(d+1, n, 2, 2) one-qubit gates: U = E . T^tau . C, C = P . R."""
    s, i = math.sqrt(0.5), 1j
    ident = np.eye(2, dtype=complex)
    had, ph = np.array([[s, s], [s, -s]], complex), np.diag([1, i])
    paulis = [ident, np.array([[0, 1], [1, 0]], complex), np.array([[0, -i], [i, 0]]), np.diag([1, -1 + 0j])]
    rots = [ident, had, ph, ph @ had, had @ ph, had @ ph @ had]
    cl = np.array([paulis[k % 4] @ rots[k // 4] for k in range(24)])
    u = cl[c["cliff"]]
    t = np.diag([1, cmath.exp(0.25j * math.pi)])
    u[:-1] = np.where(c["tmask"][..., None, None] != 0, t @ u[:-1], u[:-1])
    return u if c["extra"] is None else c["extra"] @ u


def _amplitudes64(c, k=0):
    """Amplitudes in complex128, one qubit row at a time in forward time: axes
    (bitstring, wire value, stored bits); a layer shared with the row above
    sums a stored bit out, one shared with the row below stores the wire."""
    n, d = c["n"], c["d"]
    u = _gates(c)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    nb = c["bits"].shape[0]
    bits = torch.from_numpy(c["bits"].astype(np.int64)).to(dev)

    def w(l, q):
        return -1.0 if c["phases"] is None else cmath.exp(1j * c["phases"][l, q])

    def mul(m, a, b):
        return complex(m[0]) * a + complex(m[1]) * b

    B = torch.ones((nb, 1), dtype=torch.complex128, device=dev)
    for r in range(n - k):
        a0, a1 = complex(u[0, r, 0, 0]) * B, complex(u[0, r, 1, 0]) * B
        low = 1  # entries of the bits this row has stored so far
        for l in range(d):
            if r > 0 and l % 2 == (r - 1) % 2:
                v0, v1 = (a.reshape(nb, -1, 2, low) for a in (a0, a1))
                a0 = (v0[:, :, 0] + v0[:, :, 1]).reshape(nb, -1)
                a1 = (v1[:, :, 0] + w(l, r - 1) * v1[:, :, 1]).reshape(nb, -1)
            g = u[l + 1, r]
            if r + 1 < n and l % 2 == r % 2:
                v0, v1 = a0.reshape(nb, -1, low), a1.reshape(nb, -1, low)
                a0, a1 = (torch.stack((complex(g[o, 0]) * v0, complex(g[o, 1]) * v1), 2).reshape(nb, -1)
                          for o in (0, 1))
                low *= 2
            else:
                a0, a1 = mul(g[0], a0, a1), mul(g[1], a0, a1)
        B = torch.where(bits[:, r, None] == 0, a0, a1)
    if k == 0:
        return B.reshape(nb)
    # open band: axes (bitstring, band values y, stored bits), all band qubits in step
    psi = torch.ones((1, 1), dtype=torch.complex128, device=dev)
    for j in range(k):
        col = torch.tensor(u[0, n - k + j, :, 0], dtype=torch.complex128, device=dev)
        psi = (col[:, None] * psi.reshape(1, -1)).reshape(-1, 1)
    T = (psi.reshape(1, -1, 1) * B.reshape(nb, 1, -1))
    y = torch.arange(1 << k, device=dev)
    for l in range(d):
        if l % 2 == (n - k - 1) % 2:
            v = T.reshape(nb, 1 << k, -1, 2)
            ph = torch.where(y % 2 == 1, torch.tensor(w(l, n - k - 1), dtype=torch.complex128, device=dev), 1.0)
            T = v[..., 0] + ph[None, :, None] * v[..., 1]
        for j in range(k - 1):
            if l % 2 == (n - k + j) % 2:
                both = ((y >> j) & 1) * ((y >> (j + 1)) & 1)
                T = T * torch.where(both == 1, torch.tensor(w(l, n - k + j), dtype=torch.complex128, device=dev),
                                    1.0)[None, :, None]
        for j in range(k):
            v = T.reshape(nb, 1 << (k - 1 - j), 2, -1)
            g = u[l + 1, n - k + j]
            T = torch.stack((mul(g[0], v[:, :, 0], v[:, :, 1]), mul(g[1], v[:, :, 0], v[:, :, 1])), 2)
        T = T.reshape(nb, 1 << k, -1)
    return T.reshape(nb, 1 << k)


def exact(case, seed):
    kind, k = case["kind"], case.get("k", 0)
    outs, total = [], 0.0
    for i, (n, d, nb) in enumerate(_shapes(case)):
        h = (d + 1) // 2
        cost = nb * _steps_work(n, d)
        total += cost
        if cost > 3e11 or total > 6e11 or nb * 2.0 ** (h + (k if k else 1)) > 2.0 ** 29:
            outs.append(None)
            continue
        a = _amplitudes64(_circuit(case, seed, i), k)
        outs.append(a.cpu().numpy() if kind in ("host", "open", "serve") else torch.view_as_real(a).cpu())
    if kind in ("host", "open"):
        return outs[0]
    if kind == "xeb":
        if outs[0] is None:
            return None
        p = (outs[0] ** 2).sum(1)
        f = np.euler_gamma + case["n"] * math.log(2.0) + float(torch.log(p).mean())
        return [outs[0], torch.tensor([f], dtype=torch.float64)]
    if kind == "split":
        return None if outs[0] is None else [outs[0], outs[0]]
    return None if all(o is None for o in outs) else outs
