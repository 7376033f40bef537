"""The work that programs have this framework do, as measurable cases.

A case is a dict of plain values; ``kind`` says which public entry point it
goes through:

* ``m2``        Plan.m2: stabilizer Renyi entropy of one device state (sre_m2);
* ``host``      Plan.m2_host: the same from a pinned host buffer (sre_m2_host);
* ``alpha``     Plan.m_alpha: integer order alpha (sre_m_alpha);
* ``shard``     Plan.sum4_range: one rank's range of shifts (sre_sum4_range);
* ``batch``     Plan.m2_batched: states of equal or uneven N in one submission;
* ``brickwork`` Plan.brickwork_m2_series: random-circuit dynamics, M2 per step;
* ``tfim``      Plan.tfim_m2_series: Ising quench dynamics, M2 per step.

``mode`` is the plan's arithmetic (fp32, fp16_split, bf16_split, fp64); plans
are used as created, or with the tuning that an earlier autotuner run saved
(``tuning``).  The states are the paper's families with nonzero entropy
(Haar-random, random product, brickwork circuit), drawn on the device from the
seed.  M2 values that a call leaves on the device are read back as a program
reads them; a shard's sums stay on the device for the reduction that follows.
"""
import math

import numpy as np
import torch

from paper_2512_24685_gb300 import binding

FAMILIES = ("haar", "product", "brickwork")
DEVICE = "cuda"


def listed():
    return [
        # the smallest call: one 10-qubit state inside a scan, latency and launches
        {"name": "m2_n10", "kind": "m2", "N": 10, "mode": "fp32", "family": "brickwork"},
        # a state that arrives in host memory, odd N, first size beyond one tile
        {"name": "host_n13", "kind": "host", "N": 13, "mode": "fp32", "family": "product"},
        # a higher order of the same state family the experiments look at
        {"name": "alpha3_n15", "kind": "alpha", "N": 15, "mode": "fp32", "family": "product", "alpha": 3},
        # one circuit state at the paper's upper dynamics size
        {"name": "m2_n16", "kind": "m2", "N": 16, "mode": "fp32", "family": "brickwork"},
        # a large single state in plain FP32
        {"name": "m2_n18", "kind": "m2", "N": 18, "mode": "fp32", "family": "brickwork"},
        # the benchmark's size and mode: split-precision on the tensor cores, with
        # the tuning that the benchmark's autotuner run picked
        {"name": "m2_n20_fp16", "kind": "m2", "N": 20, "mode": "fp16_split", "family": "brickwork",
         "tuning": "3,6,2,5,0"},
        # complex128 input in the default mode of such a plan
        {"name": "m2_n16_fp64", "kind": "m2", "N": 16, "mode": "fp64", "family": "product"},
        # one of several ranks' share of a 19-qubit state: a ragged shift range
        {"name": "shard_n19", "kind": "shard", "N": 19, "mode": "fp32", "family": "haar", "begin": 61813,
         "count": 58255},
        # a mixed-family batch of 16-qubit states in the split mode
        {"name": "batch_n16_fp16", "kind": "batch", "n_lo": 16, "n_hi": 16, "count": 8, "mode": "fp16_split"},
        # snapshots of uneven size in one submission, replayed on a side stream
        {"name": "batch_uneven", "kind": "batch", "n_lo": 12, "n_hi": 17, "count": 24, "mode": "fp32"},
        # random-circuit dynamics: realizations of 14 qubits, M2 after every step
        {"name": "brickwork_n14", "kind": "brickwork", "N": 14, "S": 20, "T": 3, "mode": "fp32"},
        # quench dynamics in the default (FP64) mode of a complex128 plan
        {"name": "tfim_n12", "kind": "tfim", "N": 12, "S": 20, "T": 3, "mode": "fp64"},
    ]


def draw(rng):
    """One more case of the ranges above (N 8 to 19 for one state in FP32 or a
    split mode, up to 16 in FP64; batches of N 10 to 17; dynamics of N 8 to 14)."""
    kind = rng.choice(["m2", "m2", "m2", "host", "alpha", "shard", "batch", "batch", "brickwork", "tfim"])
    family = rng.choice(FAMILIES[1:])
    if kind in ("m2", "host"):
        mode = rng.choice(["fp32", "fp32", "fp16_split", "bf16_split", "fp64"])
        N = rng.randint(8, 16) if mode == "fp64" else rng.randint(16, 19) if "split" in mode else rng.randint(8, 19)
        return {"kind": kind, "N": N, "mode": mode, "family": family}
    if kind == "alpha":
        return {"kind": kind, "N": rng.randint(9, 17), "mode": "fp32", "family": "product", "alpha": rng.randint(3, 6)}
    if kind == "shard":
        N, mode = rng.choice([(rng.randint(14, 19), "fp32"), (rng.randint(16, 19), "fp16_split"),
                              (rng.randint(14, 16), "fp64")])
        d = 1 << N
        count = rng.randint(d // 32, d // 4)
        return {"kind": kind, "N": N, "mode": mode, "family": "haar", "begin": rng.randint(1, d - count),
                "count": count}
    if kind == "batch":
        lo, hi = sorted((rng.randint(10, 17), rng.randint(10, 17)))
        mode = rng.choice(["fp32", "fp32", "fp16_split"])
        most = min(5.5, 37 - 2 * hi)
        return {"kind": kind, "n_lo": lo, "n_hi": hi, "count": int(round(2 ** rng.uniform(1, most))), "mode": mode}
    N, S, T = rng.randint(8, 14), rng.randint(2, 20), rng.randint(1, 3)
    return {"kind": kind, "N": N, "S": S, "T": T, "mode": rng.choice(["fp32", "fp64"]) if N <= 12 else "fp32"}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _randn(shape, g):
    return torch.randn(shape, dtype=torch.complex128, device=DEVICE, generator=g)


def _haar4(n, g):
    """n Haar-random 4x4 unitaries: QR of complex Gaussian matrices with the
    phases of R's diagonal moved into Q."""
    q, r = torch.linalg.qr(_randn((n, 4, 4), g))
    d = torch.diagonal(r, dim1=-2, dim2=-1)
    return (q * (d / d.abs()).unsqueeze(-2)).contiguous()


def _pair(psi, q, u):
    """Gates u (S, 4, 4) on qubits q, q + 1 of the states psi (S, 2^N)."""
    v = psi.reshape(psi.shape[0], -1, 4, 1 << q)
    return torch.einsum("sab,sibj->siaj", u, v).reshape(psi.shape)


def _bonds(N):
    return list(range(0, N - 1, 2)) + list(range(1, N - 1, 2))


def _products(S, N, g):
    """S product states with Bloch vectors uniform on the sphere."""
    r = torch.rand((S, N, 2), dtype=torch.float64, device=DEVICE, generator=g)
    half = torch.acos(2 * r[..., 0] - 1) / 2
    one = torch.polar(torch.sin(half), 2 * math.pi * r[..., 1])
    psi = torch.ones((S, 1), dtype=torch.complex128, device=DEVICE)
    for j in range(N):  # qubit j is bit j of the index
        psi = torch.cat([psi * torch.cos(half[:, j:j + 1]), psi * one[:, j:j + 1]], dim=1)
    return psi


def _state(N, family, g):
    """One complex128 state of a family."""
    if family == "haar":
        psi = _randn((1 << N,), g)
        return psi / psi.abs().square().sum().sqrt()
    if family == "product":
        return _products(1, N, g)[0]
    psi = torch.zeros((1, 1 << N), dtype=torch.complex128, device=DEVICE)
    psi[0, 0] = 1
    for _ in range(8):  # a depth-8 brickwork circuit
        u = _haar4(N - 1, g)
        for k, q in enumerate(_bonds(N)):
            psi = _pair(psi, q, u[k:k + 1])
    return psi[0]


def _batch(case, seed):
    """The states of a batch: sizes n_lo..n_hi and the families in turn."""
    g = _gen(seed)
    span = case["n_hi"] - case["n_lo"] + 1
    return [_state(case["n_lo"] + k % span, FAMILIES[(k // span if span > 1 else k) % 3], g).to(torch.complex64)
            for k in range(case["count"])]


def _input(case, seed):
    """The input of a case, as the program holds it (complex64 unless the mode
    is fp64 or the entry point evolves complex128 states)."""
    kind = case["kind"]
    if kind == "batch":
        return _batch(case, seed)
    g = _gen(seed)
    if kind == "brickwork":
        N, S, T = case["N"], case["S"], case["T"]
        return _haar4(T * S * (N - 1), g).reshape(T, S, N - 1, 4, 4).contiguous()
    if kind == "tfim":
        return _products(case["S"], case["N"], g)
    psi = _state(case["N"], case["family"], g)
    return psi if case["mode"] == "fp64" else psi.to(torch.complex64)


def prepare(case, seed):
    kind, x = case["kind"], _input(case, seed)
    dtype = "c128" if case["mode"] == "fp64" or kind in ("brickwork", "tfim") else "c64"
    plan = binding.Plan(case.get("N") or case["n_hi"], dtype, case["mode"])
    if case.get("tuning"):
        plan.set_tuning(*map(int, case["tuning"].split(",")))
    state = {"case": case, "plan": plan, "x": x}
    if kind == "host":
        state["x"] = x.cpu().pin_memory()
    if kind == "batch":
        # uneven submissions are replayed from their graph, on a stream of their own
        state["stream"] = torch.cuda.Stream() if case["n_lo"] < case["n_hi"] else torch.cuda.current_stream()
        state["out"] = torch.empty(len(x), dtype=torch.float64, device=DEVICE)
        torch.cuda.synchronize()
    if kind == "brickwork":
        state["psi"] = torch.empty((case["S"], 1 << case["N"]), dtype=torch.complex128, device=DEVICE)
    if kind == "tfim":
        state["psi"] = torch.empty_like(x)
    return state


def run(state):
    case, plan, x = state["case"], state["plan"], state["x"]
    kind = case["kind"]
    if kind == "m2":
        return plan.m2(x)
    if kind == "host":
        return plan.m2_host(x)
    if kind == "alpha":
        return plan.m_alpha(x, case["alpha"])
    if kind == "shard":
        return plan.sum4_range(x, case["begin"], case["begin"] + case["count"])
    if kind == "batch":
        with torch.cuda.stream(state["stream"]):
            return plan.m2_batched(x, out=state["out"]).tolist()
    if kind == "brickwork":
        m2, psi = plan.brickwork_m2_series(x, state["psi"])
    else:
        psi = state["psi"].copy_(x)  # the series evolves its states in place
        m2 = plan.tfim_m2_series(psi, case["T"])
    return {"m2": m2.tolist(), "states": psi}


# -------------------------------------------------------------------- work

def _terms(case):
    """Pauli terms by N of one pass: {N: terms}."""
    kind = case["kind"]
    if kind == "batch":
        span, got = case["n_hi"] - case["n_lo"] + 1, {}
        for k in range(case["count"]):
            N = case["n_lo"] + k % span
            got[N] = got.get(N, 0) + 4 ** N
        return got
    N = case["N"]
    if kind == "shard":
        return {N: case["count"] << N}
    return {N: 4 ** N * case.get("S", 1) * case.get("T", 1)}


def work(case):
    """Each state read once, each result written once; per Pauli term the N - 1
    additions of the conjugate-symmetric transform and 6 operations of product
    and power (alpha: one more product per order), and the evolution's own."""
    kind, N = case["kind"], case.get("N")
    extra = case.get("alpha", 2) - 2
    flops = sum(t * (n + 5 + extra) for n, t in _terms(case).items())
    wide = 16 if case["mode"] == "fp64" else 8
    if kind == "batch":
        nbytes = sum((t >> n) * wide + 8 for n, t in _terms(case).items())
    elif kind in ("brickwork", "tfim"):
        S, T = case["S"], case["T"]
        nbytes = S * (16 << N) + 8 * S * T
        if kind == "brickwork":  # a complex 4x4 product per bond
            nbytes += T * S * (N - 1) * 256
            flops += T * S * (N - 1) * (32 << N)
        else:  # one term of H per qubit, about ||H|| dt + 20 terms of a polynomial in H
            nbytes += S * (16 << N)
            flops += T * S * (int(0.2 * (4 * N - 1)) + 20) * ((2 * N + 12) << N)
    else:
        nbytes = (wide << N) + 16
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------- exact

def _sum_pow(psi, alpha, begin, end):
    """sum over shifts [begin, end) of sum_z |A_x(z)|^(2 alpha), by products
    and radix-2 Walsh-Hadamard transforms in 64 bits."""
    d = psi.numel()
    t = torch.arange(d, device=psi.device)
    rows, total = max(1, (1 << 26) // d), 0.0
    for x0 in range(begin, end, rows):
        x = torch.arange(x0, min(end, x0 + rows), device=psi.device)
        a = psi[t[None, :] ^ x[:, None]].conj() * psi[None, :]
        h = 1
        while h < d:
            v = a.view(-1, d // (2 * h), 2, h)
            a = torch.stack((v[:, :, 0] + v[:, :, 1], v[:, :, 0] - v[:, :, 1]), dim=2).view(-1, d)
            h *= 2
        p = a.real.square() + a.imag.square()
        total += float(p.pow(alpha).sum())
    return total


def _entropy(psi, alpha=2):
    psi = psi.to(torch.complex128)
    d, n2 = psi.numel(), float(psi.abs().square().sum())
    s = _sum_pow(psi, alpha, 0, d)
    return (math.log2(s) - math.log2(d) - 2 * alpha * math.log2(n2)) / (1 - alpha)


def _quench(psi, dt=0.2, J=1.0, hx=1.5, hz=1.5):
    """exp(-i H dt) of the open Ising chain by a Taylor series in short substeps."""
    N = psi.shape[1].bit_length() - 1
    t = torch.arange(1 << N, device=psi.device)
    spin = [1.0 - 2.0 * ((t >> i) & 1).double() for i in range(N)]
    diag = -hz * sum(spin) - J * sum((spin[i] * spin[i + 1] for i in range(N - 1)), torch.zeros_like(spin[0]))
    steps = 16
    for _ in range(steps):
        term, acc = psi, psi.clone()
        for k in range(1, 25):
            hv = diag * term - hx * sum(term[:, t ^ (1 << i)] for i in range(N))
            term = hv * (-1j * dt / steps / k)
            acc = acc + term
        psi = acc
    return psi


def exact(case, seed):
    kind, x = case["kind"], _input(case, seed)
    if kind == "shard":
        if case["count"] << case["N"] > 100e9:
            return None
        psi = x.to(torch.complex128)
        s = _sum_pow(psi, 2, case["begin"], case["begin"] + case["count"])
        return np.array([s, float(psi.abs().square().sum())])
    if sum(_terms(case).values()) > 100e9:
        return None
    if kind == "batch":
        return [_entropy(psi) for psi in x]
    if kind == "brickwork":
        psi = torch.zeros((case["S"], 1 << case["N"]), dtype=torch.complex128, device=DEVICE)
        psi[:, 0] = 1
    elif kind == "tfim":
        psi = x
    else:
        return _entropy(x, case.get("alpha", 2))
    m2 = []
    for step in range(case["T"]):
        if kind == "brickwork":
            for k, q in enumerate(_bonds(case["N"])):
                psi = _pair(psi, q, x[step, :, k].contiguous())
        else:
            psi = _quench(psi)
        m2.append([_entropy(psi[s]) for s in range(case["S"])])
    return {"m2": m2, "states": psi}
