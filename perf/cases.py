"""The work that users of this library have it do, as cases that can be timed and checked.

Every case goes through the public binding (paper_2512_07311_gb300.capi), as a program that
builds, samples and scores random-circuit states does. Five kinds ("op"):

  step    one circuit from host gates: apply, draw shots to the host, score them, look up
          amplitudes of given bitstrings. The whole pipeline, planning included.
  run     the same pipeline on a plan that was built and uploaded once (many circuits' worth
          of shots from one plan; the benchmark's timed step).
  state   a prepared plan from |0...0>, and the whole state handed over on the device.
  apply   a caller's own k-qubit unitaries on a state that already holds data.
  draw    shots from a state that already holds data, and the score of given bitstrings.
  batch   many circuits of mixed sizes in one launch: shots and scores of each.

All inputs come from the seed: the gates, the unitaries, the states and the bitstrings. The
qubits a case works on come from the case, so that every seed does the same work.
"""
import math

import numpy as np
import torch

from paper_2512_07311_gb300 import capi
from paper_2512_07311_gb300 import circuits as C

PRECISIONS = ("fp32_fused", "bf16x3", "tf32x3")
LOOKUPS = 4096  # bitstrings whose amplitudes a "step" or "run" asks for
SCORED = 1_000_000  # bitstrings a "draw" scores


def listed():
    return [
        # the smallest workload of the benchmark: a 12-qubit circuit, its plan made on the call, 10^4 shots
        dict(name="step_12q_fp32", op="step", n=12, cycles=8, pattern="ABCDCDAB", jitter=0.0, precision="fp32_fused",
             k_max=4, shots=10_000),
        # a one-off circuit of ordinary size on the tensor cores, planned on the call
        dict(name="step_21q_bf16", op="step", n=21, cycles=12, pattern="EFGH", jitter=0.05, precision="bf16x3", k_max=0,
             shots=100_000),
        # a state for another GPU program, small enough for launches to count (a ragged 4 x 5 - 1 grid)
        dict(name="state_19q_bf16", op="state", n=19, cycles=14, pattern="ABCDCDAB", jitter=0.0, precision="bf16x3",
             k_max=0),
        # the same at an ordinary size and full depth, larger than L2
        dict(name="state_27q_bf16", op="state", n=27, cycles=20, pattern="ABCDCDAB", jitter=0.0, precision="bf16x3",
             k_max=0),
        # ... with the more exact tensor-core split
        dict(name="state_28q_tf32", op="state", n=28, cycles=14, pattern="EFGH", jitter=0.05, precision="tf32x3",
             k_max=0),
        # ... in full FP32, the default precision
        dict(name="state_27q_fp32", op="state", n=27, cycles=14, pattern="EFGH", jitter=0.05, precision="fp32_fused",
             k_max=4),
        # the benchmark's 30-qubit workload on a prepared plan: state, 10^6 shots, score
        dict(name="run_30q_bf16", op="run", n=30, cycles=14, pattern="EFGH", jitter=0.05, precision="bf16x3", k_max=0,
             shots=1_000_000),
        # a caller's own six-qubit unitaries anywhere in a large state, low qubits among them
        dict(name="apply_29q_k6_bf16", op="apply", n=29, k=6, count=4, targets=3, precision="bf16x3"),
        # ... and seven-qubit ones, the widest there are, in FP32
        dict(name="apply_26q_k7_fp32", op="apply", n=26, k=7, count=2, targets=5, precision="fp32_fused"),
        # a state that is sampled and scored again and again (the paper's job array: 25 000 shots a job, 100 jobs)
        dict(name="draw_29q", op="draw", n=29, shots=2_500_000),
        # many circuits of 16 to 24 qubits at once on the tensor cores, 10^5 shots each
        dict(name="batch_24_bf16", op="batch", count=24, lo=16, hi=24, shots=100_000, precision="bf16x3", k_max=0),
        # smaller ones in FP32, the batch's default precision
        dict(name="batch_12_fp32", op="batch", count=12, lo=14, hi=22, shots=30_000, precision="fp32_fused", k_max=4),
    ]


def draw(rng):
    op = rng.choice(["step", "run", "state", "state", "apply", "apply", "draw", "batch"])

    def circuit(lo, hi):
        precision = rng.choice(PRECISIONS)
        return dict(op=op, n=rng.randint(lo, hi), cycles=rng.randint(6, 20), pattern=rng.choice(C.PATTERNS),
                    jitter=rng.choice([0.0, 0.05]), precision=precision,
                    k_max=rng.choice([3, 4, 4, 5]) if precision == "fp32_fused" else 0)

    if op in ("step", "run"):
        return dict(circuit(10, 26 if op == "step" else 28), shots=int(10 ** rng.uniform(3, 6)))
    if op == "state":
        return circuit(10, 27)
    if op == "apply":
        precision = rng.choice(PRECISIONS)
        k = 6 if precision != "fp32_fused" else rng.randint(1, 7)
        return dict(op=op, n=rng.randint(15, 28), k=k, count=rng.randint(1, 6), targets=rng.randrange(1 << 20),
                    precision=precision)
    if op == "draw":
        return dict(op=op, n=rng.randint(12, 28), shots=int(10 ** rng.uniform(3, 6.3)))
    lo = rng.randint(13, 20)
    precision = rng.choice(["fp32_fused", "bf16x3", "tf32x3"])
    return dict(op=op, count=rng.randint(2, 24), lo=lo, hi=rng.randint(lo, 23), shots=int(10 ** rng.uniform(3, 5)),
                precision=precision, k_max=rng.choice([3, 4]) if precision == "fp32_fused" else 0)


# ---------------------------------------------------------------------------- inputs


class State:
    """What a user's program keeps between calls; the library's handles go with it."""

    ctx = plan = batch = None

    def __del__(self):
        if self.plan is not None:
            capi.rcs_plan_destroy(self.plan)
        if self.batch is not None:
            capi.rcs_batch_destroy(self.batch)
        if self.ctx is not None:
            capi.rcs_destroy(self.ctx)


class _DeviceArray:
    def __init__(self, owner, ptr, count):
        self.owner = owner  # the memory lives as long as a tensor over it does
        self.__cuda_array_interface__ = dict(shape=(count,), typestr="<c8", data=(ptr, False), version=3, strides=None)


def device_state(s):
    """The context's state as a tensor (the library's own memory, caller's basis order)."""
    return torch.as_tensor(_DeviceArray(s, capi.rcs_state_device(s.ctx), 1 << s.case["n"]), device="cuda")


def circuit_of(case, seed):
    return C.generate(C.grid_for_n(case["n"]), case["cycles"], case["pattern"], seed=seed, jitter=case["jitter"])


def batch_circuits(case, seed):
    out = []
    for i in range(case["count"]):
        n = case["lo"] + i % (case["hi"] - case["lo"] + 1)
        out.append(C.generate(C.grid_for_n(n), 10 + 7 * i % 11, C.PATTERNS[i % 2], seed=seed * 1000 + i))
    return out


def random_state(n, seed):
    """Normalised complex Gaussian amplitudes: what a deep random circuit leaves (Porter-Thomas)."""
    g = torch.Generator("cuda").manual_seed(seed)
    psi = torch.randn(1 << n, dtype=torch.complex64, device="cuda", generator=g)
    norm = 0.0
    for part in psi.split(1 << 24):
        norm += float(torch.view_as_real(part).double().square().sum())
    return psi.mul_(1.0 / math.sqrt(norm))


def unitaries_of(case, seed):
    """(targets, U) pairs: targets anywhere in the register, in any order; U Haar-random."""
    where = np.random.default_rng(case["targets"])
    rng = np.random.default_rng(seed)
    d = 1 << case["k"]
    items = []
    for _ in range(case["count"]):
        targets = where.permutation(case["n"])[: case["k"]].astype(np.int32)
        q, r = np.linalg.qr(rng.standard_normal((d, d)) + 1j * rng.standard_normal((d, d)))
        items.append((targets, q * (np.diag(r) / np.abs(np.diag(r)))))
    return items


def bitstrings_of(psi, count, seed):
    """Basis indices distributed as |psi|^2, as a device would deliver them."""
    p = torch.view_as_real(psi).double().square().sum(-1).cumsum(0)
    g = torch.Generator("cuda").manual_seed(seed + 7)
    u = torch.rand(count, dtype=torch.float64, device="cuda", generator=g) * p[-1]
    return torch.searchsorted(p, u, right=True).clamp_(max=psi.numel() - 1)


def prepare(case, seed):
    s = State()
    s.case, op = case, case["op"]
    if op == "batch":
        items = [(c.n_qubits, c.gates, case["shots"], seed + i) for i, c in enumerate(batch_circuits(case, seed))]
        s.batch = capi.rcs_batch_create(items, k_max=case["k_max"], autotune=0,
                                        precision=capi.PRECISIONS[case["precision"]])
        return s
    n = case["n"]
    precision = capi.PRECISIONS[case.get("precision", "fp32_fused")]
    k_max = case.get("k_max", 0)
    s.seed = seed
    s.ctx = capi.rcs_create(n, precision, k_max=k_max)
    if op in ("step", "run", "state"):
        s.gates = circuit_of(case, seed).gates
        s.lookups = C.random_bitstrings(n, LOOKUPS, seed)
        if op != "step":
            s.plan = capi.rcs_plan_build(n, s.gates, precision, k_max=k_max)
            capi.rcs_plan_upload(s.ctx, s.plan)
    else:
        psi = random_state(n, seed)
        device_state(s).copy_(psi)
        if op == "apply":
            s.items = unitaries_of(case, seed)
        else:
            s.scored = bitstrings_of(psi, SCORED, seed)
            s.bits = torch.empty(case["shots"], dtype=torch.int64, device="cuda")
            s.xeb = torch.empty(1, dtype=torch.float64, device="cuda")
    return s


# ---------------------------------------------------------------------------- one pass


def run(s):
    case, op, ctx = s.case, s.case["op"], s.ctx
    if op in ("step", "run"):
        capi.rcs_reset(ctx)
        if op == "step":
            capi.rcs_apply_circuit(ctx, s.gates)
        else:
            capi.rcs_plan_run(ctx, s.plan)
        bits = capi.rcs_sample(ctx, case["shots"], s.seed)
        return {"bits": bits.view(np.int64), "xeb": capi.rcs_xeb(ctx, bits),
                "amplitudes": capi.rcs_amplitudes(ctx, s.lookups).astype(np.complex64)}
    if op == "state":
        capi.rcs_reset(ctx)
        capi.rcs_plan_run(ctx, s.plan)
        return device_state(s)
    if op == "apply":
        capi.rcs_apply_unitaries(ctx, s.items)
        return device_state(s)
    if op == "draw":
        capi.rcs_sample_device(ctx, case["shots"], s.seed, s.bits.data_ptr())
        capi.rcs_xeb_device(ctx, s.scored.data_ptr(), SCORED, s.xeb.data_ptr())
        return {"bits": s.bits, "xeb": s.xeb}
    capi.rcs_batch_launch(s.batch)
    capi.rcs_batch_wait(s.batch)
    got = [capi.rcs_batch_result(s.batch, i, case["shots"]) for i in range(case["count"])]
    return {"bits": np.concatenate([b for b, _ in got]).view(np.int64), "xeb": np.array([x for _, x in got]),
            "first_state": capi.rcs_batch_state_read(s.batch, 0)}


# ---------------------------------------------------------------------------- what a pass cannot do without


def work(case):
    op = case["op"]
    if op == "batch":
        parts = [work(dict(op="run", n=c.n_qubits, shots=case["shots"], gates=c.counts())) for c in batch_circuits(case, 0)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    amps = float(1 << case["n"])
    if op == "apply":  # the state in and out once
        return {"bytes": 16 * amps, "flops": 8 * amps * (1 << case["k"]) * case["count"]}
    if op == "draw":  # every probability once, the shots out, the scored bitstrings in
        return {"bytes": 8 * amps + 8 * case["shots"] + 16 * SCORED, "flops": 4 * amps}
    # the state out once; two complex multiplications and an addition per amplitude and one-qubit gate,
    # the same on half the amplitudes and a phase on a quarter per fSim gate
    gates = case.get("gates") or circuit_of(case, 0).counts()
    return {"bytes": 8 * amps + 16 * case.get("shots", 0),
            "flops": amps * (14 * gates["one_qubit"] + 8.5 * gates["fsim"])}


# ---------------------------------------------------------------------------- the same in 64 bits


def _gate_matrix(g):
    """The library's documented gate matrices (include/rcs.h), in complex128."""
    if g["kind"] == C.FSIM:
        c, s = math.cos(float(g["theta"])), math.sin(float(g["theta"]))
        m = np.array([[1, 0, 0, 0], [0, c, -1j * s, 0], [0, -1j * s, c, 0], [0, 0, 0, np.exp(-1j * float(g["phi"]))]])
    else:
        x, y = np.array([[0, 1], [1, 0]], complex), np.array([[0, -1j], [1j, 0]])
        p = {C.SQRT_X: x, C.SQRT_Y: y, C.SQRT_W: (x + y) / math.sqrt(2)}[int(g["kind"])]
        m = ((1 + 1j) * np.eye(2) + (1 - 1j) * p) / 2
    return m.conj().T if g["flags"] & C.ADJOINT else m


def _apply_exact(psi, n, targets, u):
    """psi (complex128, 2^n) with u applied on `targets` (local bit i on targets[i])."""
    k = len(targets)
    base = torch.arange(1 << (n - k), device=psi.device)
    for t in sorted(int(t) for t in targets):
        base = ((base >> t) << (t + 1)) | (base & ((1 << t) - 1))
    offs = [sum(((j >> i) & 1) << int(targets[i]) for i in range(k)) for j in range(1 << k)]
    x = [psi[base + o] for o in offs]
    if k <= 2:
        for j, o in enumerate(offs):
            terms = [complex(u[j, l]) * x[l] for l in range(1 << k) if u[j, l] != 0]
            psi[base + o] = sum(terms[1:], terms[0])
    else:
        y = torch.as_tensor(u, device=psi.device) @ torch.stack(x)
        for j, o in enumerate(offs):
            psi[base + o] = y[j]
    return psi


def _circuit_exact(n, gates):
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1
    for g in gates:
        psi = _apply_exact(psi, n, [int(g["q0"])] if g["nq"] == 1 else [int(g["q0"]), int(g["q1"])], _gate_matrix(g))
    return psi


def exact(case, seed):
    op = case["op"]
    if op == "batch":  # the shots are drawn, and the scores are of the drawn shots
        c = batch_circuits(case, seed)[0]
        return {"bits": None, "xeb": None, "first_state": _circuit_exact(c.n_qubits, c.gates)}
    n = case["n"]
    if op in ("step", "run", "state"):
        if n > 28:
            return None
        psi = _circuit_exact(n, circuit_of(case, seed).gates)
        if op == "state":
            return psi
        at = torch.as_tensor(C.random_bitstrings(n, LOOKUPS, seed).view(np.int64), device="cuda")
        return {"bits": None, "xeb": None, "amplitudes": psi[at]}
    psi = random_state(n, seed)
    if op == "apply":
        psi = psi.to(torch.complex128)
        for targets, u in unitaries_of(case, seed):
            psi = _apply_exact(psi, n, targets, u)
        return psi
    p = torch.view_as_real(psi).double().square().sum(-1)
    return {"bits": None, "xeb": ((1 << n) * p[bitstrings_of(psi, SCORED, seed)].mean() / p.sum() - 1).reshape(1)}
