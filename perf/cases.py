"""Workloads of the library, each one a call (or one batch) through its public Python entry points.

listed() names the standard ones, draw(rng) gives another of the same ranges, prepare(case, seed)
makes what a program holds before the call (device inputs, stored point sets, a workspace),
run(state) is one pass and returns its whole output, work(case) counts the bytes and operations a
pass cannot do without, and exact(case, seed) gives the output from plain integer arithmetic.

Kinds of case:
  msm      one multi-scalar multiplication sum_i a_i P_i. `form` says how the points are held:
           "standard" (n, 24) device points, "prepared" (their stored form, made once),
           "resident" (a library-owned set, the call takes a slice of it), "fixed_base" (shifted
           copies for one window width), "host" (points and scalars in pinned host memory, copied
           in by the call). `edwards` / `glv` choose the curve model and the endomorphism split.
           `scalars` is "uniform" (a random challenge or blinded vector) or "witness" (a circuit's
           assignment: many zeros and ones, many machine words, the rest full width).
  batched  independent MSMs of uneven sizes over slices of one stored set, in one call.
  padd     independent mixed point additions, 1 % each of P + P, P + (-P), O + Q and P + O.
  fq_mul   independent products in the base field, standard form in and out.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2502_11660_gb300 as pkg

P = 0x01AE3A4617C510EAC63B05C06CA1493B1A22D9F300F5138F1EF3622FBA094800170B5D44300000008508C00000000001
R = 0x12AB655E9A2CA55660B44D1E5C37B00159AA76FED00000010A11800000000001
GX = 0x008848DEFE740A67C8FC6225BF87FF5485951E2CAA9D41BB188282C8BD37CB5CD5481512FFCD394EEAB9B16EB21BE9EF
GY = 0x01914A69C5102EFF1F674F5D30AFEEC4BD7FB348CA3E52D96D182AD44FB82305C2FE3D3634A9591AFD82DE55559C8EA6

SCALAR_BITS = 253       # scalars are below 2^252 < r, declared as 253-bit values
MUL = 276               # 32 x 32 -> 64-bit limb products of one base-field product


def _msm(name, n, form, edwards, glv, c=0, signed=True, scalars="uniform"):
    return {"name": name, "kind": "msm", "n": n, "form": form, "edwards": edwards, "glv": glv, "c": c,
            "signed": signed, "scalars": scalars}


def listed() -> list[dict]:
    return [
        # A verifier-sized call with every default: arbitrary curve points, no plan, no workspace.
        _msm("msm_default_1000", 1000, "standard", False, False),
        # A small commitment with a fixed 8-bit unsigned window, points converted inside the call.
        _msm("msm_4096_c8_unsigned", 4096, "standard", False, False, c=8, signed=False),
        # A small request of a proving service: a ragged slice of a resident set.
        _msm("msm_resident_13007", 13007, "resident", True, True),
        # A mid-sized commitment over arbitrary curve points stored once (no subgroup assumed).
        _msm("msm_xyzz_150001", 150001, "prepared", False, False),
        # A prover's witness commitment: new points, skewed scalars.
        _msm("msm_witness_300007", 300007, "standard", True, True, scalars="witness"),
        # A call from a host program that holds points and scalars in pinned memory.
        _msm("msm_host_262144", 1 << 18, "host", True, True),
        # The large commitment over arbitrary curve points.
        _msm("msm_xyzz_1048576", 1 << 20, "prepared", False, False),
        # The headline: a prover's large commitment over a stored subgroup set.
        _msm("msm_edwards_glv_1048576", 1 << 20, "prepared", True, True),
        # The largest request of the proving service.
        _msm("msm_resident_4194304", 1 << 22, "resident", True, True),
        # A queue of uneven requests handed over together.
        {"name": "batched_24_jobs", "kind": "batched", "jobs": 24, "lo_log2": 10.0, "hi_log2": 18.0, "sizes": 3},
        # A stream of independent point additions (the paper's throughput experiment).
        {"name": "padd_1000003", "kind": "padd", "n": 1000003, "form": "montgomery"},
        # A vector of field products on standard-form operands.
        {"name": "fq_mul_4000037", "kind": "fq_mul", "n": 4000037, "form": "standard"},
    ]


def _log_uniform(rng: random.Random, lo: float, hi: float) -> int:
    return int(2.0 ** rng.uniform(lo, hi))


def draw(rng: random.Random) -> dict:
    kind = rng.choices(("msm", "batched", "padd", "fq_mul"), (8, 1, 1, 1))[0]
    if kind == "batched":
        return {"kind": "batched", "jobs": rng.randint(2, 40), "lo_log2": 10.0,
                "hi_log2": rng.choice((13.0, 16.0, 18.0)), "sizes": rng.randrange(1 << 16)}
    if kind == "padd":
        return {"kind": "padd", "n": _log_uniform(rng, 10, 21), "form": rng.choice(("montgomery", "standard"))}
    if kind == "fq_mul":
        return {"kind": "fq_mul", "n": _log_uniform(rng, 12, 22), "form": rng.choice(("standard", "montgomery"))}
    form = rng.choice(("standard", "prepared", "prepared", "resident", "host", "fixed_base"))
    edwards, glv = rng.choice(((False, False), (False, False), (True, True), (True, True), (True, False),
                               (False, True)))
    if form == "fixed_base":
        edwards = True
    hi = 20.0 if form in ("standard", "host") or not (edwards and glv) else 22.0
    if form == "fixed_base":
        hi = 18.0
    n = _log_uniform(rng, 6, hi)
    c, signed = 0, True
    if form == "fixed_base":    # the width is part of the set
        c = max(8, min(16, int(math.log2(n)) - 1))
    elif form != "resident" and rng.random() < 0.15:   # a caller's own width
        c, signed = rng.randint(6, 12), rng.random() < 0.5
        n = min(n, 1 << 18)
    return {"kind": "msm", "n": n, "form": form, "edwards": edwards, "glv": glv, "c": c, "signed": signed,
            "scalars": rng.choice(("uniform", "uniform", "witness"))}


# ---------------------------------------------------------------- inputs

def _words(n: int, words: int, top_mask: int, gen: torch.Generator) -> torch.Tensor:
    """n little-endian values of `words` 32-bit limbs, the top limb masked."""
    w = torch.randint(-(2 ** 31), 2 ** 31, (n, words), dtype=torch.int32, generator=gen)
    w[:, words - 1] &= top_mask
    return w


def _gen(seed: int, tag: int) -> torch.Generator:
    g = torch.Generator()
    g.manual_seed((seed * 1000003 + tag) & 0x7FFFFFFFFFFFFFFF)
    return g


def _scalars(n: int, kind: str, seed: int, tag: int) -> torch.Tensor:
    g = _gen(seed, tag)
    s = _words(n, 8, 0x0FFFFFFF, g)
    if kind == "witness":
        u = torch.rand(n, generator=g)
        s[u < 0.30] = 0                       # unused wires
        ones = (u >= 0.30) & (u < 0.50)       # booleans
        s[ones] = 0
        s[ones, 0] = 1
        s[(u >= 0.50) & (u < 0.75), 2:] = 0   # 64-bit words
    return s


def _seeds(n: int, seed: int, tag: int = 1) -> torch.Tensor:
    return _words(n, 8, 0x0FFFFFFF, _gen(seed, tag))


def _points(seeds: torch.Tensor) -> torch.Tensor:
    return pkg.g1_generator_mul(seeds.cuda())


def _sizes(case: dict) -> list[int]:
    r = random.Random(case["sizes"])
    return [_log_uniform(r, case["lo_log2"], case["hi_log2"]) for _ in range(case["jobs"])]


def _slice_offset(n: int) -> int:
    """Where a resident request's slice starts (sets are larger than the request)."""
    return min(256, n // 8)


def _prepare_msm(case: dict, seed: int) -> dict:
    n, form = case["n"], case["form"]
    mode = {"edwards": case["edwards"], "glv": case["glv"]}
    opts = {"c": case["c"], "signed": case["signed"], "scalar_bits": SCALAR_BITS}
    scalars = _scalars(n, case["scalars"], seed, 2)
    offset = _slice_offset(n) if form == "resident" else 0
    points = _points(_seeds(n + offset, seed))
    st = {"case": case, "opts": opts, "mode": mode}
    if form == "host":
        st["pinned"] = points.cpu().pin_memory(), scalars.pin_memory()
        st["points"], st["scalars"] = (t.numpy().view(np.uint32) for t in st["pinned"])
        need = pkg.msm_g1_host_workspace_bytes(n, opts["c"], opts["signed"], SCALAR_BITS, **mode)
        st["workspace"] = torch.empty(need, dtype=torch.uint8, device="cuda")
        return st
    st["scalars"] = scalars.cuda()
    if form == "standard":
        st["points"] = points
        st["workspace"] = None if n <= 1024 else pkg.msm_g1_workspace(n, **opts, **mode)
    elif form == "prepared":
        st["points"] = pkg.msm_points_prepare(points, **mode)
        st["workspace"] = pkg.msm_g1_workspace(n, prepared=True, **opts, **mode)
    elif form == "resident":
        st["offset"] = offset
        st["set"] = pkg.ResidentSet(points, scalar_bits=SCALAR_BITS, signed=case["signed"], **mode)
        st["workspace"] = st["set"].workspace(n)
    elif form == "fixed_base":
        st["points"] = pkg.msm_points_precompute(points, case["c"], SCALAR_BITS, case["signed"], case["glv"])
        st["workspace"] = pkg.msm_g1_workspace(n, precomputed=True, **opts, **mode)
    else:
        raise ValueError(form)
    return st


def _prepare_batched(case: dict, seed: int) -> dict:
    sizes = _sizes(case)
    stored = pkg.msm_points_prepare(_points(_seeds(max(sizes), seed)), edwards=True, glv=True)
    points = [stored[:2 * n] for n in sizes]
    scalars = [_scalars(n, "uniform", seed, 10 + i).cuda() for i, n in enumerate(sizes)]
    ws = pkg.msm_g1_batched_workspace(points, scalar_bits=SCALAR_BITS, prepared=True, edwards=True, glv=True)
    return {"case": case, "stored": stored, "points": points, "scalars": scalars, "workspace": ws}


def _soa(rows: torch.Tensor, parts: int) -> torch.Tensor:
    """(n, 12 parts) -> [parts][12][n]."""
    return rows.t().reshape(parts, 12, rows.shape[0]).contiguous()


def _prepare_padd(case: dict, seed: int) -> dict:
    n = case["n"]
    g = _gen(seed, 3)
    acc_seeds, q_seeds = _seeds(n, seed, 4), _seeds(n, seed, 5)
    u = torch.rand(n, generator=g)
    q_seeds[u < 0.01] = acc_seeds[u < 0.01]                         # P + P
    for i in torch.nonzero((u >= 0.01) & (u < 0.02)).flatten().tolist():
        s = R - int.from_bytes(acc_seeds[i].numpy().tobytes(), "little")   # P + (-P)
        q_seeds[i] = torch.from_numpy(np.frombuffer(s.to_bytes(32, "little"), np.int32).copy())
    q_seeds[(u >= 0.02) & (u < 0.03)] = 0                           # P + O
    inf = ((u >= 0.03) & (u < 0.04)).cuda()                         # O + Q
    acc, q = _soa(_points(acc_seeds), 2), _soa(_points(q_seeds), 2)
    one_by_one = torch.stack([acc[0], acc[1], q[0], q[1]])
    mont = torch.stack([pkg.fq_to_montgomery(x) for x in one_by_one])
    lam = _soa(_words(n, 12, 0x00FFFFFF, g).cuda(), 1)[0]
    mul = lambda a, b: pkg.fq_mul_batch(a, b, form=pkg.FORM_MONTGOMERY)
    l2 = mul(lam, lam)
    l3 = mul(l2, lam)
    acc = torch.stack([mul(mont[0], l2), mul(mont[1], l3), l2, l3])
    acc[:, :, inf] = 0
    q = mont[2:].contiguous()
    if case["form"] == "standard":
        acc = torch.stack([pkg.fq_from_montgomery(x) for x in acc])
        q = torch.stack([pkg.fq_from_montgomery(x) for x in q])
    return {"case": case, "acc": acc, "q": q, "form": _form(case)}


def _form(case: dict) -> int:
    return pkg.FORM_STANDARD if case["form"] == "standard" else pkg.FORM_MONTGOMERY


def _fq_operands(case: dict, seed: int) -> tuple[torch.Tensor, torch.Tensor]:
    g = _gen(seed, 6)
    return _words(case["n"], 12, 0x00FFFFFF, g), _words(case["n"], 12, 0x00FFFFFF, g)


def _prepare_fq_mul(case: dict, seed: int) -> dict:
    a, b = _fq_operands(case, seed)
    return {"case": case, "a": _soa(a.cuda(), 1)[0], "b": _soa(b.cuda(), 1)[0], "form": _form(case)}


def prepare(case: dict, seed: int) -> dict:
    return {"msm": _prepare_msm, "batched": _prepare_batched, "padd": _prepare_padd,
            "fq_mul": _prepare_fq_mul}[case["kind"]](case, seed)


def run(state: dict):
    case = state["case"]
    if case["kind"] == "padd":
        return pkg.padd_batch(state["acc"], state["q"], form=state["form"])
    if case["kind"] == "fq_mul":
        return pkg.fq_mul_batch(state["a"], state["b"], form=state["form"])
    if case["kind"] == "batched":
        return pkg.msm_g1_batched(state["points"], state["scalars"], workspace=state["workspace"],
                                  scalar_bits=SCALAR_BITS, prepared=True, edwards=True, glv=True)
    form, opts, mode = case["form"], state["opts"], state["mode"]
    if form == "host":
        return pkg.msm_g1_host(state["points"], state["scalars"], workspace=state["workspace"], **opts, **mode)
    if form == "resident":
        return state["set"].msm(state["scalars"], offset=state["offset"], workspace=state["workspace"])
    return pkg.msm_g1(state["points"], state["scalars"], workspace=state["workspace"], prepared=form == "prepared",
                      precomputed=form == "fixed_base", **opts, **mode)


# ---------------------------------------------------------------- work and values

def _windows(case: dict, n: int, glv: bool) -> int:
    """Digit windows of one scalar at a width near the best for n points."""
    c = case.get("c") or max(4, min(16, int(math.log2(max(n, 2))) - 2))
    return -(-(127 if glv else SCALAR_BITS) // c)


def _msm_work(case: dict, n: int, edwards: bool, glv: bool) -> tuple[int, int]:
    """Bytes in (points and scalars once) and limb products of one mixed addition per digit: 7
    field products on the Edwards curve, 5 and a square (210 limb products) between affine points."""
    adds = _windows(case, n, glv) * (2 * n if glv else n)
    return n * (96 + 32) + 96, adds * (7 * MUL if edwards else 5 * MUL + 210)


def work(case: dict) -> dict:
    if case["kind"] == "padd":
        b, ops = 480 * case["n"], case["n"] * (8 * MUL + 2 * 210)
    elif case["kind"] == "fq_mul":
        b, ops = 144 * case["n"], case["n"] * MUL
    elif case["kind"] == "batched":
        per = [_msm_work(case, n, True, True) for n in _sizes(case)]
        b, ops = sum(x for x, _ in per), sum(y for _, y in per)
    else:
        b, ops = _msm_work(case, case["n"], case["edwards"], case["glv"])
    return {"bytes": b, "flops": 2 * ops}   # a limb product is a multiply and an add


def _ints(rows: torch.Tensor) -> list[int]:
    raw, width = rows.contiguous().numpy().tobytes(), 4 * rows.shape[1]
    return [int.from_bytes(raw[i:i + width], "little") for i in range(0, len(raw), width)]


def _dot(a: torch.Tensor, b: torch.Tensor) -> int:
    """sum_i a_i b_i of 256-bit rows: 16-bit digits, exact in float64 over 2^20 rows at a time."""
    total = 0
    for lo in range(0, a.shape[0], 1 << 20):
        x = torch.from_numpy(a[lo:lo + (1 << 20)].numpy().view(np.uint16).astype(np.float64))
        y = torch.from_numpy(b[lo:lo + (1 << 20)].numpy().view(np.uint16).astype(np.float64))
        for i, row in enumerate((x.t() @ y).tolist()):
            for j, v in enumerate(row):
                total += int(v) << (16 * (i + j))
    return total


def _generator_times(k: int) -> torch.Tensor:
    """k G as (24,) int32 words, by affine double-and-add on y^2 = x^3 + 1; the identity is (0, 0)."""
    acc, base, k = None, (GX, GY), k % R
    while k:
        if k & 1:
            acc = base if acc is None else _add(acc, base)
        base = _add(base, base)
        k >>= 1
    x, y = acc or (0, 0)
    return torch.from_numpy(np.frombuffer(x.to_bytes(48, "little") + y.to_bytes(48, "little"), np.int32).copy())


def _add(a, b):
    if a is None or b is None:
        return a or b
    if a[0] == b[0]:
        if (a[1] + b[1]) % P == 0:
            return None
        m = 3 * a[0] * a[0] * pow(2 * a[1], -1, P) % P
    else:
        m = (b[1] - a[1]) * pow(b[0] - a[0], -1, P) % P
    x = (m * m - a[0] - b[0]) % P
    return x, (m * (a[0] - x) - a[1]) % P


def exact(case: dict, seed: int):
    if case["kind"] == "padd":
        return None     # projective coordinates: one of many representatives of each sum
    if case["kind"] == "fq_mul":
        a, b = (_ints(x) for x in _fq_operands(case, seed))
        # standard form: a b; Montgomery form: a b 2^-384
        f = 1 if case["form"] == "standard" else pow(1 << 384, -1, P)
        out = b"".join((x * y * f % P).to_bytes(48, "little") for x, y in zip(a, b))
        rows = torch.from_numpy(np.frombuffer(out, np.int32).reshape(case["n"], 12).copy())
        return rows.t().contiguous()
    if case["kind"] == "batched":
        sizes = _sizes(case)
        s = _seeds(max(sizes), seed)
        return [_generator_times(_dot(_scalars(n, "uniform", seed, 10 + i), s[:n])) for i, n in enumerate(sizes)]
    n = case["n"]
    offset = _slice_offset(n) if case["form"] == "resident" else 0
    out = _generator_times(_dot(_scalars(n, case["scalars"], seed, 2), _seeds(n + offset, seed)[offset:]))
    return out.numpy().view(np.uint32) if case["form"] == "host" else out
