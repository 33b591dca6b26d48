"""The work that users of the loop-hafnian engine have it do, as cases that can be timed and
whose results can be checked.

A case is one pass through the public Python entry points (`lib.lhaf`, `lib.lhaf_async`,
`lib.gbs_prob`, `lib.lhaf_batch`, `lib.gbs_prob_batch`, `sampler.Sampler`). Four kinds:

  single   one loop hafnian of a GBS kernel matrix with loop weights: the probability
           amplitude of one detection event with one photon per mode. "call" is the
           synchronous call with a host matrix, "async" the device-only call with the
           caller's workspace. FP64 is the default precision, used up to the sizes where its
           rounding still leaves nine digits; triple-float is the accurate path, used at
           every size and the only one that is trusted at N >= 34.
  prob     one photon pattern with repeated modes through `gbs_prob` (FP64 only).
  batch    many problems of uneven size at once: photon patterns of one 100-mode state
           ("gbs") or a list of unrelated matrices, odd sizes among them ("mats").
  sample   photon-number samples of a squeezed, displaced state from the served chain-rule
           sampler.
"""
import math

import numpy as np
import torch

from paper_2010_15595_gb300 import lib, sampler, workloads

_PRECISION = {"fp64": lib.PREC_FP64, "tf": lib.PREC_TF}

# Ranges of the drawn cases (the listed ones lie inside them).
_SINGLE_N = {"fp64": (4, 32), "tf": (4, 44)}
_PROB_N = (6, 24)
_GBS_COUNT, _MATS_COUNT = (16, 512), (16, 256)
_SAMPLE_MODES, _SAMPLE_COUNT = (8, 48), (1, 16)


def listed():
    return [
        # smallest real evaluation: a 16-photon event, latency of one synchronous call
        {"name": "single_fp64_n16_call", "kind": "single", "N": 16, "precision": "fp64", "api": "call"},
        # the largest size at which the default precision is still good to nine digits
        {"name": "single_fp64_n30", "kind": "single", "N": 30, "precision": "fp64", "api": "async"},
        # small accurate evaluation inside a device pipeline: launches and gaps count
        {"name": "single_tf_n16", "kind": "single", "N": 16, "precision": "tf", "api": "async"},
        # odd photon number (padded by one vertex)
        {"name": "single_tf_n25", "kind": "single", "N": 25, "precision": "tf", "api": "async"},
        # the middle of the paper's range, matrix and result on the host
        {"name": "single_tf_n32_call", "kind": "single", "N": 32, "precision": "tf", "api": "call"},
        # the headline evaluation: 2^20 subsets
        {"name": "single_tf_n40", "kind": "single", "N": 40, "precision": "tf", "api": "async"},
        # the largest evaluation that takes under a second
        {"name": "single_tf_n44", "kind": "single", "N": 44, "precision": "tf", "api": "async"},
        # probability of one pattern with several photons in some modes
        {"name": "prob_fp64_n22", "kind": "prob", "N": 22, "M": 12},
        # unrelated small matrices, every size from 1 to 16
        {"name": "batch_mats_tf_128", "kind": "batch", "form": "mats", "count": 128, "n_max": 16, "precision": "tf"},
        # probability tables: patterns of 10 to 30 photons of a 100-mode state
        {"name": "batch_gbs_fp64_512", "kind": "batch", "form": "gbs", "count": 512, "n_max": 30, "precision": "fp64"},
        {"name": "batch_gbs_tf_512", "kind": "batch", "form": "gbs", "count": 512, "n_max": 30, "precision": "tf"},
        # serving: 16 samples of a 40-mode state asked for together
        {"name": "sample_m40_16", "kind": "sample", "M": 40, "count": 16, "cutoff": 4, "n_cap": 28},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)) - 0.02))))


def draw(rng):
    # the work of a single evaluation doubles with every second photon, so a uniform N spreads
    # it over its logarithm
    kind = rng.choice(["single", "single", "single", "prob", "batch", "batch", "sample"])
    if kind == "single":
        precision = rng.choice(["fp64", "tf", "tf"])
        return {"kind": "single", "N": rng.randint(*_SINGLE_N[precision]), "precision": precision,
                "api": rng.choice(["call", "async"])}
    if kind == "prob":
        return {"kind": "prob", "N": rng.randint(*_PROB_N), "M": rng.randint(8, 40)}
    if kind == "batch":
        form, precision = rng.choice(["gbs", "mats"]), rng.choice(["fp64", "tf"])
        if form == "gbs":
            return {"kind": "batch", "form": "gbs", "count": _log_int(rng, *_GBS_COUNT),
                    "n_max": rng.randint(12, 30), "precision": precision}
        return {"kind": "batch", "form": "mats", "count": _log_int(rng, *_MATS_COUNT),
                "n_max": rng.randint(4, 22), "precision": precision}
    return {"kind": "sample", "M": _log_int(rng, *_SAMPLE_MODES), "count": _log_int(rng, *_SAMPLE_COUNT),
            "cutoff": rng.randint(3, 5), "n_cap": 28}


# ---------------------------------------------------------------------------------- inputs

def _single_matrix(case, seed):
    if case["N"] == 16:
        return workloads.single_lhaf_n16(seed)
    return workloads.single_lhaf_mid(case["N"], seed)


def _prob_inputs(case, seed):
    """Kernel matrix and fill vector of an M-mode state and a pattern of N photons, at most
    four in a mode."""
    rng = workloads.rng_for(40, seed * 10000 + case["N"] * 100 + case["M"])
    M, N = case["M"], case["N"]
    B = workloads.squeezed_kernel(workloads.haar_unitary(M, rng), rng.uniform(0.4, 0.9, M))
    gamma = workloads.complex_normal(M, 0.2, rng)
    pattern = np.zeros(M, dtype=np.int32)
    for _ in range(N):
        free = np.nonzero(pattern < 4)[0]
        pattern[free[rng.integers(len(free))]] += 1
    return B, gamma, pattern


def _mats(case, seed):
    rng = workloads.rng_for(41, seed)
    mats = []
    for i in range(case["count"]):
        N = 1 + i % case["n_max"]
        B = workloads.squeezed_kernel(workloads.haar_unitary(N, rng), rng.uniform(0.4, 0.9, N))
        mats.append(workloads.with_diagonal(B, workloads.complex_normal(N, 0.2, rng)))
    return mats


def _gbs_inputs(case, seed):
    B, gamma = workloads.batch_state(seed)
    pats = workloads.batch_patterns(case["count"], seed=seed, n_max=case["n_max"])
    p_vac = np.full(case["count"], 0.25)
    return B, gamma, pats, p_vac


def prepare(case, seed):
    kind = case["kind"]
    if kind == "single":
        A = _single_matrix(case, seed)
        prec = _PRECISION[case["precision"]]
        if case["api"] == "call":
            return {"kind": "call", "A": A, "precision": prec}
        return {"kind": "async", "A": torch.from_numpy(A).cuda(), "precision": prec,
                "out": torch.zeros(1, dtype=torch.complex128, device="cuda"),
                "ws": torch.empty(lib.workspace_size(case["N"], prec), dtype=torch.uint8, device="cuda")}
    if kind == "prob":
        B, gamma, pattern = _prob_inputs(case, seed)
        return {"kind": "prob", "B": torch.from_numpy(B).cuda(), "gamma": torch.from_numpy(gamma).cuda(),
                "pattern": pattern}
    if kind == "batch":
        prec = _PRECISION[case["precision"]]
        if case["form"] == "mats":
            return {"kind": "mats", "mats": _mats(case, seed), "precision": prec}
        B, gamma, pats, p_vac = _gbs_inputs(case, seed)
        return {"kind": "gbs", "B": torch.from_numpy(B).cuda(), "gamma": torch.from_numpy(gamma).cuda(),
                "patterns": pats, "p_vac": p_vac, "precision": prec}
    M = case["M"]
    U, r, alpha = workloads.serving_state(seed, M=M, n_squeezed=max(2, M // 4))
    served = sampler.Sampler(sampler.pure_state(U, r, alpha), cutoff=case["cutoff"],
                             n_cap=case["n_cap"], tick_subsets=1 << 16)
    return {"kind": "sample", "sampler": served, "seeds": [1000 * seed + i for i in range(case["count"])]}


def run(state):
    kind = state["kind"]
    if kind == "call":
        v = lib.lhaf(state["A"], precision=state["precision"])
        return np.array([v])
    if kind == "async":
        lib.lhaf_async(state["A"], state["out"], state["ws"], precision=state["precision"])
        return state["out"]
    if kind == "prob":
        prob, v = lib.gbs_prob(state["B"], state["gamma"], state["pattern"], p_vac=0.25, return_lhaf=True)
        return {"prob": prob, "lhaf": np.array([v])}
    if kind == "mats":
        return lib.lhaf_batch(state["mats"], precision=state["precision"])
    if kind == "gbs":
        probs, lhafs = lib.gbs_prob_batch(state["B"], state["gamma"], state["patterns"],
                                          p_vacs=state["p_vac"], precision=state["precision"])
        return {"probs": probs, "lhafs": lhafs}
    served = state["sampler"]
    ids = [served.submit(s, 1) for s in state["seeds"]]
    return np.concatenate([served.wait(i)[0] for i in ids])


# -------------------------------------------------------------------------------------- work

def _lhaf_flops(N):
    """Multiply-add flops that one N x N loop hafnian needs by the cheapest exact evaluation
    known: eliminate the n = N/2 index pairs one after the other with polynomial entries, one
    of 2^(n-1) sign patterns at a time. With p pairs left, a node of that recursion forms
    4 (p-1)^2 + 2 (p-1) + 2 truncated products of polynomials of degree n - p."""
    n = (N + 1) // 2
    total = 0.0
    for d in range(n):
        m = n - d - 1
        total += 2.0 ** max(d - 1, 0) * (4 * m * m + 2 * m + 2) * (d + 1) * (d + 2) / 2
    return 8.0 * total


def work(case):
    kind = case["kind"]
    if kind in ("single", "prob"):
        N = case["N"]
        return {"bytes": 16.0 * (N * N + 1), "flops": _lhaf_flops(N)}
    if kind == "batch":
        if case["form"] == "mats":
            Ns = [1 + i % case["n_max"] for i in range(case["count"])]
            return {"bytes": sum(16.0 * (N * N + 1) for N in Ns), "flops": sum(map(_lhaf_flops, Ns))}
        sizes = list(range(10, case["n_max"] + 1, 2))
        each = sum(map(_lhaf_flops, sizes)) / len(sizes)
        return {"bytes": 16.0 * 100 * 101 + case["count"] * (400.0 + 32), "flops": case["count"] * each}
    # about 0.2 photons in a mode: one loop hafnian per candidate at every mode
    M, d = case["M"], case["cutoff"] + 1
    flops = case["count"] * sum(sum(_lhaf_flops(round(0.22 * k) + s) for s in range(d)) for k in range(M))
    return {"bytes": case["count"] * (16.0 * M * M + 4 * M), "flops": flops}


# ------------------------------------------------------------------------------------- exact

def _masks(bits, most):
    """All `bits`-bit masks with at most `most` ones, ascending."""
    lists = [torch.zeros(1, dtype=torch.int64, device="cuda") for _ in range(most + 1)]
    for b in range(bits):
        lists = [lists[0]] + [torch.cat([lists[k], lists[k - 1] + (1 << b)]) for k in range(1, most + 1)]
    return lists[most]


_DENSE_BITS = 24  # levels of at most this many bits are held as a dense table


def _loop_hafnians(A):
    """Loop hafnians of a (count, N, N) stack by the definition, in complex128: match the
    lowest vertex i that is left with itself (weight A_ii) or a later vertex j (A_ij), with
    one value for every set of vertices above i that earlier ones have taken. At level i such
    a set has at most i members. Nothing cancels beyond what the matchings themselves do."""
    P, N, _ = A.shape
    chunk = max(1, (1 << 22) // P)
    nxt, nxt_keys = torch.ones((P, 1), dtype=torch.complex128, device="cuda"), None

    def look_up(keys):
        return nxt[:, keys if nxt_keys is None else torch.searchsorted(nxt_keys, keys)]

    for i in range(N - 1, -1, -1):
        bits = N - i  # bit b of a set stands for vertex i + b
        keys = _masks(bits, min(i, bits))
        dense = bits <= _DENSE_BITS
        cur = torch.zeros((P, 1 << bits if dense else len(keys)), dtype=torch.complex128, device="cuda")
        for c in range(0, len(keys), chunk):
            T = keys[c:c + chunk]
            free = (T & 1) == 0
            val = look_up(T >> 1)
            F = T[free]
            acc = A[:, i, i, None] * val[:, free]
            for b in range(1, bits):
                ok = ((F >> b) & 1) == 0
                acc[:, ok] += A[:, i, i + b, None] * look_up((F[ok] | (1 << b)) >> 1)
            val[:, free] = acc
            if dense:
                cur[:, T] = val
            else:
                cur[:, c:c + chunk] = val
        nxt, nxt_keys = cur, None if dense else keys
    return nxt[:, 0]


def _exact_lhafs(mats):
    out = np.zeros(len(mats), dtype=np.complex128)
    for N in sorted({m.shape[0] for m in mats}):
        which = [k for k, m in enumerate(mats) if m.shape[0] == N]
        # the largest table that is held: a dense level of at most 2^bits, or a short list
        at_once = max(1, (1 << 30) >> min(N, _DENSE_BITS))
        for c in range(0, len(which), at_once):
            part = which[c:c + at_once]
            A = torch.from_numpy(np.stack([mats[k] for k in part])).cuda()
            out[part] = _loop_hafnians(A).cpu().numpy()
    return out


def _expanded(B, gamma, pattern):
    idx = np.repeat(np.arange(len(pattern)), pattern)
    A = np.array(B[np.ix_(idx, idx)])
    A[np.diag_indices_from(A)] = gamma[idx]
    return A


def exact(case, seed):
    kind = case["kind"]
    if kind == "single":
        if case["N"] > 36:  # too long
            return None
        return _exact_lhafs([_single_matrix(case, seed)])
    if kind == "prob":
        B, gamma, pattern = _prob_inputs(case, seed)
        v = _exact_lhafs([_expanded(B, gamma, pattern)])
        fact = math.prod(math.factorial(int(s)) for s in pattern)
        return {"prob": float(0.25 * abs(v[0]) ** 2 / fact), "lhaf": v}
    if kind == "batch":
        if case["form"] == "mats":
            return _exact_lhafs(_mats(case, seed))
        B, gamma, pats, p_vac = _gbs_inputs(case, seed)
        v = _exact_lhafs([_expanded(B, gamma, p) for p in pats])
        fact = np.array([math.prod(math.factorial(int(s)) for s in p) for p in pats])
        return {"probs": p_vac * np.abs(v) ** 2 / fact, "lhafs": v}
    return None  # photon numbers: whole values
