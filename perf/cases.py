"""Performance cases of the sparse FFT library: whole transforms through the binding, over the range of
sizes, batches, precisions and layouts the library is used at.

Every case is one call a program makes again and again on new signals with the same plan:

* ``exact``    ``sfft_execute`` of an exact-mode plan (Algorithm 1) on a batch of signals in device memory;
* ``general``  ``sfft_execute`` of a general-mode plan (Algorithms 2 and 3) on noisy signals;
* ``channels`` ``sfft_execute_channels``: interleaved signals sampled at the same times;
* ``mixed``    ``BatchPlan.execute_prepared``: exact-mode requests of several (n, k) in one launch.

Inputs are those of ``workloads``: k coefficients of unit magnitude and uniform phase at uniform
frequencies (exact), or log-uniform magnitudes in [1, 10] plus complex Gaussian time noise at 20 dB
(general).  Outputs are the arrays a program passes in (indices, values, counts, flags), zeroed once:
entries past a request's count stay zero.
"""
import math

import numpy as np
import torch

from paper_1201_2501_gb300 import sfft, workloads

EXACT, GENERAL = sfft.SFFT_EXACT, sfft.SFFT_GENERAL
MAX_TAPS = 8_000_000         # window taps of a drawn exact or mixed case, all requests
MAX_GENERAL_TAPS = 80_000_000  # window taps of a drawn general case, all requests and hashings
MAX_SAMPLES = 1 << 30        # signal samples of a drawn case


def listed():
    return [
        # one small double-precision transform: the smallest call, all latency (n = 2^14, k = 8, delta = 1e-8)
        dict(name="exact fp64 n14 k8 x1", kind="exact", m=14, k=8, batch=1, fp64=True, delta=1e-8, alpha0=0.5, taps=2048),
        # one transform of a long signal, library defaults: the latency a single caller sees
        dict(name="exact n22 k64 x1", kind="exact", m=22, k=64, batch=1, fp64=False, delta=1e-6, alpha0=0.5, taps=2048),
        # a resident batch at the throughput benchmark's settings
        dict(name="exact n22 k64 x256", kind="exact", m=22, k=64, batch=256, fp64=False, delta=1e-6, alpha0=0.625,
             taps=4096),
        # a ragged batch of short signals, as a server forms it from what has arrived
        dict(name="exact n18 k61 x37", kind="exact", m=18, k=61, batch=37, fp64=False, delta=1e-6, alpha0=0.5, taps=2048),
        # many coefficients in a long signal: the largest bin counts (B = 4096 down to 16)
        dict(name="exact n24 k1000 x12", kind="exact", m=24, k=1000, batch=12, fp64=False, delta=1e-6, alpha0=0.5,
             taps=2048),
        # a double-precision batch
        dict(name="exact fp64 n20 k64 x16", kind="exact", m=20, k=64, batch=16, fp64=True, delta=1e-8, alpha0=0.5,
             taps=2048),
        # one noisy signal of moderate length: latency of the general algorithm
        dict(name="general n18 k50 x1", kind="general", m=18, k=50, batch=1),
        # the noisy workload of the benchmark's general case
        dict(name="general n22 k256 x8", kind="general", m=22, k=256, batch=8),
        # a very long noisy signal, where the sparse transform reads a tenth of it
        dict(name="general n26 k64 x4", kind="general", m=26, k=64, batch=4),
        # the largest bin count of the general algorithm (B = 4096) on a ragged batch
        dict(name="general n20 k500 x5", kind="general", m=20, k=500, batch=5),
        # a recorder's 256 channels sampled together
        dict(name="channels n21 k64 c256", kind="channels", m=21, k=64, batch=256, alpha0=0.625),
        # requests of six sizes in one launch
        dict(name="mixed n16..22 x96", kind="mixed", m_lo=16, m_hi=22, k_lo=8, k_hi=512, types=6, batch=96),
    ]


def _log_uniform(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["exact", "exact", "exact", "exact64", "general", "general", "general", "channels", "mixed"])
    while True:
        if kind in ("exact", "exact64"):
            fp64 = kind == "exact64"
            m = rng.randint(14, 20) if fp64 else rng.randint(16, 26)
            k = _log_uniform(rng, 8, min(256 if fp64 else 1024, (1 << m) // 64))
            c = dict(kind="exact", m=m, k=k, batch=_log_uniform(rng, 1, 256), fp64=fp64, delta=1e-8 if fp64 else 1e-6,
                     alpha0=rng.choice([0.5, 0.625]), taps=rng.choice([2048, 4096]) if k <= 256 else 2048)
        elif kind == "general":
            m = rng.randint(16, 26)
            c = dict(kind="general", m=m, k=_log_uniform(rng, 8, min(512, (1 << m) // 64)), batch=_log_uniform(rng, 1, 32))
        elif kind == "channels":
            c = dict(kind="channels", m=rng.randint(16, 21), k=_log_uniform(rng, 8, 64), batch=32 * rng.randint(1, 8),
                     alpha0=rng.choice([0.5, 0.625]))
        else:
            lo = rng.randint(14, 18)
            c = dict(kind="mixed", m_lo=lo, m_hi=rng.randint(lo, 22), k_lo=8, k_hi=_log_uniform(rng, 16, 512),
                     types=rng.randint(2, 6), batch=_log_uniform(rng, 8, 96))
        samples = (sum(1 << m for m, _ in _request_types(c)) if kind == "mixed" else c["batch"] << c["m"])
        taps = _total_taps(c) / (4 if c.get("fp64") else 1)
        if samples <= MAX_SAMPLES and taps <= (MAX_GENERAL_TAPS if kind == "general" else MAX_TAPS):
            return c


# ---- sizes -------------------------------------------------------------------------------------
def _pow2_at_least(v):
    return 1 << max(0, math.ceil(math.log2(v)))


def _exact_rounds(n, k, delta, alpha0):
    """(B, taps, hashings, samples) of every round of Algorithm 1's schedule."""
    out = []
    for t in range(math.ceil(math.log2(k)) + 1 if k > 1 else 1):
        kt = max(1, (k + (1 << t) - 1) >> t)
        B = min(max(_pow2_at_least(4 * kt), 16), n // 2)
        T = int(4 * B * math.log(1 / delta) / (math.pi * alpha0 * 2 ** (-t / 2)))
        Rc = min(_pow2_at_least(max(1.0, 1e-4 * n / (math.pi * B))), n // B // 2)
        H = 2 if Rc == 1 else 3
        out.append((B, 2 * T + 1, H, 2 * T + 1 + B * Rc))
    return out


def _general_rounds(n, k):
    """(B, taps, LocateInner pairs, estimation hashings) of every round of Algorithm 2's schedule."""
    out = []
    t = 1 << int(math.log2(math.log2(n)))
    while k >= 1:
        B = min(max(_pow2_at_least(8 * k), 16), n // 2)
        T = int(4 * B * math.log(1e6) / (math.pi * 0.5))
        out.append((B, 2 * T + 1, 7 * (int(math.log2(n // B)) // int(math.log2(t // 4)) + 1), 5))
        k //= 4
    return out


def _types(case):
    """The (log2 n, k) of a mixed case's plans."""
    c, out = case, []
    for i in range(c["types"]):
        m = c["m_lo"] + i * (c["m_hi"] - c["m_lo"]) // max(1, c["types"] - 1)
        f = (i * 5 % c["types"]) / max(1, c["types"] - 1)
        out.append((m, max(1, min(int(c["k_lo"] * (c["k_hi"] / c["k_lo"]) ** f), (1 << m) // 64))))
    return out


def _request_types(case):
    types = _types(case)
    return [types[r % len(types)] for r in range(case["batch"])]


def _total_taps(case):
    if case["kind"] == "general":
        return case["batch"] * sum(w * (2 * p + e) for _, w, p, e in _general_rounds(1 << case["m"], case["k"]))
    if case["kind"] == "mixed":
        return sum(sum(w for _, w, _, _ in _exact_rounds(1 << m, k, 1e-6, 0.5)) for m, k in _request_types(case))
    return case["batch"] * sum(w for _, w, _, _ in _exact_rounds(1 << case["m"], case["k"], case.get("delta", 1e-6),
                                                                 case["alpha0"]))


def work(case):
    """Bytes: the samples a transform asks for, a 32-byte sector each (contiguous rows of a channel
    batch count as they are), no more than the whole signal, and its recovered entries.  Flops: per
    tap one window product and, per hashing, one complex multiply-add into the fold."""
    def exact(n, k, delta, alpha0, elem, sector):
        rounds = _exact_rounds(n, k, delta, alpha0)
        return (min(sum(s for *_, s in rounds) * sector, n * elem) + 20 * k,
                sum(w * (2 + 8 * H) + H * 5 * B * math.log2(B) for B, w, H, _ in rounds))

    b = case["batch"]
    if case["kind"] == "general":
        n, k = 1 << case["m"], case["k"]
        rounds = _general_rounds(n, k)
        taps = sum(w * (2 * p + e) for _, w, p, e in rounds)
        return {"bytes": b * (min(taps * 32, n * 8) + 60 * k),
                "flops": b * (8 * taps + sum((2 * p + e) * 5 * B * math.log2(B) for B, _, p, e in rounds))}
    if case["kind"] == "mixed":
        per = [exact(1 << m, k, 1e-6, 0.5, 8, 32) for m, k in _request_types(case)]
        return {"bytes": sum(p[0] for p in per), "flops": sum(p[1] for p in per)}
    elem = 16 if case.get("fp64") else 8
    by, fl = exact(1 << case["m"], case["k"], case.get("delta", 1e-6), case["alpha0"], elem,
                   8 if case["kind"] == "channels" else 32)
    return {"bytes": b * by, "flops": b * fl}


# ---- inputs ------------------------------------------------------------------------------------
def _outputs(batch, cap):
    return (torch.zeros((batch, cap), dtype=torch.int32, device="cuda"),
            torch.zeros((batch, cap, 2), dtype=torch.float64, device="cuda"),
            torch.zeros((batch,), dtype=torch.int32, device="cuda"),
            torch.zeros((batch,), dtype=torch.int32, device="cuda"))


def _seeds(seed, count):
    return [int(s) for s in np.random.Generator(np.random.Philox(key=[int(seed), 41])).integers(1, 1 << 62, size=count)]


def _params(case, m, k):
    p = sfft.sfft_params_default(1 << m, k, GENERAL if case["kind"] == "general" else EXACT)
    if case["kind"] in ("exact", "channels"):
        p.alpha0 = case["alpha0"]
    if case["kind"] == "exact":
        p.delta, p.chunk_taps = case["delta"], case["taps"]
        p.precision = sfft.SFFT_FP64 if case["fp64"] else sfft.SFFT_FP32
    return p


def _signals(case, seed):
    """The case's input: [batch, n], [n, channels], or a list of signals."""
    if case["kind"] == "mixed":
        return [workloads.sparse_signal_device(1 << m, k, s, "cuda")[0]
                for (m, k), s in zip(_request_types(case), _seeds(seed, case["batch"]))]
    n, k, seeds = 1 << case["m"], case["k"], _seeds(seed, case["batch"])
    if case["kind"] == "general":
        x = torch.empty((case["batch"], n), dtype=torch.complex64, device="cuda")
        for r, s in enumerate(seeds):
            x[r] = workloads.sparse_signal_device(n, k, s, "cuda", snr_db=20.0)[0]
        return x
    chunk = max(1, min(16, (1 << 26) // n))
    if case["kind"] == "channels":
        return workloads.exact_sparse_channels_device(n, k, seeds, "cuda", chunk=chunk)[0]
    dtype = torch.complex128 if case["fp64"] else torch.complex64
    return workloads.exact_sparse_batch_device(n, k, seeds, "cuda", chunk=chunk, dtype=dtype)[0]


def prepare(case, seed):
    """A program's plan, its signals on the GPU and the arrays for the results."""
    st = {"kind": case["kind"], "x": _signals(case, seed), "seed": int(seed) + 1}
    if case["kind"] == "mixed":
        types = _types(case)
        plans = [sfft.Plan(_params(case, m, k), 1) for m, k in types]
        st["plan"] = sfft.BatchPlan(plans, case["batch"])
        of = [r % len(types) for r in range(case["batch"])]
        st["tables"] = st["plan"].prepare(of, st["x"], [st["seed"]] * case["batch"], range(case["batch"]))
        st["cap"] = max(p.params.z_cap for p in plans)
    else:
        p = _params(case, case["m"], case["k"])
        st["plan"] = sfft.Plan(p, case["batch"])
        st["cap"] = p.z_cap
    st["outputs"] = _outputs(case["batch"], st["cap"])
    return st


def run(st):
    if st["kind"] == "channels":
        return sfft.sfft_execute_channels(st["plan"], st["x"], st["seed"], 0, st["cap"], outputs=st["outputs"])
    if st["kind"] == "mixed":
        return st["plan"].execute_prepared(st["tables"], st["cap"], st["outputs"])
    return sfft.sfft_execute(st["plan"], st["x"], st["seed"], st["cap"], outputs=st["outputs"])


# ---- 64-bit results ----------------------------------------------------------------------------
def exact(case, seed):
    """The spectrum's coefficients above Algorithm 1's threshold 1/2, from a dense transform in 64 bits.
    None for the general algorithm, whose estimates of noisy coefficients have no closed form, and for
    dense supports (k > n / 1024), which Algorithm 1 recovers with constant probability only: a missed
    coefficient shifts all that follow it."""
    if case["kind"] == "general":
        return None
    types = _request_types(case) if case["kind"] == "mixed" else [(case["m"], case["k"])] * case["batch"]
    if any(k << 10 > 1 << m for m, k in types):
        return None
    x = _signals(case, seed)
    cap = max(max(64, 4 * k) for _, k in types)
    idx, val, count, flag = _outputs(case["batch"], cap)
    for r in range(case["batch"]):
        row = x[:, r] if case["kind"] == "channels" else x[r]
        X = torch.fft.fft(row.to(torch.complex128))
        at = torch.nonzero(X.abs() > 0.5).flatten()[:cap]
        idx[r, :at.numel()] = at.to(torch.int32)
        val[r, :at.numel()] = torch.view_as_real(X[at])
        count[r] = at.numel()
    return idx, val, count, flag
