"""Workloads of the FDAS library as a search program calls it, for timing and comparing builds.

A case names the form (``kind``) and its sizes.  Inputs follow the seeded recipe of the
benchmark: the Fourier bins of a real series of unit noise and a few chirps, the
constant-acceleration template bank (drifts z = -zmax .. zmax, 10 zmax + 1 taps), and for the
harmonic sums a plane of unit-exponential noise powers with a few harmonic trains.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1805_12280_gb300 as fd

PRECISIONS = {"fp32": fd.FDAS_PREC_FP32, "tc16": fd.FDAS_PREC_TC_FP16, "dft2": fd.FDAS_PREC_TC_DFT2}


def _plane(name, n, precision="fp32", seg_len=2048, zmax=42):
    return {"name": name, "kind": "plane", "n": n, "precision": precision, "seg_len": seg_len, "zmax": zmax}


def listed():
    return [
        # the small single array of the tests and the benchmark: one launch, latency counts
        _plane("plane_fp32_16384", 1 << 14),
        # a ragged trial in the middle of the range
        _plane("plane_fp32_301000", 301_000),
        # the SKA-sized array of the headline benchmark, default options
        _plane("plane_fp32_2p22", 1 << 22),
        # the shortest request of the served stream, tensor-core form
        _plane("plane_dft2_65536", 1 << 16, "dft2"),
        # the SKA-sized array, tensor-core form
        _plane("plane_dft2_2p22", 1 << 22, "dft2"),
        # dedispersion trials of uneven lengths in one call: short ones in FP32 ...
        {"name": "batch_fp32_16", "kind": "batch", "count": 16, "lo": 1 << 16, "hi": 1 << 20, "length_seed": 2001,
         "precision": "fp32", "zmax": 42},
        # ... and those of the batched benchmark's range in the tensor-core form
        {"name": "batch_dft2_24", "kind": "batch", "count": 24, "lo": 1 << 18, "hi": 1 << 22, "length_seed": 999,
         "precision": "dft2", "zmax": 42},
        # the search chain: candidates of an SKA-sized array at the 6-sigma power threshold 1 + 6
        {"name": "cand_dft2_2p22_t7", "kind": "candidates", "n": 1 << 22, "precision": "dft2", "threshold": 7.0, "zmax": 42},
        # the same in FP32 at the power whose exponential tail has the one-sided Gaussian 6-sigma
        # probability
        {"name": "cand_fp32_2p22_tg", "kind": "candidates", "n": 1 << 22, "precision": "fp32", "threshold": 20.74, "zmax": 42},
        # the stage after the plane: harmonic sums of an SKA-sized plane
        {"name": "harmonic8_2p22", "kind": "harmonic", "n": 1 << 22, "m": 85, "bin0": 210, "max_harm": 8},
        # the full-length frequency-domain FIR that overlap-save is weighed against
        {"name": "fdfir_2p22", "kind": "fdfir", "n": 1 << 22, "zmax": 42},
        # host array in, host plane out, pinned buffers (the end-to-end call of the benchmark)
        {"name": "host_fp32_2p20", "kind": "host", "n": 1 << 20, "precision": "fp32", "zmax": 42},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plane"] * 5 + ["batch"] * 2 + ["candidates"] * 2 + ["harmonic"] * 2 + ["fdfir", "host"])
    zmax = rng.choice([42, 42, 42, 21, 10])
    if kind == "plane":
        precision = rng.choice(["fp32", "fp32", "fp32", "dft2", "dft2", "tc16"])
        seg_len = rng.choice([2048, 2048, 1024, 4096]) if precision == "fp32" else 2048
        return {"kind": kind, "n": _log_uniform(rng, 1 << 14, 1 << 22), "precision": precision, "seg_len": seg_len, "zmax": zmax}
    if kind == "batch":
        lo = _log_uniform(rng, 1 << 16, 1 << 18)
        return {"kind": kind, "count": rng.randint(2, 24), "lo": lo, "hi": _log_uniform(rng, 1 << 19, 1 << 21),
                "length_seed": rng.randrange(1 << 20), "precision": rng.choice(["fp32", "dft2"]), "zmax": zmax}
    if kind == "candidates":
        precision = rng.choice(["fp32", "dft2"])
        threshold = 20.74 if precision == "fp32" else rng.choice([7.0, 20.74])
        return {"kind": kind, "n": _log_uniform(rng, 1 << 14, 1 << 22), "precision": precision, "threshold": threshold, "zmax": zmax}
    if kind == "harmonic":
        m = 2 * zmax + 1
        return {"kind": kind, "n": _log_uniform(rng, 1 << 14, 1 << 22), "m": m, "bin0": 5 * zmax, "max_harm": rng.choice([1, 4, 8, 8, 16, 32])}
    if kind == "fdfir":
        return {"kind": kind, "n": _log_uniform(rng, 1 << 18, 1 << 22), "zmax": zmax}
    return {"kind": kind, "n": _log_uniform(rng, 1 << 14, 1 << 20), "precision": rng.choice(["fp32", "dft2"]), "zmax": zmax}


@functools.lru_cache(maxsize=8)
def _bank(zmax):
    """complex64 [2 zmax + 1, 10 zmax + 1]: h_z[k] = conj(R_z(centre - k)) of unit energy, R_z by
    Gauss-Legendre quadrature of int_0^1 exp(2 pi i (-(q + z/2) t + z t^2 / 2)) dt."""
    centre = 5 * zmax
    t, w = np.polynomial.legendre.leggauss(1024)
    t, w = 0.5 * (t + 1.0), 0.5 * w
    h = np.zeros((2 * zmax + 1, 2 * centre + 1), dtype=np.complex128)
    for z in range(1, zmax + 1):
        q = np.arange(-5 * z, 5 * z + 1)
        r = np.exp(-2j * np.pi * np.outer(q, t)) @ (w * np.exp(2j * np.pi * (0.5 * z * t * t - 0.5 * z * t)))
        r /= np.sqrt(np.sum(np.abs(r) ** 2))
        h[zmax + z, centre - q] = np.conj(r)
        h[zmax - z, centre - q] = r[::-1]          # R_{-z}(q) = conj(R_z(-q))
    h[zmax, centre] = 1.0                          # z = 0: the delayed input
    return h.astype(np.complex64)


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _array(n, seed, zmax):
    """complex64 [n] on the GPU: bins 0 .. n-1 of 2n samples of unit noise and eight chirps."""
    rng = np.random.default_rng(10_000 + int(seed))
    s = torch.randn(2 * n, dtype=torch.float64, device="cuda", generator=_generator(seed))
    u = torch.arange(2 * n, dtype=torch.float64, device="cuda") / (2 * n)
    for _ in range(8):
        r, z = rng.uniform(0.05 * n, 0.95 * n), rng.integers(-zmax, zmax + 1)
        cycles = r * u + 0.5 * z * u * u
        s += 0.05 * torch.cos(2.0 * math.pi * (cycles - torch.floor(cycles)))
    return (torch.fft.rfft(s)[:n] / math.sqrt(2.0 * n)).to(torch.complex64)


def _noise_plane(case, seed):
    """float32 [m, n] on the GPU: unit-exponential powers and eight harmonic trains."""
    m, n, bin0, c = case["m"], case["n"], case["bin0"], (case["m"] - 1) // 2
    P = torch.empty((m, n), dtype=torch.float32, device="cuda").exponential_(generator=_generator(seed))
    rng = np.random.default_rng(20_000 + int(seed))
    for _ in range(8):
        r, z = int(rng.integers(1, max(2, (n - bin0) // 8))), int(rng.integers(-(c // 8), c // 8 + 1))
        for k in range(1, 9):
            if bin0 + k * r < n and abs(k * z) <= c:
                P[c + k * z, bin0 + k * r] += 12.0
    return P


def _lengths(case):
    rng = np.random.default_rng(case["length_seed"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [int(v) for v in np.rint(np.exp(rng.uniform(lo, hi, size=case["count"])))]


class State:
    """What a program holds between calls; its plan is freed with it."""

    def __init__(self, case, plan=None, **held):
        self.case, self.plan = case, plan
        self.__dict__.update(held)

    def __del__(self):
        if self.plan is not None:
            self.plan.close()


def _records(width, cells, threshold):
    """Record list with room for the noise crossings (a cell crosses with probability
    e^-threshold), the chirps' and, for the harmonic sums, the higher levels'; the counter, and the
    records' indices."""
    room = (1 << 16) + int(1.6 * cells * math.exp(-threshold))
    return {"buf": torch.empty((room, width), dtype=torch.int64, device="cuda"),
            "count": torch.empty(1, dtype=torch.int64, device="cuda"),
            "index": torch.arange(room, device="cuda")}


def prepare(case, seed):
    kind = case["kind"]
    if kind == "harmonic":
        return State(case, P=_noise_plane(case, seed), **_records(3, case["m"] * case["n"], 7.0))
    h = _bank(case["zmax"])
    m = h.shape[0]
    if kind == "batch":
        ns = _lengths(case)
        xs = [_array(n, 1000 * int(seed) + i, case["zmax"]) for i, n in enumerate(ns)]
        outs = [torch.empty((m, n), dtype=torch.float32, device="cuda") for n in ns]
        return State(case, fd.Plan(h, max(ns), precision=PRECISIONS[case["precision"]]), xs=xs, outs=outs)
    n = case["n"]
    x = _array(n, seed, case["zmax"])
    if kind == "fdfir":
        return State(case, fd.FdFir(h, n), x=x, out=torch.empty((m, n), dtype=torch.float32, device="cuda"))
    plan = fd.Plan(h, n, seg_len=case.get("seg_len", 2048), precision=PRECISIONS[case["precision"]])
    if kind == "candidates":
        return State(case, plan, x=x, **_records(2, m * n, case["threshold"]))
    if kind == "host":
        xh = torch.empty(n, dtype=torch.complex64, pin_memory=True)
        xh.copy_(x)
        out = torch.empty((m, n), dtype=torch.float32, pin_memory=True)
        return State(case, plan, xh=xh, x=xh.numpy(), outh=out, out=out.numpy())
    return State(case, plan, x=x, out=torch.empty((m, n), dtype=torch.float32, device="cuda"))


def _sorted_records(buf, count, index, n, level_rows=0):
    """The stored records in (level, template, bin) order, as the sifting stage takes them, the
    rest of the list filled up; on the device, without waiting for the count."""
    words = buf.view(torch.int32)
    row = words[:, 0]
    if level_rows:
        row = row + level_rows * torch.log2(words[:, 4].to(torch.float32)).to(torch.int32)
    found = index < count
    cell = torch.where(found, row * n + buf[:, 1].to(torch.int32), 2**31 - 1)   # levels x rows x n < 2^31
    cell, order = torch.sort(cell)
    return {"count": count, "cell": cell, "power": torch.where(found, words[:, 1].view(torch.float32), 0.0)[order]}


def run(state):
    case = state.case
    kind = case["kind"]
    if kind == "batch":
        return state.plan.convolve_batch(state.xs, outs=state.outs)
    if kind == "candidates":
        buf, count = state.plan.candidates(state.x, case["threshold"], buf=state.buf, count=state.count)
        return _sorted_records(buf, count, state.index, case["n"])
    if kind == "harmonic":
        buf, count = fd.harmonic_sum(state.P, case["bin0"], case["max_harm"], buf=state.buf, count=state.count)
        return _sorted_records(buf, count, state.index, case["n"], case["m"])
    if kind == "host":
        return state.plan.convolve_host(state.x, state.out)
    return state.plan.convolve(state.x, out=state.out)


def _ols_flops(n, m, k, seg_len=2048):
    """Operations of overlap-save with the forward transform shared by the m filters, and |y|^2."""
    levels = int(math.log2(seg_len))
    return -(-n // (seg_len - k + 1)) * seg_len * (m * (6 + 5 * levels) + 5 * levels) + 3 * m * n


def work(case):
    kind = case["kind"]
    if kind == "harmonic":
        m, n, c = case["m"], case["n"], (case["m"] - 1) // 2
        adds = sum((2 * (c // k) + 1) * max(0, (n - 1 - case["bin0"]) // k) for k in range(2, case["max_harm"] + 1))
        return {"bytes": 4 * m * n, "flops": adds}
    m, k = 2 * case["zmax"] + 1, 10 * case["zmax"] + 1
    ns = _lengths(case) if kind == "batch" else [case["n"]]
    seg_len = case.get("seg_len", 2048)
    if kind == "fdfir":
        n, p = case["n"], 1 << 21
        while p < n + k - 1:
            p *= 2
        return {"bytes": 8 * n + 4 * m * n + 8 * m * p, "flops": 5 * p * int(math.log2(p)) * (1 + m) + 6 * m * p + 3 * m * n}
    flops = sum(_ols_flops(n, m, k, seg_len) for n in ns)
    planes = 0 if kind == "candidates" else 4 * m * sum(ns)
    records = int(16 * m * sum(ns) * math.exp(-case["threshold"])) if kind == "candidates" else 0
    return {"bytes": 8 * sum(ns) + 8 * m * k + planes + records, "flops": flops}


def _exact_plane(x, h):
    """|x * h_z|^2 in 64 bits: full-length transforms."""
    n, k = x.numel(), h.shape[1]
    p = 1 << (n + k - 2).bit_length()
    X = torch.fft.fft(x.to(torch.complex128), p)
    out = torch.empty((h.shape[0], n), dtype=torch.float64, device=x.device)
    for z in range(h.shape[0]):
        y = torch.fft.ifft(X * torch.fft.fft(torch.from_numpy(h[z]).to(x.device).to(torch.complex128), p))[:n]
        out[z] = y.real * y.real + y.imag * y.imag
    return out


def _exact_harmonics(case, P):
    m, n, bin0, c = case["m"], case["n"], case["bin0"], (case["m"] - 1) // 2
    levels = fd.harmonic_levels(case["max_harm"])
    thresholds = [float(np.float32(t)) for t in fd.harmonic_thresholds(case["max_harm"])]
    cells, powers = [], []
    for y in range(m):
        z = y - c
        acc = None
        for k in range(1, case["max_harm"] + 1):
            last = (n - 1 - bin0) // k              # fundamentals r = 1 .. last
            if abs(k * z) > c or last < 1:
                break
            v = P[c + k * z, bin0 + k: bin0 + k * last + 1: k].to(torch.float64)
            acc = v if acc is None else acc[:last] + v
            if k in levels:
                r = torch.nonzero(acc > thresholds[levels.index(k)]).reshape(-1)
                cells.append((y + m * levels.index(k)) * n + bin0 + 1 + r)
                powers.append(acc[r])
    power = torch.zeros(_records(3, m * n, 7.0)["index"].numel(), dtype=torch.float64, device=P.device)
    if cells:
        _, order = torch.sort(torch.cat(cells))
        power[: order.numel()] = torch.cat(powers)[order]
    return power


def exact(case, seed):
    kind = case["kind"]
    if kind == "candidates":
        return None
    if kind == "harmonic":
        return {"count": None, "cell": None, "power": _exact_harmonics(case, _noise_plane(case, seed))}
    h = _bank(case["zmax"])
    if kind == "batch":
        return [_exact_plane(_array(n, 1000 * int(seed) + i, case["zmax"]), h) for i, n in enumerate(_lengths(case))]
    out = _exact_plane(_array(case["n"], seed, case["zmax"]), h)
    return out.cpu().numpy() if kind == "host" else out
