"""Timed cases of the quench library, each through the entry points that a user's program calls.

Kinds (key "kind"):
  quench   T = infinity start, sweeps to log-spaced times, a full record at each, the final state:
           the library's ordinary run (R lattices in one context, default kernel choice).
  segment  n sweeps between two measurements of one large lattice and its checkpoint, with the
           whole-sweep kernel that the autotuner picks for such sizes.
  measure  one full measurement (M, B, D_a(r) on three axes, e, m, l_E, l_C) of a coarsened state.
  radial   radially averaged C(r) and S(k) of a coarsened state.
  batch    lattice classes of uneven size through the batched form's schedule call.
  serve    the continuous-batching server on a short list of requests.

A context's work is enqueued on one stream of this module, as in a program that runs its quenches
one after the other (the server gives each request a stream of its own).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2305_12161_gb300 import inputs, ising, serve

_streams: dict[int, torch.cuda.Stream] = {}


def _stream() -> torch.cuda.Stream:
    dev = torch.cuda.current_device()
    if dev not in _streams:
        _streams[dev] = torch.cuda.Stream()
    return _streams[dev]


def listed() -> list[dict]:
    return [
        # the smallest instance, byte-per-spin form, 1000 MCS with 20 log-spaced records: launches
        {"name": "quench_L32_plain", "kind": "quench", "L": 32, "R": 1, "t_max": 1000, "K": 20, "form": 1, "cycle": 0},
        # the serving mix's smallest size at a middling replica count
        {"name": "quench_L64_R12", "kind": "quench", "L": 64, "R": 12, "t_max": 256, "K": 8, "form": 0, "cycle": 0},
        # the same at the next size
        {"name": "quench_L128_R6", "kind": "quench", "L": 128, "R": 6, "t_max": 256, "K": 8, "form": 0, "cycle": 0},
        # eight L = 256 replicas: the paper's histogram size, sweeps and records in proportion
        {"name": "quench_L256_R8", "kind": "quench", "L": 256, "R": 8, "t_max": 256, "K": 8, "form": 0, "cycle": 0},
        # a size that is no multiple of 128, rows of an odd number of words, mixed cycle
        {"name": "quench_L320_R2_mixed", "kind": "quench", "L": 320, "R": 2, "t_max": 128, "K": 6, "form": 0, "cycle": 1},
        # the largest class of the mixed-size batch as a context of its own
        {"name": "quench_L512_R4", "kind": "quench", "L": 512, "R": 4, "t_max": 256, "K": 6, "form": 0, "cycle": 0},
        # the largest serving size, resumed from a checkpoint of a coarsened state
        {"name": "segment_L1024_R2", "kind": "segment", "L": 1024, "R": 2, "n": 32, "start": "domains", "cycle": 0},
        # the largest lattice from its T = infinity start: the headline sweep
        {"name": "segment_L2048", "kind": "segment", "L": 2048, "R": 1, "n": 24, "start": "random", "cycle": 0},
        # one full measurement of the largest lattice
        {"name": "measure_L2048", "kind": "measure", "L": 2048, "R": 1},
        # the paper's own correlation measurement, single precision
        {"name": "radial_L512", "kind": "radial", "L": 512, "precision": 0},
        # the mixed-size batch: sweeps and records as one graph
        {"name": "batch_mix", "kind": "batch", "classes": "64x512 128x64 256x16 512x4", "t_max": 100, "K": 5},
        # short requests served together
        {"name": "serve_8", "kind": "serve", "requests": 8, "sizes": "64 128 256 512", "t_lo": 2.0, "t_hi": 3.0, "R": 6},
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["quench", "quench", "quench", "quench", "segment", "measure", "radial", "batch", "serve"])
    if kind == "quench":
        L = rng.choice([16, 32, 64, 64, 128, 128, 192, 256, 256, 320, 384, 448, 512, 512, 576])
        R = _log_int(rng, 1, 24 if L <= 256 else 6)
        K = rng.randint(3, 10)
        return {"kind": kind, "L": L, "R": R, "t_max": max(K, _log_int(rng, 24, 512 if L <= 128 else 256)), "K": K,
                "form": 1 if L <= 128 and rng.random() < 0.15 else 0, "cycle": 1 if rng.random() < 0.25 else 0}
    if kind == "segment":
        L = rng.choice([256, 512, 1024, 1024, 2048])
        R = rng.randint(1, 4) if L < 2048 else 1
        return {"kind": kind, "L": L, "R": R, "n": _log_int(rng, 3, 20), "start": rng.choice(["random", "domains"]),
                "cycle": 1 if rng.random() < 0.25 else 0}
    if kind == "measure":
        L = rng.choice([64, 128, 192, 256, 384, 512, 640, 768, 1024, 1536])
        return {"kind": kind, "L": L, "R": rng.randint(1, 8) if L <= 512 else 1}
    if kind == "radial":
        return {"kind": kind, "L": rng.choice([64, 128, 256, 256, 320, 384]), "precision": rng.randint(0, 1)}
    if kind == "batch":
        sizes = sorted(rng.sample([32, 64, 128, 192, 256, 512], 3))
        cl = " ".join("%dx%d" % (L, max(1, _log_int(rng, 1, 64) * 64 // max(64, L))) for L in sizes)
        return {"kind": kind, "classes": cl, "t_max": _log_int(rng, 16, 100), "K": rng.randint(2, 5)}
    return {"kind": kind, "requests": rng.randint(3, 8), "sizes": rng.choice(["64 128", "64 128 256", "128 256 512"]),
            "t_lo": 1.5, "t_hi": 2.5, "R": rng.randint(2, 6)}


# ---- inputs -------------------------------------------------------------------------------
def _domains(L: int, seed: int) -> torch.Tensor:
    """Packed words [2, L, L, L/64] (int32) of a coarsened state: cells of 8^3 equal spins of random
    sign, shifted along y and z, and one spin in 64 reversed."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    W, c = L // 64, L // 8
    cells = torch.randint(0, 256, (c, c, W), generator=g, device="cuda", dtype=torch.int64)
    word = torch.zeros_like(cells)
    for i in range(8):  # a cell is four consecutive sites of each sublattice
        word |= ((cells >> i) & 1) * (15 << (4 * i))
    word = torch.where(word >= 2**31, word - 2**32, word).to(torch.int32)
    dy, dz = (int(v) for v in torch.randint(0, 8, (2,), generator=g, device="cuda").tolist())
    word = word.repeat_interleave(8, 0).repeat_interleave(8, 1).roll((dz, dy), (0, 1))
    out = torch.empty((2, L, L, W), dtype=torch.int32, device="cuda")
    for q in range(2):
        for z0 in range(0, L, 256):
            z1 = min(L, z0 + 256)
            flip = None
            for _ in range(6):
                r = torch.randint(-2**31, 2**31, (z1 - z0, L, W), generator=g, device="cuda", dtype=torch.int32)
                flip = r if flip is None else flip.bitwise_and_(r)
            out[q, z0:z1] = word[z0:z1] ^ flip
    return out


def _spins(words: torch.Tensor, L: int) -> torch.Tensor:
    """+1 / -1 spins [z, y, x] (int8) of packed words [2, L, L, L/64]."""
    out = torch.empty((L, L, L), dtype=torch.int8, device=words.device)
    sh = torch.arange(32, device=words.device, dtype=torch.int32)
    y = torch.arange(L, device=words.device)
    for z in range(L):
        bits = (((words[:, z].unsqueeze(-1) >> sh) & 1) * 2 - 1).to(torch.int8).reshape(2, L, L // 2)
        odd = ((y + z) & 1).bool().unsqueeze(-1)
        v = out[z].reshape(L, L // 2, 2)
        v[..., 0] = torch.where(odd, bits[1], bits[0])
        v[..., 1] = torch.where(odd, bits[0], bits[1])
    return out


def _classes(case: dict, seed: int) -> list[tuple]:
    out, s = [], int(seed) * 1000 + 1
    for item in case["classes"].split():
        L, R = (int(v) for v in item.split("x"))
        out.append((L, R, s))
        s += R
    return out


def _requests(case: dict, seed: int) -> list:
    rng = np.random.default_rng(int(seed))
    sizes = [int(v) for v in case["sizes"].split()]
    # sizes and durations spread over their ranges whatever the seed; the lattices' seeds differ
    n = case["requests"]
    return [serve.Request(id=i, L=sizes[i % len(sizes)],
                          t_max=int(round(10 ** (case["t_lo"] + (case["t_hi"] - case["t_lo"]) * ((i * 5) % n) / n))),
                          replicas=1 + (i * 3) % case["R"], seed=int(rng.integers(1, 2**31)), arrival_s=0.0, K=6)
            for i in range(n)]


class _State:
    pass


def prepare(case: dict, seed: int):
    st = _State()
    st.case, st.seed, kind = case, int(seed) * 64 + 1, case["kind"]
    if kind in ("quench", "segment", "measure", "radial"):
        L, R = case["L"], case.get("R", 1)
        kw = dict(stream=_stream())
        if kind == "quench":
            kw.update(form=case["form"], cycle=case["cycle"])
        if kind == "segment":  # what the autotuner picks at L = 2048, given as explicit options
            kw.update(variant=ising.VARIANT_ZFUSE, tile_z=64, depth=26, cycle=case["cycle"])
        st.ctx = ising.Ising(L, replicas=R, seed=st.seed, **kw)
        if kind in ("quench", "segment"):
            st.words = torch.empty((R, ising.ising_packed_words(L)), dtype=torch.int32, device="cuda")
        if kind == "quench":
            st.times = inputs.log_schedule(case["t_max"], case["K"])
            st.rec = torch.empty((case["K"], R, st.ctx.record_len), dtype=torch.int64, device="cuda")
        if kind == "segment":
            st.start = None
            if case["start"] == "domains":
                st.start = [_domains(L, st.seed + r) for r in range(R)]
        if kind in ("measure", "radial"):
            torch.cuda.synchronize()
            for r in range(R):
                w = _domains(L, st.seed + r)
                torch.cuda.synchronize()
                st.ctx.set_packed(w, replica=r, device=True)
                st.ctx.sync()
        if kind == "measure":
            st.rec = torch.empty((R, st.ctx.record_len), dtype=torch.int64, device="cuda")
            st.der = torch.empty((R, 4), dtype=torch.float64, device="cuda")
        st.ctx.sync()
    elif kind == "batch":
        st.batch = ising.Batch(_classes(case, seed), stream=_stream())
        # what the autotuner settles on for the mixed-size batch
        st.batch.set_weights(0.4, 1.0)
        st.batch.set_overlap(True)
        st.times = inputs.log_schedule(case["t_max"], case["K"])
        st.rec = torch.empty((case["K"], st.batch.record_words), dtype=torch.int64, device="cuda")
    else:
        st.requests = _requests(case, seed)
    return st


def run(st):
    case, kind = st.case, st.case["kind"]
    if kind == "quench":
        q, t = st.ctx, 0
        q.reinit(st.seed)
        for k, tk in enumerate(st.times):
            q.sweep(tk - t)
            t = tk
            q.measure_device(st.rec[k])
        for r in range(case["R"]):
            q.get_packed(r, out=st.words[r], device=True)
        return {"state": st.words, "records": st.rec}
    if kind == "segment":
        q = st.ctx
        if st.start is None:
            q.reinit(st.seed)
        else:
            for r, w in enumerate(st.start):
                q.set_packed(w, replica=r, device=True)
            q.t = 1000
        q.sweep(case["n"])
        for r in range(case["R"]):
            q.get_packed(r, out=st.words[r], device=True)
        return {"state": st.words}
    if kind == "measure":
        st.ctx.measure_device(st.rec, st.der)
        return {"records": st.rec, "derived": st.der}
    if kind == "radial":
        # not returned: in single precision the count of inexact lags is a count of rounding noise
        r = st.ctx.measure_radial(0, precision=case["precision"])
        return {"C": r["C"], "S": r["S"], "count": r["count"], "ell": r["ell"]}
    if kind == "batch":
        st.batch.reinit()
        st.batch.run(st.times, rec=st.rec, device=True)
        return {"records": st.rec}
    srv = serve.QuenchServer(tune=False)
    done = sorted(srv.run(st.requests), key=lambda r: r.request.id)
    return {"records": [r.records for r in done], "derived": [r.derived for r in done]}


# ---- what a pass cannot do without --------------------------------------------------------
_OPS_PER_128 = 90  # 32-bit operations of 128 spin updates: one Philox4x32-10 draw and the majority logic


def _rec_bytes(L: int) -> int:
    return 8 * (3 + 3 * (L // 2 + 1))


def _sweep_ops(L: int, R: int, n: int) -> float:
    return float(n) * R * L**3 / 128 * _OPS_PER_128


def _measure_ops(L: int, R: int) -> float:
    return 3.0 * R * L**3 * 5 * math.log2(L)  # the three axes' autocorrelations by transforms


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind == "quench":
        L, R, K = case["L"], case["R"], case["K"]
        return {"bytes": R * (L**3 / 8 + K * _rec_bytes(L)),
                "flops": _sweep_ops(L, R, case["t_max"]) + K * _measure_ops(L, R)}
    if kind == "segment":
        L, R = case["L"], case["R"]
        ends = 2 if case["start"] == "domains" else 1
        return {"bytes": R * L**3 / 8 * ends, "flops": _sweep_ops(L, R, case["n"])}
    if kind == "measure":
        L, R = case["L"], case["R"]
        return {"bytes": R * (L**3 / 8 + _rec_bytes(L) + 32), "flops": _measure_ops(L, R)}
    if kind == "radial":
        L = case["L"]
        return {"bytes": L**3 / 8 + 24 * math.sqrt(3) * L / 2, "flops": 2 * 2.5 * L**3 * 3 * math.log2(L)}
    if kind == "batch":
        cl = _classes(case, 0)
        return {"bytes": sum(R * (L**3 / 8 + case["K"] * _rec_bytes(L)) for L, R, _ in cl),
                "flops": sum(_sweep_ops(L, R, case["t_max"]) + case["K"] * _measure_ops(L, R) for L, R, _ in cl)}
    rq = _requests(case, 0)
    return {"bytes": sum(r.replicas * (r.L**3 / 8 + r.K * (_rec_bytes(r.L) + 32)) for r in rq),
            "flops": sum(_sweep_ops(r.L, r.replicas, r.t_max) + r.K * _measure_ops(r.L, r.replicas) for r in rq)}


# ---- the same in 64 bits by plain torch ---------------------------------------------------
def _axis_sums(s: torch.Tensor, dim: int) -> torch.Tensor:
    """sum_i s_i s_(i + r e) for r = 0 .. L/2 along `dim`, through float64 transforms."""
    L = s.shape[0]
    other = (dim + 1) % 3
    step = max(1, min(L, 2**26 // (L * L)))
    power = torch.zeros(L // 2 + 1, dtype=torch.float64, device=s.device)
    for a in range(0, L, step):
        part = s.narrow(other, a, min(step, L - a)).movedim(dim, 2).to(torch.float64)
        f = torch.fft.rfft(part, dim=2)
        power += (f.real**2 + f.imag**2).sum((0, 1))
    return torch.round(torch.fft.irfft(power, n=L)[: L // 2 + 1])


def _exact_derived(words: torch.Tensor, L: int) -> torch.Tensor:
    s = _spins(words, L)
    N = float(L) ** 3
    G = sum(_axis_sums(s, d) for d in range(3))
    C = (G / (3 * N)).cpu().numpy()
    M = float(s.sum(dtype=torch.int64))
    B = float((3 * N - G[1]) / 2)  # broken bonds: lag 1 of the three axes
    ell = math.nan
    for r in range(L // 2):
        if C[r] >= 0.5 > C[r + 1]:
            ell = r + (C[r] - 0.5) / (C[r] - C[r + 1])
            break
    return torch.tensor([-3 + 2 * B / N, M / N, N / B if B else math.inf, ell], dtype=torch.float64)


def _exact_radial(words: torch.Tensor, L: int) -> dict:
    s = _spins(words, L).to(torch.float64)
    N = float(L) ** 3
    f = torch.fft.fftn(s)
    del s
    P = f.real**2 + f.imag**2
    G = torch.round(torch.fft.ifftn(P).real)
    j = torch.arange(L, device=P.device)
    j = torch.where(j <= L // 2, j, j - L)
    D = (j * j).view(L, 1, 1) + (j * j).view(1, L, 1) + (j * j).view(1, 1, L)
    b = torch.round(torch.sqrt(D.to(torch.float64))).to(torch.int64).reshape(-1)
    count = torch.bincount(b)
    C = torch.zeros(len(count), dtype=torch.float64, device=P.device).index_add_(0, b, G.reshape(-1)) / (N * count)
    S = torch.zeros(len(count), dtype=torch.float64, device=P.device).index_add_(0, b, P.reshape(-1)) / (N * count)
    c = C.cpu().numpy()
    ell = math.nan
    for r in range(L // 2):
        if c[r] >= 0.5 > c[r + 1]:
            ell = r + (c[r] - 0.5) / (c[r] - c[r + 1])
            break
    return {"C": c, "S": S.cpu().numpy(), "count": None, "ell": float(ell)}


def exact(case: dict, seed: int):
    kind, s = case["kind"], int(seed) * 64 + 1
    if kind == "measure":
        L = case["L"]
        der = torch.stack([_exact_derived(_domains(L, s + r), L) for r in range(case["R"])])
        return {"records": None, "derived": der}
    if kind == "radial":
        return _exact_radial(_domains(case["L"], s), case["L"])
    return None  # whole numbers, or (server) derived values of states that only a whole quench gives
