"""The work that users of this library have it do, as cases that can be timed and compared.

Kinds of case:

layers     a compressed state that a program has in hand (prepared by the first part of a
           circuit) is advanced by the next part and read out: the long-running simulation
whole      a handle is reset, a whole circuit runs on it from |0...0> and one basis state is
           measured: the serving loop, where latency and launches count
batch      many handles of uneven size are reset and run their circuits in shared launches
codec      the device encoder and decoder on caller buffers (write a trace, read it back)
readout    measurement, a ragged range of amplitudes and the fidelity against a reference
sv         the uncompressed state vector under a random-circuit layer

Circuits come from the package's generators (random circuits, QAOA MaxCut, QFT, Grover),
bounds from the sweep 1e-5 / 1e-4 / 1e-3 / lossless, chunks from 2^8 to 2^11 amplitudes.
Images, and so decoded amplitudes and byte counts, are fixed bit for bit by the format.
"""
import math
import random

import numpy as np
import torch

from paper_1911_04034_gb300 import circuits as Cc
from paper_1911_04034_gb300 import qcsim

EXACT_MAX_N = 24  # largest register that exact() follows with a plain state vector


def listed():
    return [
        # the benchmark's workload: one layer of the 5x6 random circuit at 30 qubits (16 GiB
        # uncompressed) on a dense lossy state
        dict(name="rcs30", kind="layers", family="rcs", n=30, chunk=10, eps=1e-4, ladder=0, depth=4, layers=1, selector=0),
        # QAOA p=2 under the guarded ladder: the second cost-and-mixer round (CNOTs, RZ, RX)
        dict(name="qaoa26", kind="layers", family="qaoa", n=26, chunk=10, eps=1e-4, ladder=2, depth=1, layers=1, selector=0),
        # an ordinary register with an odd qubit count, smaller chunks and a loose bound
        dict(name="rcs21", kind="layers", family="rcs", n=21, chunk=9, eps=1e-3, ladder=0, depth=4, layers=2, selector=0),
        # the lossless stage: 64-bit values all the way
        dict(name="rcs23_lossless", kind="layers", family="rcs", n=23, chunk=10, eps=0.0, ladder=0, depth=3, layers=1, selector=0),
        # Grover with every mode tried on every chunk (Solution D and the palette): the
        # setting for the least memory, and what writes selector training data
        dict(name="grover22_trials", kind="layers", family="grover", n=22, chunk=10, eps=1e-4, ladder=0, depth=1, layers=1, selector=1),
        # Grover search, 12 qubits, blocks of 2^8 amplitudes, 50 iterations: the smallest
        # states, where every gate is a launch
        dict(name="grover12", kind="whole", family="grover", n=12, chunk=8, eps=1e-4, ladder=0, depth=50, selector=0),
        # one circuit of the batch workload's kind by itself, end to end
        dict(name="rcs14", kind="whole", family="rcs", n=14, chunk=9, eps=1e-4, ladder=0, depth=12, selector=0),
        # QFT of a random basis state with the paper's ladder: starts sparse, ends dense
        dict(name="qft18", kind="whole", family="qft", n=18, chunk=10, eps=1e-4, ladder=1, depth=1, selector=0),
        # independent random circuits of uneven size in shared launches under a graph
        dict(name="batch16", kind="batch", count=16, n_lo=14, n_hi=20, d_lo=12, d_hi=24, chunk=9, eps=1e-4),
        # the codec alone, 1 GiB of amplitudes at the default bound
        dict(name="codec26", kind="codec", n=26, chunk=10, eps=1e-4),
        # readout of a state in hand
        dict(name="readout26", kind="readout", n=26, chunk=10, eps=1e-4),
        # the uncompressed comparator
        dict(name="sv27", kind="sv", n=27),
    ]


def draw(rng):
    kind = rng.choice(["layers", "layers", "layers", "layers", "whole", "whole", "batch", "codec", "readout", "sv"])
    eps = rng.choice([1e-5, 1e-4, 1e-4, 1e-3, 0.0])
    chunk = rng.choice([8, 9, 10, 10, 11])
    if kind == "layers":
        family = rng.choice(["rcs", "rcs", "qaoa", "grover"])
        n = rng.randint(13, 27 if eps else 24)
        if family == "qaoa":
            n -= n % 2  # 3-regular graphs have an even number of vertices
        selector = rng.choice([0, 0, 0, 1]) if n <= 22 else 0
        return dict(kind=kind, family=family, n=n, chunk=chunk, eps=eps, ladder=rng.choice([0, 1, 2]),
                    depth=1 if family != "rcs" else rng.randint(2, 5), layers=1 if family == "qaoa" else rng.randint(1, 2),
                    selector=selector)
    if kind == "whole":
        family = rng.choice(["rcs", "qft", "grover"])
        n = rng.randint(9, 19)
        depth = {"rcs": rng.randint(6, 20), "qft": 1, "grover": rng.randint(2, 20)}[family]
        return dict(kind=kind, family=family, n=n, chunk=min(chunk, n - 2), eps=eps, ladder=rng.choice([0, 1]), depth=depth,
                    selector=0)
    if kind == "batch":
        lo = rng.randint(11, 15)
        return dict(kind=kind, count=rng.randint(3, 24), n_lo=lo, n_hi=lo + rng.randint(2, 5), d_lo=8, d_hi=rng.randint(9, 20),
                    chunk=rng.choice([8, 9, 10]), eps=eps)
    if kind == "codec":
        return dict(kind=kind, n=rng.randint(14, 26), chunk=chunk, eps=eps)
    if kind == "readout":
        return dict(kind=kind, n=rng.randint(15, 26), chunk=chunk, eps=eps or 1e-4)
    return dict(kind="sv", n=rng.randint(10, 27))


# ------------------------------------------------------------------ inputs -- #


def _rcs_edges(n):
    cols = int(math.ceil(math.sqrt(n))) if n != 30 else 6
    return int(math.ceil(n / cols)) if n != 30 else 5, cols


def _gates(case, seed):
    """(gates that prepare the state, gates of the pass)."""
    n, family = case["n"], case["family"]
    if family == "rcs":
        rows, cols = _rcs_edges(n)
        d = case["depth"]
        g = Cc.rcs(rows, cols, d + case.get("layers", 0), seed, n=n)
        return (g[: Cc.rcs(rows, cols, d, seed, n=n).shape[0]] if "layers" in case else g), g
    if family == "qaoa":
        g, edges = Cc.qaoa_maxcut(n, 2, 3, seed)
        return g[: n + 3 * len(edges) + n], g
    if family == "qft":
        g, _ = Cc.qft(n, seed)
        return g, g
    g, _ = Cc.grover(n, case["depth"] + case.get("layers", 0), seed)
    return (g[: n + (4 * n + 2) * case["depth"]] if "layers" in case else g), g


def _sim(n, chunk, eps, ladder):
    raw = 16 << n
    return qcsim.Sim(n, max(chunk, min(20, n - 4)), eps, chunk_log2=chunk, budget=raw // 4 if eps else raw + raw // 8,
                     ladder=ladder, pool_bytes=raw + raw // 8 + (64 << 20))


def _dense(n, seed, device="cuda"):
    """A normalised Gaussian state of 2^n amplitudes (2^(n+1) doubles): what deep random
    circuits leave."""
    gen = torch.Generator(device=device)
    gen.manual_seed(seed)
    x = torch.randn(2 << n, generator=gen, dtype=torch.float64, device=device)
    return x / x.norm()


def _measure_seed(seed):
    return (seed * 2654435761 + 12345) & 0xFFFFFFFF


def _batch(case, seed):
    """(qubits, gates) of every circuit; the sizes belong to the case, the gates to the seed."""
    sizes = random.Random(1000 * case["count"] + case["n_hi"])
    return [(n, Cc.rcs_n(n, sizes.randint(case["d_lo"], case["d_hi"]), seed % 1000003 + 7919 * k))
            for k, n in enumerate(sizes.randint(case["n_lo"], case["n_hi"]) for _ in range(case["count"]))]


def _range(case):
    """A ragged range of amplitudes: (first, count)."""
    r, n = random.Random(case["n"]), 1 << case["n"]
    return r.randrange(n // 3), n // 3 + r.randrange(n // 3)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case, seed=seed)
    if kind in ("layers", "readout"):
        c = case if kind == "layers" else dict(case, family="rcs", depth=3, layers=0, ladder=0, selector=0)
        first, whole = _gates(c, seed)
        s = _sim(case["n"], case["chunk"], case["eps"], c["ladder"])
        if c["selector"]:
            s.set_selector(c["selector"])
        s.apply_circuit(first)
        st.update(sim=s, gates=whole[first.shape[0]:])
        if kind == "layers":
            st["out"] = torch.empty(2 << case["n"], dtype=torch.float64, device="cuda")
        else:
            st["ref"] = _dense(case["n"], seed)
            st["first"], st["count"] = _range(case)
            st["out"] = torch.empty(2 * st["count"], dtype=torch.float64, device="cuda")
    elif kind == "whole":
        st.update(sim=_sim(case["n"], case["chunk"], case["eps"], case["ladder"]), gates=_gates(case, seed)[1],
                  out=torch.empty(2 << case["n"], dtype=torch.float64, device="cuda"))
    elif kind == "batch":
        circ = _batch(case, seed)
        st.update(sims=[_sim(n, case["chunk"], case["eps"], 0) for n, _ in circ], circuits=[g for _, g in circ],
                  outs=[torch.empty(2 << n, dtype=torch.float64, device="cuda") for n, _ in circ])
    elif kind == "codec":
        k = (1 << case["n"]) >> case["chunk"]
        stride = qcsim.codec_stride(case["chunk"])
        st.update(values=_dense(case["n"], seed), chunks=k, stride=stride,
                  back=torch.empty(2 << case["n"], dtype=torch.float64, device="cuda"))
    else:
        rows, cols = _rcs_edges(case["n"])
        sv = qcsim.StateVector(case["n"])
        sv.apply_circuit(Cc.rcs(rows, cols, 1, seed, n=case["n"]))
        st.update(sv=sv, gates=Cc.rcs(rows, cols, 2, seed, n=case["n"])[Cc.rcs(rows, cols, 1, seed, n=case["n"]).shape[0]:],
                  out=torch.empty(2 << case["n"], dtype=torch.float64, device="cuda"))
    return st


# -------------------------------------------------------------------- pass -- #


def _figures(s):
    d = s.stats()
    return [d["encoded_bytes"], d["max_encoded_bytes"], d["gates"], d["sig_bits_current"], d["peak_pages_bytes"]] + \
        d["chunks_by_mode"][:7]


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "layers":
        s = st["sim"]
        s.apply_circuit(st["gates"])
        return dict(amplitudes=s.amplitudes(out=st["out"]), figures=_figures(s))
    if kind == "whole":
        s = st["sim"]
        s.reset()
        s.apply_circuit(st["gates"])
        outcome, prob = s.measure(_measure_seed(st["seed"]))
        return dict(amplitudes=s.amplitudes(out=st["out"]), figures=_figures(s), outcome=outcome, prob=prob)
    if kind == "batch":
        for s in st["sims"]:
            s.reset()
        qcsim.batch_apply(st["sims"], st["circuits"])
        return dict(amplitudes=[s.amplitudes(out=o) for s, o in zip(st["sims"], st["outs"])],
                    figures=np.array([_figures(s) for s in st["sims"]], dtype=np.int64))
    if kind == "codec":
        images, lens, stride = qcsim.codec_encode(st["values"], case["chunk"], case["eps"])
        rc = qcsim.lib().sim_codec_decode(images.data_ptr(), stride, lens.data_ptr(), st["chunks"], case["chunk"],
                                          st["back"].data_ptr(), 1)
        if rc != qcsim.OK:
            raise RuntimeError("sim_codec_decode: %d" % rc)
        return dict(images=images, lens=lens, back=st["back"])
    if kind == "readout":
        s = st["sim"]
        outcome, prob = s.measure(_measure_seed(st["seed"]))
        f = s.fidelity(st["ref"])
        return dict(amplitudes=s.amplitudes(st["first"], st["count"], out=st["out"]), outcome=outcome, prob=prob, norm2=f["norm2"])
    st["sv"].apply_circuit(st["gates"])
    return st["sv"].amplitudes(out=st["out"])


# ------------------------------------------------------------ expectations -- #


def _sig_bits(eps):
    return 64 if eps == 0.0 else 12 - (math.frexp(eps)[1] - 1)


def _image_bytes(n, eps):
    """About what a dense state of 2^n amplitudes takes coded: 2 code bits a value and its S
    bits less the leading bytes shared with its predecessor (about half a byte)."""
    S = _sig_bits(eps)
    return (2 << n) * min(64.0, 2 + S - 3.5) / 8


def _flops(gates, n):
    """FP64 operations of the kept-term sums over every amplitude pair of every gate."""
    total = 0.0
    for g in gates:
        u = [float(x) for x in g["u"]]
        rows = ((u[0], -u[1], u[2], -u[3]), (u[0], u[1], u[2], u[3]), (u[4], -u[5], u[6], -u[7]), (u[4], u[5], u[6], u[7]))
        per = 0
        for r in rows:
            kept = [x for x in r if x != 0.0]
            per += 2 * len(kept) - 1 if kept and abs(kept[0]) != 1.0 else 2 * max(0, len(kept) - 1)
        total += per * 2.0 ** (n - 1 - bin(int(g["ctrl_mask"])).count("1"))
    return total


def work(case):
    kind = case["kind"]
    if kind in ("layers", "whole"):
        first, whole = _gates(case, 1)
        n = case["n"]
        code, raw = _image_bytes(n, case["eps"]), 16 << n
        if kind == "layers":  # the state read, written, and decoded once more for the readout
            return dict(bytes=3 * code + raw, flops=_flops(whole[first.shape[0]:], n))
        return dict(bytes=2 * code + raw, flops=_flops(whole, n))
    if kind == "batch":
        b = f = 0.0
        for n, g in _batch(case, 1):
            b += 2 * _image_bytes(n, case["eps"]) + (16 << n)
            f += _flops(g, n)
        return dict(bytes=b, flops=f)
    code, raw = _image_bytes(case["n"], case.get("eps", 0.0)), 16 << case["n"]
    if kind == "codec":
        return dict(bytes=2 * raw + 2 * code, flops=0)
    if kind == "readout":
        return dict(bytes=2.5 * code + 1.5 * raw, flops=11.0 * (1 << case["n"]))
    rows, cols = _rcs_edges(case["n"])
    g = Cc.rcs(rows, cols, 2, 1, n=case["n"])[Cc.rcs(rows, cols, 1, 1, n=case["n"]).shape[0]:]
    return dict(bytes=4 * raw, flops=_flops(g, case["n"]))


def tolerance(case):
    # images and decoded values are fixed to the bit; a probability and a norm are sums of
    # 2^n doubles in any order
    if case["kind"] in ("whole", "readout"):
        return dict(rel=1e-12, max=1e-11, differ=0.0)
    return "exact"


def _plain(gates, n):
    """The state vector after the gates, from |0...0>, as 2^(n+1) doubles."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=dev)
    psi[0] = 1.0
    idx = torch.arange(1 << n, device=dev)
    for g in gates:
        t, cm, cv = int(g["target"]), int(g["ctrl_mask"]), int(g["ctrl_vals"])
        u = [float(x) for x in g["u"]]
        v = psi.view(-1, 2, 1 << t)
        a, b = v[:, 0, :], v[:, 1, :]
        na = complex(u[0], u[1]) * a + complex(u[2], u[3]) * b
        nb = complex(u[4], u[5]) * a + complex(u[6], u[7]) * b
        if cm:
            on = ((idx & cm) == cv).view(-1, 2, 1 << t)[:, 0, :]
            na, nb = torch.where(on, na, a), torch.where(on, nb, b)
        psi = torch.stack((na, nb), dim=1).reshape(-1)
    return torch.view_as_real(psi).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "codec":
        v = _dense(case["n"], seed)
        S = _sig_bits(case["eps"])
        bits = v.view(torch.int64) & (-1 << (64 - S))
        return dict(images=None, lens=None, back=bits.view(torch.float64))
    if kind == "batch":
        circ = _batch(case, seed)
        return dict(amplitudes=[_plain(g, n) for n, g in circ], figures=None)
    if case["n"] > EXACT_MAX_N:
        return None
    if kind == "sv":
        rows, cols = _rcs_edges(case["n"])
        return _plain(Cc.rcs(rows, cols, 2, seed, n=case["n"]), case["n"])
    if kind == "readout":
        psi = _plain(_gates(dict(case, family="rcs", depth=3, layers=0), seed)[0], case["n"])
        first, count = _range(case)
        return dict(amplitudes=psi[2 * first: 2 * (first + count)], outcome=None, prob=None, norm2=float(psi.square().sum()))
    psi = _plain(_gates(case, seed)[1], case["n"])
    out = dict(amplitudes=psi, figures=None)
    if kind == "whole":
        out.update(outcome=None, prob=None)
    return out
