"""The streaming gate kernel (one warp pair per work item, values kept in registers from
decoder to encoder) against the oracle and against the general kernel.

Every gate of a lossy run at chunk sizes 2^7..2^11 goes through the streaming kernel
first; items it cannot finish as STREAM images go to the general kernel.  Both must give
the oracle's bytes.  The circuits cover every work-item kind of the streaming kernel:
cross-chunk targets, in-chunk targets 0-1 (partner in the lane), 2-6 (partner in another
lane of the warp), diagonal gates on any in-chunk target, in-chunk controls, and targets
7..kc-1 (partner in another pass).
"""
import numpy as np
import pytest

import oracle as O
from paper_1911_04034_gb300 import circuits as Cc

pytestmark = pytest.mark.gpu


def qc():
    from paper_1911_04034_gb300 import qcsim

    return qcsim


def all_images(s):
    return [s.chunk_image(c) for c in range(s.n_chunks)]


def every_target_circuit(n, seed):
    """A random layer to leave the lossless stage, then on every qubit a dense gate,
    T, a gate under an in-chunk control and CZ to the next qubit, in a seeded order."""
    rng = np.random.default_rng(seed)
    g = []
    for q in range(n):
        g.append(Cc.gate(q, Cc.H))
    for q in range(n):
        g.append(Cc.gate(q, [Cc.SX, Cc.SY, Cc.T][int(rng.integers(3))]))
    for q in rng.permutation(n):
        q = int(q)
        g.append(Cc.gate(q, Cc.SY))
        g.append(Cc.gate(q, Cc.T))
        c = (q + 3) % n
        g.append(Cc.gate(q, Cc.SX, {c: 1}))
        g.append(Cc.gate((q + 1) % n, Cc.Z, {q: 1}))
        g.append(Cc.gate(q, Cc.X, {(q + 5) % n: 0}))
    return Cc.to_array(g)


@pytest.mark.parametrize("kc,n", [(7, 12), (8, 13), (10, 14), (11, 14)])
def test_streaming_kernel_every_gate_bit_exact(kc, n):
    """Every gate's images equal the oracle's, with the streaming kernel on."""
    gates = every_target_circuit(n, seed=kc)
    eps = 1e-4
    budget = (16 << n) // 4
    orc = O.CSim(n, n, kc, eps, budget)
    gpu = qc().Sim(n, n, eps, chunk_log2=kc, budget=budget, pool_bytes=2 * (16 << n) + (64 << 20))
    for k in range(len(gates)):
        gpu.apply_gate(gates[k])
        orc.apply(gates[k])
        assert all_images(gpu) == [orc.image(c) for c in range(orc.nchunks)], f"gate {k} target {int(gates[k]['target'])}"
    st = gpu.stats()
    assert st["fast_items"] > 0
    assert st["encoded_bytes"] == orc.stats()["encoded_bytes"]


@pytest.mark.parametrize("eps", [1e-5, 1e-4, 1e-3])
@pytest.mark.parametrize("kc", [7, 9, 10])
def test_streaming_and_general_kernels_write_the_same_bytes(eps, kc):
    """Random circuit, QAOA, QFT and Grover: the same run with the streaming kernel on
    and off gives identical images, counters and amplitudes, and both the oracle's."""
    n = 14
    circuits = [Cc.rcs_n(n, 8, seed=3 + kc), Cc.qaoa_maxcut(n, 2, 3, seed=4)[0], Cc.qft(n, seed=5)[0],
                Cc.grover(n, 2, seed=6)[0]]
    for ci, gates in enumerate(circuits):
        budget = (16 << n) // 4
        sims = []
        for fast in (1, 0):
            s = qc().Sim(n, n, eps, chunk_log2=kc, budget=budget, pool_bytes=2 * (16 << n) + (64 << 20))
            s.set_option("fast_path", fast)
            sims.append(s)
        for k in range(0, len(gates), 17):
            for s in sims:
                s.apply_circuit(gates[k:k + 17])
            assert all_images(sims[0]) == all_images(sims[1]), (ci, k)
        a, b = (s.stats() for s in sims)
        for key in ("encoded_bytes", "max_encoded_bytes", "eps_switch_gate", "chunks_by_mode", "fidelity_lb_sum"):
            assert a[key] == b[key], key
        assert b["fast_items"] == 0
        if ci == 0:
            assert a["fast_items"] > 0
        orc = O.CSim(n, n, kc, eps, budget)
        orc.apply(gates)
        assert all_images(sims[0]) == [orc.image(c) for c in range(orc.nchunks)]
        assert np.array_equal(sims[0].amplitudes().view(np.uint64), orc.amplitudes().view(np.uint64))


def test_streaming_kernel_takes_the_lossy_random_circuit():
    """On a lossy random-circuit state nearly every work item is a STREAM pair the
    streaming kernel finishes; the general kernel sees the rest."""
    n, kc = 16, 10
    gates = Cc.rcs(4, 4, 6, seed=11)
    s = qc().Sim(n, n, 1e-4, chunk_log2=kc, budget=(16 << n) // 4, pool_bytes=2 * (16 << n) + (64 << 20))
    s.apply_circuit(gates[: len(gates) // 2])
    st0 = s.stats()
    s.apply_circuit(gates[len(gates) // 2:])
    st = s.stats()
    done = st["fast_items"] - st0["fast_items"]
    left = st["fast_deferred"] - st0["fast_deferred"]
    assert done > 0 and left <= done // 20
    orc = O.CSim(n, n, kc, 1e-4, (16 << n) // 4)
    orc.apply(gates)
    assert all_images(s) == [orc.image(c) for c in range(orc.nchunks)]


def test_power_of_two_gates_near_the_bottom_of_the_normal_range():
    """sqrt(X) and sqrt(Y) (every coefficient part +-1/2) run as signed sums scaled by
    1/2.  With qubit 3 at |0>, a rotation on it with cos = 1e-300 puts c * a, near
    1e-300 (normal, exponent field below 64), beside every amplitude a: items holding
    such values go to the general kernel, the rest stay on the streaming kernel; the
    images equal the oracle's gate by gate."""
    n, kc, eps = 13, 8, 1e-4
    c = 1e-300
    s_ = np.sqrt(1.0 - c * c)
    g = [Cc.gate(q, Cc.H) for q in range(n) if q != 3]
    g.append(Cc.gate(3, np.array([[c, -s_], [s_, c]], dtype=np.complex128)))
    rng = np.random.default_rng(5)
    for q in rng.permutation(n):
        g.append(Cc.gate(int(q), Cc.SX))
        g.append(Cc.gate(int(q), Cc.SY))
    gates = Cc.to_array(g)
    budget = (16 << n) // 4
    orc = O.CSim(n, n, kc, eps, budget)
    gpu = qc().Sim(n, n, eps, chunk_log2=kc, budget=budget, pool_bytes=2 * (16 << n) + (64 << 20))
    for k in range(len(gates)):
        gpu.apply_gate(gates[k])
        orc.apply(gates[k])
        assert all_images(gpu) == [orc.image(q) for q in range(orc.nchunks)], k
    st = gpu.stats()
    assert st["fast_items"] > 0 and st["fast_deferred"] > 0


@pytest.mark.parametrize("modes", [0x1F, 0x7F])
@pytest.mark.parametrize("kc", [3, 7, 9, 11])
def test_gate_by_gate_and_whole_circuit_agree(kc, modes):
    """The same circuit gate by gate (a launch of the streaming or the image-exchange kernel
    per gate), as whole circuits in one launch, and through the general kernel alone: the
    oracle's images and the same counters, trials of a mode set with SPLIT and PALETTE
    included, in a pool with room and (one launch) in one that just holds every chunk RAW."""
    n = 13
    raw = 16 << n
    circuits = [Cc.rcs_n(n, 6, seed=kc), Cc.qaoa_maxcut(n + 1, 1, 3, seed=4)[0], Cc.qft(n, seed=5)[0], Cc.grover(n, 2, seed=6)[0]]
    keys = ("gates", "encoded_bytes", "max_encoded_bytes", "eps_switch_gate", "chunks_by_mode", "fidelity_lb_sum", "wide_images",
            "split_trials", "palette_trials", "pages_in_use_bytes", "peak_pages_bytes", "amp_updates")
    for ci, gates in enumerate(circuits):
        m = n + (ci == 1)
        got = []
        for how in ("gates", "circuit", "general", "tight"):
            s = qc().Sim(m, m, 1e-4, chunk_log2=kc, budget=raw // 3,
                         pool_bytes=(512 * ((16 << kc) // 512 + 1) << (m - kc)) if how == "tight" else 2 * (16 << m) + (64 << 20))
            s.set_modes(modes)
            if how == "general":
                s.set_option("fast_path", 0)
            if how == "gates":
                for g in gates:
                    s.apply_gate(g)
            else:
                s.apply_circuit(gates[:50])
                s.apply_circuit(gates[50:])
            got.append((all_images(s), {k: s.stats()[k] for k in keys}))
        for g in got[1:]:
            assert g == got[0], ci
        orc = O.CSim(m, m, kc, 1e-4, raw // 3, modes=modes)
        orc.apply(gates)
        assert got[0][0] == [orc.image(c) for c in range(orc.nchunks)], ci


@pytest.mark.parametrize("eps", [0.0, 1e-4])
def test_readout_of_many_chunks(eps):
    """Enough chunks for the warp-per-chunk readout: ragged ranges into aligned and
    unaligned buffers, measurement and fidelity, with STREAM and other images mixed."""
    import torch

    n, kc = 20, 8
    s = qc().Sim(n, n, eps, chunk_log2=kc, budget=(16 << n) // 2 if eps else 2 * (16 << n), pool_bytes=2 * (16 << n) + (64 << 20))
    s.apply_circuit(Cc.rcs_n(n, 3, seed=2))
    s.apply_circuit(Cc.to_array([Cc.gate(n - 1, Cc.X, {q: 1 for q in range(8, n - 1)})]))
    whole = np.concatenate([s.amplitudes(a, 1 << 17) for a in range(0, 1 << n, 1 << 17)])  # few chunks a call: a CTA each
    assert np.array_equal(s.amplitudes().view(np.uint64), whole.view(np.uint64))
    for first, count, skew in ((0, 1 << n, 0), (12345, (1 << n) - 20000, 0), (1, (1 << n) - 1, 1)):
        out = torch.full((2 * count + 3,), 7.0, dtype=torch.float64, device="cuda")
        s.amplitudes(first, count, out=out[skew: skew + 2 * count])
        got = out.cpu().numpy()
        assert np.array_equal(got[skew: skew + 2 * count].view(np.uint64), whole[first: first + count].view(np.float64).view(np.uint64))
        assert (got[skew + 2 * count:] == 7.0).all() and (got[:skew] == 7.0).all()
    ref = np.random.default_rng(1).standard_normal(2 << n).view(np.complex128)
    ref /= np.linalg.norm(ref)
    for skew in (0, 1):
        dev = torch.empty((2 << n) + 1, dtype=torch.float64, device="cuda")[skew: skew + (2 << n)]
        dev.copy_(torch.from_numpy(ref.view(np.float64).copy()))
        f = s.fidelity(dev)
        assert f["F"] == pytest.approx(abs(np.vdot(ref, whole)), rel=1e-10)
        assert f["norm2"] == pytest.approx(float(np.vdot(whole, whole).real), rel=1e-12)
    p = np.abs(whole) ** 2
    for seed in range(5):
        outcome, prob = s.measure(seed)
        assert prob == pytest.approx(p[outcome] / p.sum(), rel=1e-10)


def group_circuit(n, kc, seed):
    """Lossy after its first layers, then runs of gates that share a pass over the state:
    gates of every class inside chunks, diagonal gates and controls anywhere, several gates
    on one cross-chunk target (a controlled X, RZ and a controlled X among them), image
    exchanges in between, more gates in a run than a group holds."""
    rng = np.random.default_rng(seed)
    g = [Cc.gate(q, Cc.H) for q in range(n)] + [Cc.gate(q, [Cc.SX, Cc.SY, Cc.T][int(rng.integers(3))]) for q in range(n)]
    some = lambda lo, hi, t, k: {int(q): int(rng.integers(2)) for q in rng.permutation(np.arange(lo, hi))[:k] if q != t}
    for hi in rng.permutation(np.arange(kc, n))[:3]:
        hi = int(hi)
        for _ in range(14):
            t = int(rng.integers(0, kc))
            g.append(Cc.gate(t, [Cc.SX, Cc.SY, Cc.rx(0.3), Cc.ry(0.4), Cc.X, Cc.H][int(rng.integers(6))], some(0, n, t, int(rng.integers(3)))))
            t = int(rng.integers(0, n))
            g.append(Cc.gate(t, [Cc.T, Cc.Z, Cc.rz(0.7)][int(rng.integers(3))], some(0, n, t, int(rng.integers(3)))))
        for c in (int(rng.integers(0, kc)), int((hi + 1 - kc) % (n - kc) + kc)):
            g += [Cc.gate(hi, Cc.X, {c: 1}), Cc.gate(hi, Cc.rz(0.3)), Cc.gate(hi, Cc.X, {c: 1})]
        g += [Cc.gate(hi, Cc.SY), Cc.gate(3, Cc.SX), Cc.gate(hi, Cc.SX, some(0, kc, hi, 1))]
    g.append(Cc.gate(0, Cc.ry(2.0 ** -900)))  # a coefficient below 2^-52: subnormal and tiny results
    g += [Cc.gate(1, Cc.SX), Cc.gate(kc - 1, Cc.SY), Cc.gate(n - 1, Cc.H)]
    return Cc.to_array(g)


@pytest.mark.parametrize("kc,n", [(7, 17), (8, 18), (9, 19), (10, 20), (11, 20)])
def test_groups_of_gates_on_larger_states(kc, n):
    """States of more chunk pairs than one round of a whole-circuit launch (lossless ones run
    by it all the same): once the bound is settled, groups of gates per pass (pairs of chunks that leave the STREAM form on the way
    taken through the same gates by the general path) end in the oracle's images, and in the
    counters of the same circuit gate by gate: bytes and pages after every gate."""
    keys = ("gates", "encoded_bytes", "max_encoded_bytes", "eps_switch_gate", "chunks_by_mode", "fidelity_lb_sum", "wide_images",
            "pages_in_use_bytes", "peak_pages_bytes", "amp_updates", "level", "sig_bits_current")
    for gates, eps, ladder in ((group_circuit(n, kc, kc), 1e-4, 0), (Cc.grover(n, 1, seed=6)[0][: 3 * n], 1e-3, 1),
                               (group_circuit(n, kc, n)[: 120], 0.0, 0)):
        sims = []
        budget = (16 << n) // 4 if eps else 2 * (16 << n)
        for whole in (True, False):
            s = qc().Sim(n, n, eps, chunk_log2=kc, budget=budget, ladder=ladder, pool_bytes=2 * (16 << n) + (64 << 20))
            if whole:
                s.apply_circuit(gates[: n + 5])
                s.apply_circuit(gates[n + 5:])
            else:
                for x in gates:
                    s.apply_gate(x)
            sims.append(s)
        a, b = (s.stats() for s in sims)
        assert {k: a[k] for k in keys} == {k: b[k] for k in keys}
        assert a["kernel_launches"] < b["kernel_launches"]
        orc = O.CSim(n, n, kc, eps, budget, ladder=ladder)
        orc.apply(gates)
        want = [orc.image(c) for c in range(orc.nchunks)]
        assert all_images(sims[0]) == want
        assert all_images(sims[1]) == want


@pytest.mark.parametrize("ladder", [0, 1])
def test_pages_freed_by_a_whole_circuit_come_back_once(ladder):
    """A pool that just holds every chunk RAW (no CTA keeps a page id between steps), and
    bounds that settle in between: a step then frees thousands of pages at once, and the
    bookkeeping has to put each of them on the stack once.  A page handed out twice or lost
    shows in the images that follow, or as a dry pool."""
    n, kc, eps = 15, 8, 1e-3
    raw = 16 << n
    gates = Cc.rcs_n(n, 10, seed=21)
    orc = O.CSim(n, 9, kc, eps, raw * 9 // 10, ladder=ladder)
    orc.apply(gates)
    want = [orc.image(c) for c in range(orc.nchunks)]
    s = qc().Sim(n, 9, eps, chunk_log2=kc, budget=raw * 9 // 10, ladder=ladder, pool_bytes=512 * ((16 << kc) // 512 + 1) << (n - kc))
    for _ in range(12):
        s.apply_circuit(gates)
        assert all_images(s) == want
        assert s.stats()["max_encoded_bytes"] > 2 * s.stats()["encoded_bytes"]
        s.reset()
