"""What the library's host code does around its launches, without a GPU: a child process
loads the library on top of a CUDA runtime whose kernels do nothing (fake_cudart.c), so the
state stays lossless and calls that fail can be chosen."""
import os
import shutil
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))), "include")

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None or shutil.which("gcc") is None, reason="no compilers")

PRELUDE = """
import ctypes as C
from paper_1911_04034_gb300 import circuits as Cc, qcsim as q
fake = C.CDLL(None)
num = lambda name: C.c_int.in_dll(fake, name)
def log():
    return C.string_at(C.addressof(C.c_char.in_dll(fake, "fake_log")), num("fake_ops").value).decode()
# two SMs of one block each: 16 pairs of chunks are many rounds, 1 or 2 are one
def make(n, kc=7, eps=1e-4, **kw):
    return q.Sim(n, kc, eps, chunk_log2=kc, budget=16 << n, pool_bytes=4 << 20, **kw)
def code(f, *a):
    try:
        f(*a)
    except q.SimError as e:
        return e.code
    return 0
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1911_04034_gb300 import build

    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-I" + CUDA, os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", so], check=True)

    def go(body):
        r = subprocess.run([sys.executable, "-c", PRELUDE + textwrap.dedent(body)], cwd=ROOT, capture_output=True, text=True,
                           timeout=120, env={**os.environ, "LD_PRELOAD": so})
        assert r.returncode == 0, r.stdout[-1000:] + r.stderr[-3000:]

    return go


@pytest.mark.parametrize("n,how", [(9, "circuit"), (12, "circuit"), (12, "gate"), (12, "batch")])
def test_call_that_fails_halfway_poisons_its_handle(run, n, how):
    """A launch that fails after others of the same call were made leaves gates half applied:
    the call returns SIM_ERR_CUDA and the handle refuses further work -- a launch per segment
    of a small state (9 qubits), gate kernels of a large one (12), also as the large state of
    a batch, and a single gate's kernels.  If it is the first one, the handle stays usable."""
    run(f"""
    gates = Cc.rcs_n({n}, 12, seed=1)
    for nth in (1, 2, 3):
        s, other = make({n}), make(9)
        num("fake_fail_launch").value = num("fake_launches").value + nth
        if "{how}" == "circuit":
            got = code(s.apply_circuit, gates)
        elif "{how}" == "gate":
            got = code(s.apply_gate, gates[0])
        else:
            got = code(q.batch_apply, [s, other], [gates, Cc.h_all(9)])
        assert got == q.ERR_CUDA, (nth, got)
        num("fake_fail_launch").value = 0
        assert code(s.apply_circuit, gates) == (0 if nth == 1 else q.ERR_STATE), nth
        assert code(other.apply_circuit, Cc.h_all(9)) == 0
    """)


def test_looking_for_the_settled_bound_keeps_the_queue_full(run):
    """A large lossy state whose bound never settles: apart from the first look the host never
    waits for gates it enqueued last, until it synchronises at the end of the call."""
    run("""
    gates = Cc.rcs_n(12, 20, seed=1)
    s = make(12)
    start = num("fake_ops").value
    s.apply_circuit(gates)
    ops = log()[start:]
    assert ops.count("L") >= 2 * len(gates) > 400
    assert ops.count("W") + ops.count("S") <= 2 and ops.rstrip("S").count("S") == 0, ops
    assert ops.count("w") >= len(gates) // 8
    """)


def test_autotuner_times_the_call_that_is_made(run):
    """A probe on a small state runs whole-circuit launches in both halves, as
    sim_apply_circuit does, and no gate kernel of its own per gate."""
    run("""
    probe = Cc.rcs_n(9, 6, seed=1)
    s = make(9)
    a = fake.fake_count(b"k_run")
    s.apply_circuit(probe[: len(probe) // 2]); s.apply_circuit(probe[len(probe) // 2:])
    per_point = fake.fake_count(b"k_run") - a
    a = fake.fake_count(b"k_run")
    best, rates = q.autotune_chunk(9, 8, 1e-4, probe, candidates=(7, 8))
    assert all(r > 0 for r in rates.values()) and best in rates
    assert fake.fake_count(b"k_run") - a == 2 * per_point and fake.fake_count(b"k_gate") == 0
    """)


def test_device_bytes_is_what_the_handle_allocated(run):
    """sim_stats_t.device_bytes against the runtime's own count: after creation, a circuit's
    staged gate records (a small state's and a longer circuit's), a kept batch graph, readout
    scratch, the block cache, timing, the selector network and training records."""
    run("""
    import numpy as np
    s = make(9)
    count = C.c_longlong.in_dll(fake, "fake_device_bytes")
    def check(what):
        assert s.stats()["device_bytes"] == count.value, (what, s.stats()["device_bytes"], count.value)
    check("created")
    s.apply_circuit(Cc.h_all(9)); check("circuit")
    s.apply_circuit(Cc.rcs_n(9, 40, seed=1)); check("longer circuit")
    q.batch_apply([s], [Cc.h_all(9)], use_graph=True); check("batch graph")
    s.amplitudes(0, 4); check("readout")
    s.set_block_cache(True); check("block cache")
    s.set_timing(1); check("timing")
    s.apply_circuit(Cc.h_all(9)); check("timed circuit")
    s.set_selector(2, np.zeros(1864, dtype=np.uint16)); check("selector")
    s.trace(100); check("trace")
    s.trace(0); s.set_block_cache(False); check("given back")
    """)
