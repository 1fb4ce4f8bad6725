"""The library's host code when a CUDA call or a launch fails, without a GPU:
its objects are linked against a CUDA runtime on the host (fake_cuda.cpp), in
which kernels do nothing and any call can be made to return an error.  What is
checked is what the host does next: whether the call fails, and what the one
after it launches."""
import glob
import os
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1511_07482_gb300 import build
    objs = sorted(glob.glob(os.path.join(build.BUILD, "*.o")))
    if len(objs) != len(build.SOURCES):
        pytest.skip("the library is not built")
    lib = str(tmp_path_factory.mktemp("fake") / "libkdefft_fake.so")
    subprocess.run([build.nvcc(), "-shared", "-cudart", "none", "-Xcompiler", "-fPIC", "-Xcompiler", "-pthread",
                    "-o", lib, *objs, os.path.join(HERE, "fake_cuda.cpp")], check=True, capture_output=True)
    return lib


def _run(fake, body):
    """Run `body` in a process of its own: the library of a process is loaded once
    (without torch, which takes longer to import than the rest)."""
    code = (f"import sys; sys.path[:0] = [{ROOT!r}, {HERE!r}]; sys.modules['torch'] = None\n"
            f"from test_host_errors_cpu import Fake\nfk = Fake({fake!r})\n{body}")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


class Fake:
    def __init__(self, path):
        from paper_1511_07482_gb300 import _lib
        self.lib = _lib.load(path)
        self.lib.fake_log.restype = __import__("ctypes").c_char_p

    def context(self):
        from paper_1511_07482_gb300 import Context
        return Context(0, stream=8)   # a handle that the fake's own never equal

    def data(self, ctx, d=2, M=40, **opts):
        X = np.random.default_rng(1).random((200, d))
        return ctx.bin(X, np.zeros(d), np.ones(d), [M] * d, **opts)

    def call(self, f, fail=None, nth=1):
        """(did it raise, did the failure happen, log lines)"""
        from paper_1511_07482_gb300 import KdefftError
        self.lib.fake_clear()
        self.lib.fake_fail((fail or "-").encode(), nth if fail else 0)
        try:
            f()
            raised = False
        except KdefftError:
            raised = True
        hit = self.lib.fake_hits()
        self.lib.fake_fail(b"-", 0)
        return raised, bool(hit), self.lib.fake_log().decode().splitlines()


@pytest.mark.parametrize("what", ["cudaMemcpyAsync", "cudaMallocHost", "launch", "cudaStreamSynchronize"])
def test_an_error_ends_with_its_call(fake, what):
    """The runtime keeps a failed call's error until it is asked for; the next
    call of the library must not report it as its own."""
    _run(fake, f"""
import numpy as np
failed = 0
for nth in range(1, 60):
    ctx = fk.context()
    ds = fk.data(ctx)
    raised, hit, log = fk.call(lambda: ds.scv(0.02 * np.eye(2), 0.01 * np.eye(2), grad=True), {what!r}, nth)
    if raised:
        failed += 1
        again, _, log2 = fk.call(lambda: ds.scv(0.02 * np.eye(2), 0.01 * np.eye(2), grad=True))
        assert not again, (nth, log, log2)
    ctx.close()
    if not hit:
        break
assert not hit and failed >= 2
""")


@pytest.mark.parametrize("what", ["cudaMalloc", "k_line", "cudaMemcpyAsync"])
def test_no_box_is_claimed_that_was_not_computed(fake, what):
    """A call that fails on its way to the count autocorrelation, at whichever
    step, leaves nothing that the next call would take for computed: one of the
    two launches all three passes."""
    _run(fake, f"""
import numpy as np
failed = 0
passes = lambda log: sum("k_line" in l and l.endswith(" 8") for l in log)
for grown in (False, True):
    for nth in range(1, 60):
        ctx = fk.context()
        ds = fk.data(ctx)
        if grown:
            ds.psi(1e-4 * np.eye(2), 2)
        raised, hit, log = fk.call(lambda: ds.psi(0.02 * np.eye(2), 2), {what!r}, nth)
        assert hit or not raised
        if raised:
            failed += 1
            again, _, log2 = fk.call(lambda: ds.psi(0.02 * np.eye(2), 2))
            assert not again and (passes(log) == 3 or passes(log2) == 3), (grown, nth, log, log2)
        ctx.close()
        if not hit:
            break
    assert not hit and nth > 1
assert failed >= 4
""")


CALLS = {"bin": "lambda: fk.data(ctx)", "psi": "lambda: ds.psi(0.02 * I, 2)",
         "scv": "lambda: ds.scv(0.02 * I, 0.01 * I, grad=True)", "autocorr": "lambda: ds.autocorr([30, 30])",
         "fft": "lambda: (ctx.set_engine(3), ds.psi(0.02 * I, 2))",
         "ise": "lambda: ds.ise_mixture(0.02 * I, [1.0], np.zeros(2), I)"}


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("what", ["cudaStreamBeginCapture", "cudaStreamEndCapture", "cudaGraphInstantiate"])
def test_a_failed_capture_is_no_error(fake, call, what):
    """The work of a new launch sequence is issued before it is captured, so a
    capture that fails must not fail the call (whose copies and launches are on
    their way); the sequence is captured the next time."""
    _run(fake, f"""
import numpy as np
I = np.eye(2)
ctx = fk.context()
ds = fk.data(ctx)
n0 = ctx.runtime_stats()["graphs_captured"]
raised, hit, log = fk.call({CALLS[call]}, {what!r})
assert hit and not raised, log
assert not fk.call({CALLS[call]})[0]
assert ctx.runtime_stats()["graphs_captured"] > n0 or {call == "autocorr"}   # (a box is computed once)
""")


@pytest.mark.parametrize("graphs", [True, False])
@pytest.mark.parametrize("call", CALLS)
def test_nothing_is_in_flight_after_an_error(fake, call, graphs):
    """Where the n-th launch, copy or event of a call fails, the stream is
    waited for before the call returns: what was issued reads pinned buffers
    and writes results that the next call uses."""
    _run(fake, f"""
import numpy as np
I = np.eye(2)
failed = 0
for what in ("launch", "cudaMemcpyAsync 8", "cudaEventRecord", "cudaStreamWaitEvent"):
    for nth in range(1, 60):
        ctx = fk.context()
        ctx.set_graphs({graphs})
        ds = fk.data(ctx)
        raised, hit, log = fk.call({CALLS[call]}, what, nth)
        if raised:
            failed += 1
            at = next(i for i, l in enumerate(log) if l.endswith("FAILS"))
            issued = any(l.startswith(("launch", "cudaMemcpyAsync", "cudaMemsetAsync")) and l.endswith(" 8") for l in log[:at])
            assert not issued or "cudaStreamSynchronize 8" in log[at:], (what, nth, log)
        ctx.close()
        if not hit:
            break
    assert not hit
assert failed >= 2
""")
