"""Objects of different sizes used from two threads at once: the launches of one
must not depend on limits that the other's calls set."""
import threading

import pytest

from tests.gpu_util import lib

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _run_together(calls):
    errors = []
    start = threading.Barrier(len(calls))

    def work(call):
        try:
            start.wait()
            for _ in range(400):
                call()
        except Exception as e:  # reported by the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors


def test_batches_of_different_sizes_in_two_threads():
    dn = lib()
    calls, refs, batches = [], [], []
    for n in (1, 24):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            B = dn.Batch([dn.default_config(level_solve=2, precision=1, obstacle_i0=2, obstacle_j0=1)
                          for _ in range(n)], stream=s)
            B.linearize()
            b = torch.ones(B.length, device="cuda")
            x = torch.empty_like(b)
            refs.append(B.vcycle(b).clone())
            s.synchronize()
        batches.append((B, b, x))
        calls.append(lambda B=B, b=b, x=x: B.vcycle(b, x))
    _run_together(calls)
    torch.cuda.synchronize()
    for (B, b, x), ref in zip(batches, refs):
        assert torch.equal(x, ref)


def test_networks_of_different_sizes_in_two_threads():
    dn = lib()
    calls = []
    for replaced in (1, 2):
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            c = dn.Context(level_solve=2, replaced_levels=replaced, hidden=32, gru_layers=1, stream=s)
            k = 2 ** replaced + 1
            x = torch.zeros(300, 4 * k * k + 4, dtype=torch.bfloat16, device="cuda")
            h = torch.zeros(1, 300, 32, device="cuda")
            out = torch.empty(300, 2 * k * k, device="cuda")
            s.synchronize()
        calls.append(lambda c=c, x=x, h=h, out=out: c._check(c.lib.dnnmg_patch_infer(
            c.h, x.data_ptr(), h.data_ptr(), out.data_ptr(), 300)))
    _run_together(calls)
