"""Calls of different shapes from several host threads, each on a stream and a workspace of its own
(run on a GB300: pytest -m gpu): the results of calls one after the other."""
import threading

import numpy as np
import pytest

from paper_2608_18147_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def E():
    import torch
    assert torch.cuda.is_available(), "these tests need a CUDA GPU"
    import paper_2608_18147_gb300 as E
    E.lib()
    return E


def test_concurrent_calls_of_different_shapes(E):
    import torch

    def solve(x, s, flags):
        Q, r = E.ecasq_solve(x, s, budget_bits=1.5, refine_max_rounds=5, flags=flags)
        return [Q.cpu().numpy(), r["lambda"], r["mse"]]

    def rows(X, s):
        Q, m, r = E.ecasq_solve_batched(X, s, budget_bits=1.5)
        return [Q.cpu().numpy(), m.cpu().numpy(), r.field("mse")]

    rng = np.random.default_rng(0)
    jobs = [lambda: solve(workloads.signed_lognormal(6000, 1), 16, E.RESIDENT_COSTS),
            lambda: solve(workloads.normal(1100, 2), 8, 0),
            lambda: solve(workloads.student_t(3000, 3, scale=1.0), 32, 0),
            lambda: solve(workloads.normal(2500, 4), 5, E.RESIDENT_COSTS),
            lambda X=rng.standard_normal((40, 100)).astype(np.float32): rows(X, 8),
            lambda X=rng.standard_normal((10, 700)).astype(np.float32): rows(X, 16)]
    want = [job() for job in jobs]
    wrong = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(5):
                    for a, b in zip(jobs[i](), want[i]):
                        np.testing.assert_array_equal(a, b)
        except Exception as e:  # noqa: BLE001 -- reported below, with the job
            wrong.append((i, repr(e)))

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong


def test_overlapping_noalloc_encodes_keep_their_counts(E):
    """ecasq_quantize_noalloc from several threads at once: the calls share the library's status record, their
    counts and entropies are their own."""
    import torch
    rng = np.random.default_rng(3)
    jobs = []
    for m in (4, 8, 16, 24, 33, 40):
        x = torch.as_tensor(rng.uniform(-1, 1, 4000003).astype(np.float32)).cuda()
        Q = torch.linspace(-1, 1, m, device="cuda")
        _, counts, h = E.ecasq_quantize(x, Q, m)
        jobs.append((x, Q, m, counts, h))
    torch.cuda.synchronize()
    wrong = []

    def work(x, Q, m, want, h):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                idx = torch.empty(x.numel(), dtype=torch.uint8, device="cuda")
                for _ in range(30):
                    counts = torch.full((m,), -1, dtype=torch.int32, device="cuda")
                    assert E.ecasq_quantize_noalloc(x, Q, m, idx, counts) == pytest.approx(h, rel=1e-12)
                    assert torch.equal(counts, want)
        except Exception as e:  # noqa: BLE001 -- reported below, with the codebook
            wrong.append((m, repr(e)))

    threads = [threading.Thread(target=work, args=job) for job in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
