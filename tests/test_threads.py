"""Host threads that call the library at once, each on a stream and a workspace of its own, with sizes whose
kernels are the same functions with different amounts of shared memory."""
import threading

import pytest

from paper_2512_13368_b200 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes,rounds", [
    (((4, 220, {}), (4, 400, {}), (4, 300, {}), (2, 130, {})), 400),                  # short histories
    (((4, 600, {}), (2, 2000, {}), (1, 4096, {}), (2, 1100, {})), 100),               # tile lists of other lengths
    (((2, 600, {"per_query": 1}), (2, 900, {"per_query": 1}), (1, 1500, {"per_query": 1})), 100),
])
def test_threads_do_not_disturb_each_other(sizes, rounds):
    import torch
    from paper_2512_13368_b200 import runner
    problems, want = [], []
    for B, L, opts in sizes:
        w = workloads.make("threads", "bf16", B, 2, L, 64, 32, 4, 40, seed=L)
        w.per_query = opts.get("per_query", 0)
        problems.append(runner.DeviceProblem(w))
        problems[-1].step()
    torch.cuda.synchronize()
    keys = ("idx", "out", "lse", "dq", "dk", "dv", "dgate")
    for p in problems:
        want.append({k: getattr(p, k).clone() for k in keys})
    failures, start = [], threading.Barrier(len(problems))

    def work(p):
        try:
            stream = torch.cuda.Stream()
            start.wait()
            for _ in range(rounds):
                p.step(stream=stream.cuda_stream)
            stream.synchronize()
        except Exception as e:  # noqa: BLE001
            failures.append(e)

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(p,)) for p in problems]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures, failures
    torch.cuda.synchronize()
    for p, first in zip(problems, want):
        for k in keys:
            assert torch.equal(first[k], getattr(p, k)), k
