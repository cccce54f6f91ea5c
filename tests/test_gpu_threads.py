"""Two host threads, each with handles and a stream of its own, whose calls launch the same kernel with different
amounts of shared memory: different handles are independent, so neither may refuse or change the other's call."""
import threading

import pytest
import torch

from synth import boxes, inr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    import __graft_entry__ as g
    g.build()
    import paper_2402_13861_gb300 as p
    torch.cuda.set_device(0)
    return p


def run_threads(jobs):
    """Each job, a callable, in a thread with its own stream; the first exception is raised here."""
    errors, start = [], threading.Barrier(len(jobs))

    def body(job):
        try:
            torch.cuda.set_device(0)
            with torch.cuda.stream(torch.cuda.Stream()):
                start.wait()
                job()
                torch.cuda.current_stream().synchronize()
        except Exception as e:          # noqa: BLE001 - handed to the main thread
            errors.append(e)

    threads = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    if errors:
        raise errors[0]


@pytest.mark.parametrize("w", [64, 256])
def test_reduced_bounds_of_short_and_long_lists(pkg, w):
    layers = inr.random_inr([3, w, w, 1], 120 + w)
    lo, hi = (torch.tensor(x, device="cuda") for x in boxes.random_boxes(40003, 121, -10, -2))
    cases = [(pkg.Inr(layers), n) for n in (7, 40003)]
    want = [net.bound_cells(lo[:n], hi[:n], mode="rafixed") for net, n in cases]
    torch.cuda.synchronize()
    got = [None] * len(cases)

    def job(i):
        net, n = cases[i]
        for _ in range(1500):
            got[i] = net.bound_cells(lo[:n], hi[:n], mode="rafixed")

    run_threads([lambda i=i: job(i) for i in range(len(cases))])
    for a, b in zip(got, want):
        assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])
    for net, _ in cases:
        net.close()


@pytest.mark.parametrize("w", [128, 256])
def test_tensor_core_evaluation_of_shallow_and_deep_networks(pkg, w):
    x = torch.rand((1000, 3), device="cuda") * 2 - 1
    nets = [pkg.Inr(inr.random_inr([3] + [w] * H + [1], 130 + H)) for H in (2, 12)]
    want = [net.eval_points(x, prec="bf16") for net in nets]
    torch.cuda.synchronize()
    got = [None] * len(nets)

    def job(i):
        for _ in range(1500):
            got[i] = nets[i].eval_points(x, prec="bf16")

    run_threads([lambda i=i: job(i) for i in range(len(nets))])
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    for net in nets:
        net.close()
