"""Contexts whose coarse tails need different amounts of shared memory, alive at the same time: in turn in one
thread and in two host threads.  The kernels of a context are the same whatever else runs, so every result is
compared bit for bit with that of the context used alone."""
import threading

import numpy as np
import pytest
import torch

from paper_1410_2240_gb300 import synth

from _gpu_util import dev, host

pytestmark = pytest.mark.gpu

# tails that start at 20^3, 8^3 and 16^3: 50, 4 and 20 KB of shared memory per CTA in FP64 (48 KB is what a kernel
# has without asking)
SHAPES = [(40, 40, 40), (16, 16, 16), (32, 32, 32)]


@pytest.fixture(scope="module")
def mgp():
    import __graft_entry__
    __graft_entry__.build()
    from paper_1410_2240_gb300 import mgproj
    return mgproj


def _inputs(mgp, shape):
    case = synth.small_case(*shape, solid="ellipsoid", seed=71)
    beta = mgp.face_coeffs(dev(case.phi), case.h, dev(case.solid, dtype=torch.uint8), rho_air=case.lam)
    rhs = dev(case.rhs)
    torch.cuda.synchronize()
    return beta, case.h, rhs


def _make(mgp, shape, **kw):
    beta, h, rhs = _inputs(mgp, shape)
    return mgp.Context(beta, h, coarse_max_cells=2048, **kw), rhs


def _cycles(mgp, ctx, rhs, n):
    p = torch.zeros_like(rhs)
    for _ in range(n):
        ctx.vcycle(rhs, p)
    return p


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_contexts_in_turn(mgp, prec, graph):
    alone = []
    for shape in SHAPES:
        ctx, rhs = _make(mgp, shape, prec=prec, coarse_graph=graph)
        l0 = mgp.kernel_launches()
        alone.append(host(_cycles(mgp, ctx, rhs, 4)))
        tail = mgp.kernel_launches() - l0
        ctx.close()
        ctx, _ = _make(mgp, shape, prec=prec, coarse_graph=graph, coarse_tail=0)
        l0 = mgp.kernel_launches()
        _cycles(mgp, ctx, rhs, 4)
        assert mgp.kernel_launches() - l0 > tail  # (the tail ran)
        ctx.close()
    made = [_make(mgp, shape, prec=prec, coarse_graph=graph) for shape in SHAPES]
    p = [torch.zeros_like(rhs) for _, rhs in made]
    for _ in range(4):
        for (ctx, rhs), q in zip(made, p):
            ctx.vcycle(rhs, q)
    for q, want in zip(p, alone):
        assert np.array_equal(host(q), want)


@pytest.mark.parametrize("graph", [0, 1])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_contexts_in_two_threads(mgp, prec, graph):
    """With coarse_graph = 0 a thread launches its tail in every cycle while the other launches its own; with
    1 each context is set up, captured and replayed beside the other's work."""
    streams = [torch.cuda.Stream() for _ in range(2)]
    rounds, cycles = (4 if graph == 0 else 40), (500 if graph == 0 else 3)
    inputs, want = [_inputs(mgp, shape) for shape in SHAPES[:2]], []
    for beta, h, rhs in inputs:
        ctx = mgp.Context(beta, h, coarse_max_cells=2048, prec=prec, coarse_graph=graph)
        want.append(host(_cycles(mgp, ctx, rhs, cycles)))
        ctx.close()
    failed = []
    barrier = threading.Barrier(2, timeout=120)

    def work(t):
        try:
            with torch.cuda.stream(streams[t]):
                beta, h, rhs = inputs[t]
                barrier.wait()
                for _ in range(rounds):
                    ctx = mgp.Context(beta, h, coarse_max_cells=2048, stream=streams[t], prec=prec, coarse_graph=graph)
                    p = _cycles(mgp, ctx, rhs, cycles)
                    streams[t].synchronize()
                    if not np.array_equal(p.cpu().numpy(), want[t]):
                        failed.append((t, "other bits"))
                    ctx.close()
        except Exception as e:  # reported by the main thread
            failed.append((t, repr(e)))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(2)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not failed, failed


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("shape,tail", [((32, 64, 32), True), ((28, 32, 36), True), ((36, 36, 28), False), ((36, 36, 36), False)])
def test_tail_up_to_512_cells_of_the_coarsest_grid(mgp, shape, tail, prec):
    """Coarsest grids of 256, 504, 567 and 729 cells: a larger one is solved by a launch of its own on every SM."""
    launches = []
    for t in (0, 1):
        ctx, rhs = _make(mgp, shape, prec=prec, coarse_tail=t)
        p = torch.zeros_like(rhs)
        l0 = mgp.kernel_launches()
        ctx.vcycle(rhs, p)
        launches.append(mgp.kernel_launches() - l0)
        ctx.close()
    assert (launches[1] < launches[0]) == tail
