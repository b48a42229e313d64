"""Runs of plain steps on the multi-step kernels.

A small domain's plain steps run in one launch (a thread-block cluster, or a
grid whose CTAs keep the state in shared memory or in L2).  Whatever its form,
the populations, the check values and the clock must equal those of the same
steps launched kernel by kernel, bit for bit (the arithmetic is the same), at
the sizes where the forms and their work split change: one pair of nodes,
empty second lanes (odd nz), one and several CTAs, one and several pairs per
thread, the state in L2, and links that wrap or mirror across CTAs.
"""
import numpy as np
import pytest

from parity_util import problem, seeded_state

pytestmark = pytest.mark.gpu

SHAPES = [
    (1, 1), (3, 2), (64, 4), (9, 255),   # one CTA or a few of a cluster
    (64, 64), (65, 64), (64, 65),        # the largest cluster (FP32 pairs), the smallest grids
    (4099, 3), (3, 1999),                # rows longer than a CTA's range, columns across many CTAs
    (199, 391),                          # several pairs per thread
]


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_0282_gb300 import build
    build.build()
    from paper_1003_0282_gb300 import axlbm
    return axlbm


def both_ways(B, pb, precision, calls, seed=3):
    st = seeded_state(pb, seed)
    out = []
    for graphs in (True, False):
        dom = B.Domain(pb, precision)
        dom.use_graphs(graphs)
        dom.set_populations(st.f, st.g if pb.swirl else None, st.h if pb.temperature else None, time=6)
        for n in calls:
            dom.step(n)
        assert dom.time == 6 + sum(calls)
        out.append((dom.get_populations(), dom.residual()))
        dom.close()
    (p0, r0), (p1, r1) = out
    assert r0 == r1
    for x, y in zip(p0, p1):
        assert (x is None and y is None) or np.array_equal(x, y)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("mix", ["pipe", "crystal", "annulus-mixed"])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_equals_single_steps(B, shape, mix, precision):
    both_ways(B, problem(*shape, mix), precision, [11, 12])


@pytest.mark.parametrize("swirl,temp,collision", [(False, False, "bgk"), (True, False, "mrt"), (False, True, "mrt")])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_distributions_and_collisions(B, swirl, temp, collision, precision):
    for shape in ((37, 23), (130, 97)):
        both_ways(B, problem(*shape, "closed", swirl=swirl, temperature=temp, collision=collision), precision, [21])


def test_state_in_l2(B):
    both_ways(B, problem(701, 809, "crystal", temperature=False), "fp32", [12])


def test_long_runs_refresh_the_force(B):
    """An oscillating force over more steps than a launch keeps ready, from an odd level."""
    pb = problem(40, 11, "pipe", swirl=False, temperature=False)
    both_ways(B, pb, "fp64", [1, 600, 301])


@pytest.mark.parametrize("scale", [1, 4])
def test_small_batches(B, scale):
    """Domains of uneven size, with and without temperature, in one multi-step launch."""
    probs = [problem(17 * scale, 29 * scale, "crystal"), problem(43 * scale, 8 * scale, "pipe", temperature=False),
             problem(50 * scale, 63, "annulus-mixed", collision="mrt", tau=0.55), problem(1, 1, "closed"),
             problem(64, 33 * scale, "free-top", temperature=False)]
    out = []
    for graphs in (True, False):
        batch = B.Batch(probs, "fp32")
        batch.use_graphs(graphs)
        for d, pb in enumerate(probs):
            st = seeded_state(pb, 40 + d)
            batch.set_populations(d, st.f, st.g, st.h if pb.temperature else None)
        batch.step(1)
        batch.step(24)
        batch.step(13)
        caps, launches = batch.graph_stats()
        assert (caps, launches) == ((1, 2) if graphs else (0, 0))
        out.append(([batch.get_populations(d) for d in range(len(probs))], batch.residuals(), batch.time))
        batch.close()
    (p0, r0, t0), (p1, r1, t1) = out
    assert t0 == t1 == 38 and np.array_equal(r0, r1)
    for d in range(len(probs)):
        for x, y in zip(p0[d], p1[d]):
            assert (x is None and y is None) or np.array_equal(x, y), d


@pytest.mark.parametrize("kind", ["domain", "batch"])
def test_captured_calls_replay(B, kind):
    """A call that the caller captures advances the state on every replay, as calls in between do."""
    import torch

    pb = problem(64, 48, "crystal") if kind == "domain" else None
    probs = [problem(33, 40, "crystal"), problem(20, 31, "pipe", temperature=False)]
    got = []
    for captured in (True, False):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            if kind == "domain":
                sim = B.Domain(pb, "fp32", stream=stream)
                st = seeded_state(pb, 3)
                sim.set_populations(st.f, st.g, st.h, time=0)
            else:
                sim = B.Batch(probs, "fp32", stream=stream)
                for d, p in enumerate(probs):
                    st = seeded_state(p, 3 + d)
                    sim.set_populations(d, st.f, st.g, st.h if p.temperature else None)
            sim.step(20)
            stream.synchronize()
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                    sim.step(20)
                for _ in range(3):
                    graph.replay()
            else:
                for _ in range(3):
                    sim.step(20)
            stream.synchronize()
            got.append([sim.get_populations()] if kind == "domain" else [sim.get_populations(d) for d in range(2)])
            sim.close()
    for x, y in zip(*got):
        for u, v in zip(x, y):
            assert (u is None and v is None) or np.array_equal(u, v)


@pytest.mark.parametrize("shape", [(1, 1), (2, 5), (64, 4), (9, 255), (40, 60), (65, 64), (4099, 3), (199, 391)])
@pytest.mark.parametrize("mix", ["pipe", "crystal", "annulus-mixed"])
@pytest.mark.parametrize("swirl,temp,collision", [(True, True, "bgk"), (False, False, "bgk"), (True, False, "mrt"), (False, True, "mrt")])
@pytest.mark.parametrize("precision", ["fp16", "bf16"])
def test_16_bit_storage(B, shape, mix, swirl, temp, collision, precision):
    """The outer ring keeps the ring kernels' own arithmetic; every store rounds to the storage type."""
    both_ways(B, problem(*shape, mix, swirl=swirl, temperature=temp, collision=collision), precision, [11, 52])


def test_small_fp16_batch(B):
    probs = [problem(17, 29, "crystal"), problem(143, 208, "pipe", temperature=False),
             problem(50, 63, "annulus-mixed", collision="mrt", tau=0.55), problem(1, 1, "closed")]
    out = []
    for graphs in (True, False):
        batch = B.Batch(probs, "fp16")
        batch.use_graphs(graphs)
        for d, pb in enumerate(probs):
            st = seeded_state(pb, 40 + d)
            batch.set_populations(d, st.f, st.g, st.h if pb.temperature else None)
        batch.step(1)
        batch.step(24)
        out.append(([batch.get_populations(d) for d in range(len(probs))], batch.residuals()))
        batch.close()
    (p0, r0), (p1, r1) = out
    assert np.array_equal(r0, r1)
    for x, y in zip(p0, p1):
        for u, v in zip(x, y):
            assert (u is None and v is None) or np.array_equal(u, v)


# a cluster, one pair per thread, several pairs per thread, the state in L2, a batch
REPLAYED = {
    "cluster": ("fp32", [(64, 48)], {}),
    "one": ("fp32", [(128, 192)], {}),
    "slab": ("fp64", [(199, 391)], {}),
    "l2": ("fp32", [(701, 809)], {"temperature": False}),
    "batch": ("fp32", [(33, 40), (90, 61)], {}),
}


@pytest.mark.parametrize("kind", sorted(REPLAYED))
def test_direct_calls_around_replays(B, kind):
    """Direct calls before, between and after replays of a captured call continue from the level that the replays
    reached: with an oscillating force a call that took its level from elsewhere would have the wrong phase."""
    import torch

    precision, shapes, extra = REPLAYED[kind]
    probs = [problem(*s, "crystal", **extra) for s in shapes]
    assert all(pb.omega_t != 0 and pb.az0 != 0 for pb in probs)
    states = [seeded_state(pb, 3 + d) for d, pb in enumerate(probs)]
    got = []
    for captured in (True, False):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            if kind == "batch":
                sim = B.Batch(probs, precision, stream=stream)
                for d, (pb, st) in enumerate(zip(probs, states)):
                    sim.set_populations(d, st.f, st.g, st.h)
            else:
                pb, st = probs[0], states[0]
                sim = B.Domain(pb, precision, stream=stream)
                sim.set_populations(st.f, st.g, st.h if pb.temperature else None, time=0)
            if not captured:
                sim.use_graphs(False)
            sim.step(20)
            stream.synchronize()
            if captured:
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
                    sim.step(20)
                again = graph.replay
            else:
                again = lambda: sim.step(20)
            again()
            again()
            sim.step(20)
            again()
            sim.step(40)
            sim.step(20)
            stream.synchronize()
            got.append([sim.get_populations(d) for d in range(len(probs))] if kind == "batch"
                       else [sim.get_populations()])
            sim.close()
    for x, y in zip(*got):
        for u, v in zip(x, y):
            assert (u is None and v is None) or np.array_equal(u, v)
