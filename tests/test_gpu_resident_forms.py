"""Each form of the multi-step launches, known to be the one that ran.

The library says which form a domain or a batch takes.  The shapes that
test_gpu_resident.py compares with single steps take a multi-step launch; here
the form with the state in L2, whose thread blocks wait for their neighbours'
step counters, is compared over its lists of neighbours (periodic ends, an odd
number of rows, uneven domains of a batch), both precisions, with and without
the temperature, and with one block per SM.  Populations, check values and the
clock must be those of single steps bit for bit.
"""
import numpy as np
import pytest

from parity_util import problem, seeded_state
from test_gpu_resident import SHAPES

pytestmark = pytest.mark.gpu

STEPS, CLUSTER, ONE, SEVERAL, L2 = range(5)


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_0282_gb300 import build
    build.build()
    from paper_1003_0282_gb300 import axlbm
    return axlbm


def test_shapes_take_multi_step_launches(B):
    seen = set()
    for precision in ("fp32", "fp64", "fp16", "bf16"):
        for shape in SHAPES + [(37, 23), (130, 97)]:
            dom = B.Domain(problem(*shape, "crystal"), precision)
            dom.step(12)
            form, ctas = dom.step_form()
            assert form != STEPS and ctas >= 1, (precision, shape)
            assert dom.graph_stats() == (1, 1), (precision, shape)
            dom.close()
            seen.add(form)
    assert {CLUSTER, ONE, SEVERAL} <= seen
    wet = B.Domain(problem(37, 23, "nee-cavity"), "fp32")
    assert wet.step_form() == (STEPS, 0)
    wet.close()


def equal(got):
    (p0, r0, t0), (p1, r1, t1) = got
    assert t0 == t1 and np.array_equal(r0, r1)
    for d, (x, y) in enumerate(zip(p0, p1)):
        for u, v in zip(x, y):
            assert (u is None and v is None) or np.array_equal(u, v), d


# A block's shared memory holds 12 bytes a pair (FP64: 16 a node) and, for the pairs on the domain's outline, their slots
# (168 bytes a pair with every population): rows of 601 pairs and more leave room for one block per SM.
L2_DOMAINS = [
    # precision, shape, mix, changes to the problem, one block per SM
    ("fp32", (300, 2225), "pipe", {}, False),
    ("fp32", (601, 1111), "pipe", {}, True),
    ("fp32", (613, 901), "annulus-mixed", {"collision": "mrt"}, True),
    ("fp32", (1001, 1201), "pipe", {"temperature": False, "swirl": False}, False),
    ("fp64", (401, 777), "annulus-mixed", {}, False),
    ("fp64", (701, 997), "pipe", {"temperature": False, "swirl": False}, False),
    ("fp32", (185000, 2), "pipe", {}, True),   # every pair is on the outline
]


@pytest.mark.parametrize("precision,shape,mix,changes,alone", L2_DOMAINS)
def test_state_in_l2(B, precision, shape, mix, changes, alone):
    import torch
    pb = problem(*shape, mix, **changes)
    st = seeded_state(pb, 9)
    got = []
    for graphs in (True, False):
        dom = B.Domain(pb, precision)
        form, ctas = dom.step_form()
        assert form == L2
        assert (ctas <= torch.cuda.get_device_properties(0).multi_processor_count) == alone
        dom.use_graphs(graphs)
        dom.set_populations(st.f, st.g if pb.swirl else None, st.h if pb.temperature else None, time=4)
        for n in (1, 24, 13):
            dom.step(n)
        assert dom.graph_stats() == ((1, 2) if graphs else (0, 0))
        got.append(([dom.get_populations()], dom.residual(), dom.time))
        dom.close()
    equal(got)


def test_batch_in_l2(B):
    probs = [problem(401, 611, "crystal"), problem(523, 499, "pipe", temperature=False),
             problem(300, 701, "annulus-mixed", collision="mrt", tau=0.55), problem(1, 1, "closed")]
    states = [seeded_state(pb, 60 + d) for d, pb in enumerate(probs)]
    got = []
    for graphs in (True, False):
        batch = B.Batch(probs, "fp32")
        assert batch.step_form()[0] == L2
        batch.use_graphs(graphs)
        for d, (pb, st) in enumerate(zip(probs, states)):
            batch.set_populations(d, st.f, st.g, st.h if pb.temperature else None)
        for n in (1, 24, 13):
            batch.step(n)
        assert batch.graph_stats() == ((1, 2) if graphs else (0, 0))
        got.append(([batch.get_populations(d) for d in range(len(probs))], batch.residuals(), batch.time))
        batch.close()
    equal(got)


def test_small_batches_take_multi_step_launches(B):
    """The batches that test_gpu_resident.py compares."""
    for precision in ("fp32", "fp16"):
        batch = B.Batch([problem(17, 29, "crystal"), problem(143, 208, "pipe", temperature=False)], precision)
        assert batch.step_form()[0] in (ONE, SEVERAL)
        batch.step(1)
        batch.step(24)
        assert batch.graph_stats() == (1, 1)
        batch.close()


@pytest.mark.parametrize("precision", ["fp32", "fp64", "fp16", "bf16"])
@pytest.mark.parametrize("shape", [(1, 1), (64, 48), (128, 192), (199, 391)])
def test_zeros_keep_their_sign(B, shape, precision):
    """Bit for bit to the sign of zeros: swirl and temperature populations of either zero, on their way through the axis,
    off walls at rest and round periodic ends."""
    for mix in ("pipe", "crystal", "annulus-pipe"):
        pb = problem(*shape, mix)
        pb.omega, pb.t_wall, pb.t_ref, pb.gbeta = {}, {"outer": 0.0}, 0.0, 0.0
        st = seeded_state(pb, 21)
        rng = np.random.default_rng(5)
        st.g[...] = np.where(rng.random(st.g.shape) < 0.5, 0.0, -0.0)
        st.h[...] = np.where(rng.random(st.h.shape) < 0.5, 0.0, -0.0)
        got = []
        for graphs in (True, False):
            dom = B.Domain(pb, precision)
            assert dom.step_form()[0] != STEPS
            dom.use_graphs(graphs)
            dom.set_populations(st.f, st.g, st.h, time=0)
            dom.step(11)
            got.append(dom.get_populations())
            dom.close()
        for u, v in zip(*got):
            assert np.array_equal(u.view(np.uint64), v.view(np.uint64))


def test_streams_and_threads(B):
    """Domains and a batch stepped by threads of their own, on streams of two priorities beside other work: each launch
    needs all its blocks on the card at once, whatever else runs, and ends with what it gives alone."""
    import threading

    import torch
    cases = [(problem(64, 48, "crystal"), "fp32"), (problem(128, 192, "crystal"), "fp32"),
             (problem(199, 391, "annulus-mixed"), "fp32"), (problem(199, 391, "crystal"), "fp64"),
             (problem(1001, 1201, "pipe", temperature=False, swirl=False), "fp32")]
    states = [seeded_state(pb, 70 + i) for i, (pb, _) in enumerate(cases)]

    def make(i, stream):
        (pb, precision), st = cases[i], states[i]
        with torch.cuda.stream(stream):
            dom = B.Domain(pb, precision, stream=stream)
            dom.set_populations(st.f, st.g if pb.swirl else None, st.h if pb.temperature else None, time=0)
        return dom

    want = []
    for i in range(len(cases)):
        dom = make(i, torch.cuda.Stream())
        dom.use_graphs(False)
        for _ in range(6):
            dom.step(34)
        want.append((dom.get_populations(), dom.residual()))
        dom.close()
    doms = [make(i, torch.cuda.Stream(priority=-(i % 2))) for i in range(len(cases))]
    assert {d.step_form()[0] for d in doms} == {CLUSTER, ONE, SEVERAL, L2}
    errors = []

    def run(dom):
        try:
            torch.cuda.set_device(0)
            for _ in range(6):
                dom.step(34)
        except Exception as e:  # noqa: BLE001 (reported below)
            errors.append(e)

    other = torch.cuda.Stream()
    a = torch.randn(4096, 4096, device="cuda")
    threads = [threading.Thread(target=run, args=(d,)) for d in doms]
    for t in threads:
        t.start()
    with torch.cuda.stream(other):
        for _ in range(20):
            a = torch.tanh(a @ a)
    for t in threads:
        t.join()
    assert not errors
    for dom, (pops, residual) in zip(doms, want):
        assert dom.residual() == residual
        for u, v in zip(dom.get_populations(), pops):
            assert (u is None and v is None) or np.array_equal(u, v)
        dom.close()
