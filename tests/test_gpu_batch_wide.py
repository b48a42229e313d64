"""The step kernels of batches whose planes reach 4 GiB (64-bit offsets in a
plane), at small size: the library runs them on request.  A batch of that
size holds 56 GB of populations.
"""
import numpy as np
import pytest

from parity_util import problem, seeded_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1003_0282_gb300 import build
    build.build()
    from paper_1003_0282_gb300 import axlbm
    return axlbm


WIDE = {
    "cold": [("closed", (37, 61), {"temperature": False}), ("pipe", (150, 40), {"temperature": False})],
    "mixed": [("crystal", (131, 47), {}), ("pipe", (64, 90), {"temperature": False}), ("annulus-mixed", (20, 33), {}),
              ("axis-node-crystal", (50, 26), {})],
    "wet": [("nee-cavity", (140, 30), {"temperature": False}), ("crystal", (33, 70), {})],
}


@pytest.mark.parametrize("precision", ["fp32", "fp16"])
@pytest.mark.parametrize("mix", sorted(WIDE))
def test_wide_offsets_match(B, precision, mix):
    """The step kernels of planes of 4 GiB or more against those of smaller ones, bit for bit, in every tile shape."""
    probs = [problem(*shape, name, collision="mrt" if name == "crystal" else "bgk", **extra)
             for name, shape, extra in WIDE[mix]]
    states = [seeded_state(pb, 80 + d) for d, pb in enumerate(probs)]
    for tile in [(4, 128), (8, 64)] + ([(8, 128)] if precision == "fp16" else []):
        got = []
        for wide in (True, False):
            batch = B.Batch(probs, precision)
            assert B.lib().axlbm_batch_set_tile_shape(batch.handle, *tile) == B.OK
            batch.wide_offsets(wide)
            batch.use_graphs(mix == "wet")  # (a batch with wet walls replays pairs of step kernels)
            for d, (pb, st) in enumerate(zip(probs, states)):
                batch.set_populations(d, st.f, st.g, st.h if pb.temperature else None)
            for n in (1, 4, 26):
                batch.step(n)
            got.append(([batch.get_populations(d) for d in range(len(probs))], batch.residuals()))
            batch.close()
        (p0, r0), (p1, r1) = got
        assert np.array_equal(r0, r1), tile
        for d, (x, y) in enumerate(zip(p0, p1)):
            for u, v in zip(x, y):
                assert (u is None and v is None) or np.array_equal(u, v), (tile, d)
