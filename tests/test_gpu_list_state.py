"""Lists over rebuilds: a rebuild on a side stream into a batch with many more pairs (lists
and workspace grow), evaluated at once on that stream, against a list built anew."""
import numpy as np
import pytest
import torch

from paper_2507_00528_gb300 import gnep, synth

pytestmark = pytest.mark.gpu

KW = dict(n_max=(4, 4), basis=(8, 8), hidden=30, seed=3)


def _spread(b, f):
    return synth.Batch(b.struct_off, b.pos * f, b.types, b.cell * f)


def test_growing_rebuild_on_a_side_stream():
    rng = np.random.default_rng(5)
    dense = synth.make_batch([300, 200, 400], [1, 2, 0], rng)
    m = gnep.GNEP(**KW)
    want = [t.clone() for t in m.forward(m.neighbors(gnep.DeviceBatch.from_host(dense)))]
    arg = gnep.DeviceBatch.from_host(dense)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    for _ in range(20):
        nl = m.neighbors(gnep.DeviceBatch.from_host(_spread(dense, 1.6)))
        few = nl.info()
        torch.cuda.synchronize()
        with torch.cuda.stream(side):
            nl.rebuild(arg)
            got = m.forward(nl)
            again = m.forward(nl)
        side.synchronize()
        assert nl.info()[0] > 2 * few[0] and nl.info()[1] > 2 * few[1]
        for out in (got, again):
            for x, y in zip(out, want):
                assert torch.equal(x, y)
