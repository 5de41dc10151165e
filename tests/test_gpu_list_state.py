"""What a list and the graphs captured on it keep over rebuilds: a rebuild on a side
stream into a batch with many more pairs (lists and workspace grow), evaluated at once
on that stream, against a list built anew; and training graphs over rebuilds that are
refused; and what an evaluation leaves in host and device outputs."""
import numpy as np
import pytest
import torch

from paper_2507_00528_gb300 import gnep, synth

from gpu_common import Case, small_cells_batch

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


@pytest.mark.parametrize("what", ["ends", "order", "type", "wrap", "nan"])
def test_training_graph_outlives_a_refused_rebuild(what):
    b = small_cells_batch()
    c = Case("nmax4_basis8_h30", b)
    sched = dict(lr_start=1e-3, lr_stop=1e-6, n_warmup=10, n_total=100)
    g = gnep.TrainGraph(c.m, c.nl, c.gpu_labels(), **sched)
    off, pos, typ = b.struct_off.copy(), b.pos.copy(), b.types.copy()
    if what == "ends":
        off[-1] -= 1
    elif what == "order":
        off[1] = off[2]
    elif what == "type":
        typ[5] = 7
    else:
        pos[3] = 100.0 if what == "wrap" else np.nan
    bad = synth.Batch(off, pos, typ, b.cell)
    with pytest.raises(gnep._lib.GnepError, match="INVALID_ARG"):
        c.nl.rebuild(gnep.DeviceBatch.from_host(bad))
    g.launch()
    d = Case("nmax4_basis8_h30", b)
    h = gnep.TrainGraph(d.m, d.nl, d.gpu_labels(), **sched)
    h.launch()
    assert torch.equal(g.loss, h.loss) and torch.equal(c.m.get_params(), d.m.get_params())
    c.nl.rebuild(gnep.DeviceBatch.from_host(b))
    with pytest.raises(gnep._lib.GnepError, match="rebuilt or retuned"):
        g.launch()


def test_outputs_to_host_and_device_agree():
    b = small_cells_batch()
    c = Case("nmax4_basis8_h30", b, labels=False)
    dev = c.m.forward(c.nl)
    host = [np.full(tuple(t.shape), -1.0, dtype=np.float32 if t.dtype == torch.float32 else np.float64) for t in dev]
    st = torch.cuda.current_stream().cuda_stream
    L = gnep._lib.load()
    gnep.check(L.gnep_forward(c.m.h, c.nl.h, *(h.ctypes.data for h in host), st))
    for d, h in zip(dev, host):
        np.testing.assert_array_equal(d.cpu().numpy(), h)
    # two outputs in host memory and two on the device, one of them off its alignment
    raw = torch.zeros(4 * b.n_atoms * 3 + 8, dtype=torch.uint8, device="cuda")
    Es, W = np.zeros(b.n_struct), torch.zeros(b.n_struct, 6, dtype=torch.float64, device="cuda")
    gnep.check(L.gnep_forward(c.m.h, c.nl.h, None, Es.ctypes.data, raw.data_ptr() + 2, W.data_ptr(), st))
    torch.cuda.synchronize()
    F = raw[2:2 + 4 * b.n_atoms * 3].cpu().numpy().tobytes()
    assert F == host[2].tobytes() and (Es == host[1]).all() and (W.cpu().numpy() == host[3]).all()
