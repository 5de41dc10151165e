"""The harmonics of degrees 5 to 8 along bonds near the polar axis, where P_l' is steepest.
An atom with one neighbour has q_nl = g_n^2 for every l (addition theorem), so q_nl / q_n1
= 1 in exact arithmetic.  A homogeneous recurrence passes the rounding of the unit vector
(each component and 1 / r: at most 6e-8 RMS in |u|) on 2 l times, 1.2e-7 l, and its own
roundings come to about the same: 2.5e-7 l RMS holds both with a margin of half.  With
r^2 taken as 1 the factor is l (l + 1): an FP32 emulation gives 1.9e-6 at l = 6 and
3.2e-6 at l = 8, against 0.9e-6 and 1.4e-6 here."""
import numpy as np
import pytest

from paper_2507_00528_gb300 import gnep, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("l_max,four_body", [(6, False), (8, True)])
def test_dimers_near_the_pole(l_max, four_body):
    rng = np.random.default_rng(5)
    n = 1000
    tilt, phi, r = rng.uniform(0.0, 0.2, n), rng.uniform(0.0, 2 * np.pi, n), rng.uniform(2.3, 3.6, n)
    d = r[:, None] * np.stack([np.sin(tilt) * np.cos(phi), np.sin(tilt) * np.sin(phi), np.cos(tilt)], 1)
    pos = np.stack([4.5 - d / 2, 4.5 + d / 2], 1).reshape(-1, 3)
    b = synth.Batch(np.arange(0, 2 * n + 1, 2, dtype=np.int32), pos, rng.integers(0, 2, 2 * n).astype(np.int32),
                    np.repeat(9.0 * np.eye(3)[None], n, 0))
    m = gnep.GNEP(n_max=(4, 4), basis=(8, 8), hidden=30, l_max=l_max, four_body=four_body, seed=2)
    nl = m.neighbors(gnep.DeviceBatch.from_host(b))
    assert nl.info()[1] == 2 * n
    G = m.descriptors(nl).double().cpu().numpy()[:, 5:5 + 5 * l_max].reshape(2 * n, 5, l_max)
    ratio = G[:, :, l_max - 1] / G[:, :, 0]
    assert np.sqrt(np.mean((ratio - 1.0) ** 2)) < 2.5e-7 * l_max
