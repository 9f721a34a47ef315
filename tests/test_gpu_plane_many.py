"""Tube bias of the two-dimensional models with so many replicas that they run one per lane: the
same bits as the same replicas run a few at a time, one per warp."""
import numpy as np
import pytest

from test_gpu_plane import pkg, start, system, tube  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,K", [(4000, 8), (9001, 33), (24000, 100)])
def test_many_replicas_equal_a_few(pkg, R, K):  # noqa: F811
    ids = np.r_[0:40, R // 2:R // 2 + 40, R - 40:R]
    out = []
    for rid in (np.arange(R), ids):
        s = system(pkg, len(rid), rid=rid, x0=start(R)[rid], every=7, path=tube(K))
        s.step(45)
        assert s.status()[0] == 0
        sel = ids if len(rid) == R else slice(None)
        st = s.get_state()
        out.append([st[q][sel] for q in ("x", "T", "step")])
        lo = s.collect_paths(rep0=len(rid) - 40, nrep=40)
        out[-1] += [np.stack([p[q] for p in lo]) for q in ("z", "zmin", "T", "frames")]
        s.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
