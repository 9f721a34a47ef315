"""Replicas that stop inside a call, in every cluster size: all CTAs of a cluster leave at the
same step with the same half of it done, and the other replicas of the launch go on.

The update that overflows: free atoms 50 nm apart (no pair, bond or contact: every force is
zero), dt = 1.5 / gamma, one atom of the odd replicas at v = 3e38. Its position after k updates
is the sum of 0.75 (1 + c1) c1^j 3e38 over j < k, c1 = exp(-1.5): 2.75e38, 3.37e38, and beyond
the FP32 range in the first half of the third. The other atoms of that replica have then taken three
updates; with zero force the closing half step changes nothing, so they stand where a run of
three steps leaves them, bit for bit."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N, BAD = 200, 137  # seven tiles of 32, one CTA holds the atom that overflows
# cluster sizes 1 and 2 as asked for, 4 and 8 as chosen for this many replicas
SHAPES = [(6, 1, 1), (6, 2, 2), (24, 0, 4), (6, 0, 8)]


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    import paper_1705_02180_gb300 as p
    p.load()
    return p


def gas(pkg, R, bad, cluster_size):
    none = dict(bonds=np.zeros((0, 2), np.int32), b0=[], kb=[], angles=np.zeros((0, 3), np.int32), th0=[],
                kth=[], excl=np.zeros((0, 2), np.int32))
    t = dict(mass=np.full(N, 10.0), charge=np.zeros(N), sigma=np.full(N, 0.3), eps=np.full(N, 0.5), **none)
    k = np.arange(N)
    x = 50.0 * np.stack([k % 6, k // 6 % 6, k // 36], axis=1)
    v = np.random.default_rng(1).normal(0.0, 0.5, (R, N, 3)).astype(np.float32).astype(np.float64)
    if bad:
        v[1::2, BAD] = (3e38, 0.0, 0.0)
    return pkg.System(topologies=[t], replica_topology=[0] * R, x0=np.tile(x, (R, 1)),
                      v0=v.reshape(-1, 3), dt=1.5, gamma=1.0, kT=2.494, seed=3, cluster_size=cluster_size)


@pytest.mark.parametrize("R,cluster_size,expected", SHAPES)
def test_overflow_in_the_update_stops_all_ctas_of_a_cluster_together(pkg, R, cluster_size, expected):
    s = gas(pkg, R, True, cluster_size)
    assert s.info()["cluster_size"] == expected
    s.step(12)
    rc, st = s.status()
    got = s.get_state()
    s.close()
    assert rc == -3 and np.array_equal(st, np.arange(R) % 2)  # 1: non-finite
    assert np.array_equal(got["step"], np.where(np.arange(R) % 2, 2, 12))
    for n, odd in ((3, 1), (12, 0)):
        s = gas(pkg, R, False, cluster_size)
        s.step(n)
        ref = s.get_state()
        s.close()
        others = np.arange(N) != BAD if odd else np.ones(N, bool)
        for q in ("x", "v"):
            a, b = (g[q].reshape(R, N, 3)[odd::2][:, others] for g in (got, ref))
            assert np.array_equal(a, b), q
    x = got["x"].reshape(R, N, 3)[1::2, BAD]
    assert not np.isfinite(x[:, 0]).any() and np.isfinite(x[:, 1:]).all()


def test_force_out_of_range_in_every_cluster_size(pkg):
    c = synth.make_chain(19, seed=1)
    x0 = np.stack([c.x_unfolded] * 2).astype(np.float32).astype(np.float64)
    x0[1, 3] += 1e30  # its bonds leave the fixed-point range at the first evaluation
    out = []
    for cluster_size, expected in ((1, 1), (2, 2), (0, 8)):
        s = pkg.System(topologies=[pkg.chain_topology(c)], replica_topology=[0, 0],
                       x0=x0.reshape(-1, 3), dt=0.002, gamma=1.0, kT=2.494, seed=11,
                       cluster_size=cluster_size)
        assert s.info()["cluster_size"] == expected
        s.step(5)
        rc, st = s.status()
        assert rc == -3 and st[0] == 0 and st[1] & 2
        out.append(s.get_state())
        s.close()
    assert np.isfinite(out[0]["x"][:c.n_atoms]).all() and out[0]["step"][0] == 5
    for g in out[1:]:
        for q in ("x", "v", "step"):
            assert np.array_equal(out[0][q], g[q], equal_nan=True), q
