"""Launch shapes of the two-dimensional models: replica counts on both sides of a CTA, a warp
and the SM count, and tube paths on both sides of the line between one lane and one warp per
replica, of a block of 32 slices and of the slices kept in registers. Two steps from many
start points against the FP64 oracle; longer runs against the same run taken step by step.

Tolerance of the two steps: the curvature of the funnel is below 510 (its three terms at
their steepest), so a step stretches a difference by at most 1 + 510 dt = 11; a step itself
rounds about 50 operations on values below 400 dt, 5e-14 in all. Two steps stay below 6e-13:
1e-11 is asked for."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

DT, KT, SEED = 0.02, 0.3, 9


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    import paper_1705_02180_gb300 as p
    p.load()
    return p


def start(R):
    a = np.linspace(0.3, 5.9, R)
    return np.stack([4.0 * np.cos(a), 4.0 * np.sin(a)], axis=1)


def system(pkg, R, rid=None, x0=None, every=1, path=None):
    s = pkg.System(model=pkg.MODEL_FUNNEL2D, x0=start(R) if x0 is None else x0, replica_id=rid,
                   integrator=pkg.INT_EM, dt=DT, gamma=1.0, kT=KT, seed=SEED, save_interval=every,
                   max_frames=16)
    if path is not None:
        s.set_tube_bias(*path, 0.3, 3.0, 3.0, path[1][-1])
    else:
        s.set_radial_bias(70.0)
    return s


def tube(K):
    t = (np.arange(K) + 1) * 0.5
    return np.stack([0.4 * np.sin(t), 5.0 - 5.0 * t / t[-1]], axis=1), t


CASES = [(R, 0) for R in (1, 3, 153, 1217, 4865)] + [
    (1, 1), (33, 7), (5, 8), (153, 32), (7, 33), (610, 64), (3, 97), (9, 128), (4, 129), (2, 300)]


@pytest.mark.parametrize("R,K", CASES)
def test_two_steps_match_the_oracle(pkg, R, K):
    kw = dict(save_every=1, max_frames=2)
    if K:
        path, t = tube(K)
        ref = oracle.run_2d(oracle.MODEL_FUNNEL, oracle.BIAS_2D_TUBE, start(R), np.zeros(R),
                            np.arange(R), SEED, DT, 1.0, KT, 2, ref=path, tref=t, lam=0.3, k_s=3.0,
                            k_w=3.0, t_path=t[-1], **kw)
    else:
        ref = oracle.run_2d(oracle.MODEL_FUNNEL, oracle.BIAS_2D_RADIAL, start(R), np.zeros(R),
                            np.arange(R), SEED, DT, 1.0, KT, 2, k_R=70.0, **kw)
    s = system(pkg, R, path=tube(K) if K else None)
    s.step(2)
    got = s.get_state()
    assert s.status()[0] == 0
    assert np.abs(got["x"] - ref["x"]).max() < 1e-11
    assert np.allclose(got["T"], ref["T"], rtol=1e-9, atol=1e-10)
    for r, p in enumerate(s.collect_paths()):
        assert len(p["z"]) == 2
        assert np.abs(p["z"] - ref["z"][r]).max() < 1e-11
        assert np.abs(p["zmin"] - ref["zmin"][r]).max() < 1e-11
        assert np.abs(p["frames"][:, 0, :] - ref["frames"][r]).max() < 1e-6  # stored in FP32
    s.close()


@pytest.mark.parametrize("R,K", CASES)
def test_one_call_equals_single_steps(pkg, R, K):
    n, out = 70, []
    for parts in ([n], [1] * n):
        s = system(pkg, R, every=5, path=tube(K) if K else None)
        for k in parts:
            s.step(k)
        paths = s.collect_paths()
        out.append((s.get_state(), [np.stack([p[q] for p in paths]) for q in ("z", "zmin", "T", "frames")]))
        s.close()
    for k in ("x", "T", "step"):
        assert np.array_equal(out[0][0][k], out[1][0][k])
    for a, b in zip(out[0][1], out[1][1]):
        assert a.shape[1] == 14 and np.array_equal(a, b)


@pytest.mark.parametrize("K", [0, 5, 40])
def test_replica_ranges_are_bit_identical(pkg, K):
    R, lo, hi = 700, 331, 336
    out = []
    for ids in (np.arange(R), np.arange(lo, hi)):
        s = system(pkg, len(ids), rid=ids, x0=start(R)[ids], path=tube(K) if K else None)
        s.step(60)
        out.append(s.get_state())
        s.close()
    for k in ("x", "T", "step"):
        assert np.array_equal(out[0][k][lo:hi], out[1][k])
