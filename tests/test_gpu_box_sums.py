"""Force sums of the periodic box far outside the thermal range: terms of colliding sites, which
are taken pair by pair, against the FP64 oracle. Tolerances: the force tolerance of 1e-5 of
the rms force, over the colliding pair (13 powers of 1/r from an FP32 distance: 5e-6) and over
the other sites by themselves."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def sites(x, q, eps=0.5, sigma=0.2):
    n = len(x)
    z2, z3 = np.zeros((0, 2), np.int32), np.zeros((0, 3), np.int32)
    return dict(mass=np.full(n, 6.0), charge=q, sigma=np.full(n, sigma), eps=np.full(n, eps), bonds=z2, b0=[],
                kb=[], angles=z3, th0=[], kth=[], excl=z2)


def forces(torch, pkg, s, x):
    X = torch.from_numpy(np.asarray(x, np.float32)[None]).cuda()
    U = torch.zeros(1, dtype=torch.float64, device="cuda")
    F = torch.zeros_like(X)
    s.energy_forces(0, X, U, F)
    torch.cuda.synchronize()
    return F[0].cpu().numpy(), U.item()


def oracle_forces(t, x, **kw):
    ff = oracle.ForceField(t["mass"], t["charge"], t["sigma"], t["eps"], t["bonds"], [], [], t["angles"],
                           [], [], t["excl"], **kw)
    return ff.forces(np.asarray(x, np.float32).astype(np.float64))[0]


@pytest.mark.parametrize("r", [0.06, 0.033, 0.0305])  # 7.5e8, 1.8e12, 5e12 kJ mol^-1 nm^-1
def test_colliding_sites(r):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_02180_gb300 as pkg
    L, m = 3.2, 9
    k = np.arange(m ** 3)
    x0 = (np.stack([k % m, k // m % m, k // m ** 2], 1) + 0.5) * (L / m)
    x0 += np.random.default_rng(4).uniform(-0.02, 0.02, x0.shape)
    t = sites(x0, np.where(k % 2, 0.4, -0.4))
    x = x0.copy()
    x[300] = x[301] + r * np.array([1.0, 2.0, -2.0]) / 3.0
    s = pkg.System(topologies=[t], replica_topology=[0], x0=x0, cutoff=1.0, elec=pkg.ELEC_RF, box=L,
                   dt=0.002, gamma=1.0, kT=2.494, seed=5)
    plain, U0 = forces(torch, pkg, s, x0)
    F, _ = forces(torch, pkg, s, x)
    Fr = oracle_forces(t, x, cutoff=1.0, elec=oracle.ELEC_RF, box=L)
    pair = np.isin(k, (300, 301))
    for sel in (pair, ~pair):
        rms = np.sqrt((Fr[sel] ** 2).sum(1).mean())
        assert np.abs(F[sel] - Fr[sel]).max() <= 1e-5 * rms
    again, U1 = forces(torch, pkg, s, x0)  # nothing of the collision is left
    assert np.array_equal(plain, again) and U0 == U1
    s.close()


def test_more_lists_than_the_coarsest_unit_allows():
    # A strongly charged site in the focus of a ring of 25 800 weakly charged ones, all later in slot
    # order than the ring: it is in some 3 200 lists, each of which adds a force below half the
    # coarsest unit (128 kJ mol^-1 nm^-1) with the same sign, 2.86e5 in all: beyond the 2^31 units
    # of 2^-13 that the modular word holds. (A ring, so that no single list holds all of it.) Its
    # force is the plain shifted-force Coulomb sum (no LJ), in FP64 from the FP32 positions.
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_02180_gb300 as pkg
    L, rc, n, shells = 5.0, 2.0, 25800, 6
    k = np.arange(n // shells) + 0.5
    c0, c1 = np.cos(np.radians((40.0, 50.0)))
    cos = c0 - k / len(k) * (c0 - c1)  # Fibonacci points between 40 and 50 degrees from -x
    phi, sin = np.pi * (1.0 + 5.0 ** 0.5) * k, np.sqrt(1.0 - cos * cos)
    ring = np.stack([-cos, sin * np.cos(phi), sin * np.sin(phi)], 1)
    focus = np.array([4.2, 2.5, 2.5])
    x = np.concatenate([[focus]] + [focus + r * ring for r in np.linspace(1.78, 1.82, shells)])
    x = x.astype(np.float32).astype(np.float64)
    q = np.full(len(x), 0.001)
    q[0] = 1930.0
    t = sites(x, q, eps=0.0)
    s = pkg.System(topologies=[t], replica_topology=[0], x0=x, cutoff=rc, elec=pkg.ELEC_PLAIN, box=L, dt=0.002,
                   gamma=1.0, kT=2.494, seed=5, skin=0.05, save_interval=1, max_frames=1)
    F, _ = forces(torch, pkg, s, x)
    s.step(1)
    assert s.status()[0] == 0  # (the lists fit)
    s.close()
    d = x[0] - x[1:]
    r = np.linalg.norm(d, axis=1)
    ref = (138.935458 * q[0] * q[1] * (1.0 / r ** 2 - 1.0 / rc ** 2) / r)[:, None] * d
    assert 2.0 ** 31 / 8192 < ref.sum(0)[0] and 8 * ref[:, 0].max() < 128.0
    assert np.abs(F[0] - ref.sum(0)).max() <= 1e-5 * np.abs(ref.sum(0)).max()
