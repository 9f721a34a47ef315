"""Periodic boxes little wider than 2 (r_c + skin): the nearest image of an atom is often not that
of its cluster. Forces against the FP64 oracle within the force tolerance of 1e-5 of the rms
force; energies of frames saved during a short run, which use the live lists, within 2e-5."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

KT = 2.494


@pytest.mark.parametrize("solvent,cutoff,skin", [
    (1200, 0.9, 0.2),   # L = 2.31 nm, 2 (r_c + skin) = 2.2
    (1200, 1.0, 0.1),
    (2500, 1.3, 0.15),  # L = 2.94
])
def test_smallest_boxes_match_the_oracle(solvent, cutoff, skin):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_02180_gb300 as pkg
    b = synth.make_box(2, solvent, seed=3, cache=False)
    x = np.asarray(b.x, np.float32)
    v = b.velocities(1, KT, 2).astype(np.float32).astype(np.float64)
    t = b.topology()
    s = pkg.System(topologies=[t], replica_topology=[0], x0=x.astype(np.float64), v0=v.reshape(-1, 3),
                   cutoff=cutoff, elec=pkg.ELEC_RF, box=b.box, dt=0.002, gamma=1.0, kT=KT, seed=5,
                   skin=skin, save_interval=15, max_frames=2)
    X = torch.from_numpy(x[None]).cuda()
    U = torch.zeros(1, dtype=torch.float64, device="cuda")
    F = torch.zeros_like(X)
    s.energy_forces(0, X, U, F)
    torch.cuda.synchronize()
    ff = oracle.ForceField(t["mass"], t["charge"], t["sigma"], t["eps"], t["bonds"], t["b0"], t["kb"],
                           t["angles"], t["th0"], t["kth"], t["excl"], cutoff=cutoff,
                           elec=oracle.ELEC_RF, box=b.box)
    Fr, Er = ff.forces(x.astype(np.float64))
    rms = np.sqrt((Fr ** 2).sum(1).mean())
    assert np.abs(F[0].cpu().numpy() - Fr).max() <= 1e-5 * rms
    assert abs(U.item() - Er.sum()) <= 2e-5 * abs(Er.sum())
    s.step(30)
    assert s.status()[0] == 0
    p = s.collect_paths()[0]
    s.close()
    for k in range(2):
        E = ff.forces(p["frames"][k].astype(np.float64))[1].sum()
        assert abs(p["epot"][k] - E) <= 2e-5 * abs(E)
