"""Pair lists of the periodic box at the edges of the list build (few columns, ranges of
columns that wrap around a face, more candidate tiles than one segment holds): forces against
the FP64 oracle within the force tolerance of 1e-5 of the rms force."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solvent,cutoff,skin", [
    (1200, 0.4, 0.1),    # three columns a side, all in reach
    (4001, 0.3, 0.05),   # five columns, reach of one: ranges wrap
    (20003, 1.5, 0.2),   # reach of three of nine: several segments of candidate tiles
])
def test_box_lists_hold_every_pair(solvent, cutoff, skin):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1705_02180_gb300 as pkg
    b = synth.make_box(2, solvent, seed=3, cache=False)
    x = np.asarray(b.x, np.float32)
    t = b.topology()
    s = pkg.System(topologies=[t], replica_topology=[0], x0=x.astype(np.float64), cutoff=cutoff,
                   elec=pkg.ELEC_RF, box=b.box, dt=0.002, gamma=1.0, kT=2.494, seed=5, skin=skin)
    X = torch.from_numpy(x[None]).cuda()
    U = torch.zeros(1, dtype=torch.float64, device="cuda")
    F = torch.zeros_like(X)
    s.energy_forces(0, X, U, F)
    torch.cuda.synchronize()
    ff = oracle.ForceField(t["mass"], t["charge"], t["sigma"], t["eps"], t["bonds"], t["b0"], t["kb"],
                           t["angles"], t["th0"], t["kth"], t["excl"], cutoff=cutoff,
                           elec=oracle.ELEC_RF, box=b.box)
    Fr = ff.forces(x.astype(np.float64))[0]
    rms = np.sqrt((Fr ** 2).sum(1).mean())
    assert np.abs(F[0].cpu().numpy() - Fr).max() <= 1e-5 * rms
    s.close()
