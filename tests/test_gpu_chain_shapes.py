"""Launch shapes and sum formats of the chain kernels: clusters of 1, 2, 4 and 8 CTAs give the
same bits (all sums are integers), and forces far beyond thermal ones (the coarse words of
the partials, the pair-by-pair path of an item) match the FP64 oracle within the force
tolerance of 1e-5 of the rms force."""
import dataclasses

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

KT = 2.494


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    return torch


def cut(c, n):
    """The first n atoms of a chain."""
    kb, ka = (c.bonds < n).all(1), (c.angles < n).all(1)
    return dataclasses.replace(
        c, n_atoms=n, mass=c.mass[:n], charge=c.charge[:n], sigma=c.sigma[:n], eps=c.eps[:n],
        bonds=c.bonds[kb], b0=c.b0[kb], kb=c.kb[kb], angles=c.angles[ka], th0=c.th0[ka],
        kth=c.kth[ka], exclusions=c.exclusions[(c.exclusions < n).all(1)], x_native=c.x_native[:n],
        x_unfolded=c.x_unfolded[:n], contacts=c.contacts[(c.contacts < n).all(1)])


def system(c, R=1, **kw):
    import paper_1705_02180_gb300 as pkg
    x0 = np.tile(c.x_unfolded.astype(np.float32).astype(np.float64), (R, 1))
    v0 = c.velocities(R, KT, 3).astype(np.float32).astype(np.float64).reshape(-1, 3)
    s = pkg.System(topologies=[pkg.chain_topology(c)], replica_topology=[0] * R, x0=x0, v0=v0,
                   dt=0.002, gamma=1.0, kT=KT, seed=4, **kw)
    s.set_contact_bias([c.contacts], [c.x_native], k_R=0.1)
    return s


def evaluate(torch, s, X):
    U = torch.empty(len(X), dtype=torch.float64, device="cuda")
    F, Z = torch.empty_like(X), torch.empty_like(U)
    s.energy_forces(0, X, U, F, Z)
    torch.cuda.synchronize()
    return U.cpu().numpy(), F.cpu().numpy(), Z.cpu().numpy()


@pytest.mark.parametrize("n", [17, 129, 160, 161, 449, 560])
def test_frame_batches_of_every_cluster_size_agree(torch_cuda, n):
    torch = torch_cuda
    c = cut(synth.make_chain(35, seed=1), n)
    s = system(c)
    g = np.random.default_rng(2)
    X = torch.from_numpy((c.x_unfolded[None] + g.normal(0, 0.01, (180, n, 3))).astype(np.float32)).cuda()
    whole = evaluate(torch, s, X)  # one CTA per frame
    for m in (60, 20, 3, 1):       # two, four, eight
        part = evaluate(torch, s, X[:m].contiguous())
        for a, b in zip(whole, part):
            assert np.array_equal(a[:m], b)
    Fr, Er = oracle.ForceField.from_chain(c).forces(X[0].double().cpu().numpy())
    rms = np.sqrt((Fr ** 2).sum(1).mean())
    assert np.abs(whole[1][0] - Fr).max() <= 1e-5 * rms
    s.close()


@pytest.mark.parametrize("n", [96, 129, 193, 449, 560])
def test_resident_clusters_agree(torch_cuda, n):
    c = cut(synth.make_chain(35, seed=1), n)
    runs = []
    for kw in (dict(), dict(cluster_size=1), dict(cluster_size=2), dict(cluster_size=2, threads=256)):
        s = system(c, R=3, save_interval=10, max_frames=4, **kw)
        s.step(45)
        assert s.status()[0] == 0
        st, paths = s.get_state(), s.collect_paths()
        runs.append([st[k] for k in ("x", "v", "zm", "T")] +
                    [np.stack([p[k] for p in paths]) for k in ("frames", "z", "epot", "T")])
        s.close()
    for r in runs[1:]:
        for a, b in zip(runs[0], r):
            assert np.array_equal(a, b)


@pytest.mark.parametrize("scale", [0.93, 0.85, 0.7])
def test_large_forces_match_the_oracle(torch_cuda, scale):
    torch = torch_cuda
    c = synth.make_chain(19, seed=1)
    s = system(c)
    x = (scale * c.x_unfolded).astype(np.float32)
    X = torch.from_numpy(np.stack([x] * 200)).cuda()
    U, F, _ = evaluate(torch, s, X)
    U1, F1, _ = evaluate(torch, s, X[:1].contiguous())
    assert np.array_equal(F[0], F1[0]) and U[0] == U1[0] and np.array_equal(F[0], F[199])
    Fr, Er = oracle.ForceField.from_chain(c).forces(x.astype(np.float64))
    rms = np.sqrt((Fr ** 2).sum(1).mean())
    assert np.abs(F[0] - Fr).max() <= 1e-5 * rms
    assert np.abs(Fr).max() > 2000.0  # beyond the first coarse word
    s.close()


@pytest.mark.parametrize("n", [9, 64, 161, 257, 559])
def test_hvp_of_every_cluster_size_agrees(torch_cuda, n):
    # 1e-5 of the rms, as for the other Hessian-vector products
    torch = torch_cuda
    c = cut(synth.make_chain(35, seed=1), n)
    s = system(c)
    g = np.random.default_rng(6)
    X = torch.from_numpy((c.x_unfolded[None] + g.normal(0, 0.01, (180, n, 3))).astype(np.float32)).cuda()
    V = torch.from_numpy(g.normal(0, 1, (180, n, 3)).astype(np.float32)).cuda()
    whole = torch.empty_like(X)
    s.hvp(0, X, V, whole)
    for m in (60, 20, 3):
        part = torch.empty_like(X[:m])
        s.hvp(0, X[:m].contiguous(), V[:m].contiguous(), part)
        assert torch.equal(whole[:m], part)
    W = V.clone()
    s.hvp(0, X, W, W)  # in place
    assert torch.equal(whole, W)
    _, ref = oracle.ForceField.from_chain(c).hvp(X[0].double().cpu().numpy(), V[0].double().cpu().numpy())
    assert np.abs(whole[0].cpu().numpy() - ref).max() <= 1e-5 * np.sqrt((ref ** 2).sum(1).mean())
    s.close()


def test_replicas_beyond_one_per_sm_agree(torch_cuda):
    # a few replicas more than SMs: some run as clusters of four beside the others
    n_sm = torch_cuda.cuda.get_device_properties(0).multi_processor_count
    c, R = cut(synth.make_chain(19, seed=1), 290), n_sm + 9
    runs = []
    for kw in (dict(), dict(cluster_size=1, threads=768)):
        s = system(c, R=R, save_interval=10, max_frames=4, **kw)
        assert s.info()["launch_groups"] == (1 if kw else 2)
        s.step(25)
        assert s.status()[0] == 0
        st, paths = s.get_state(), s.collect_paths()
        runs.append([st[k] for k in ("x", "v", "zm", "T", "step")] +
                    [np.stack([p[k] for p in paths]) for k in ("frames", "z", "epot", "T")])
        s.close()
    for a, b in zip(*runs):
        assert np.array_equal(a, b)
