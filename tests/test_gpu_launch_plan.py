"""Launch shapes that a system reports or that the tuner has cached mean the same launch again."""
import numpy as np
import pytest

import synth
from test_gpu_chain_shapes import cut, system, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu

SHAPE = ("plan", "cluster_size", "threads", "launch_groups")


@pytest.mark.parametrize("n,first", [(290, {}), (300, dict(cluster_size=1, threads=768))])
def test_a_cached_plan_is_the_plan_that_was_timed(torch_cuda, n, first):  # noqa: F811
    # a few replicas more than SMs: with the shape left open some run as clusters of four in a
    # launch of their own, with the shape given none do. The second system takes the plan of the first.
    n_sm = torch_cuda.cuda.get_device_properties(0).multi_processor_count
    c, R = cut(synth.make_chain(19, seed=1), n), n_sm + 9
    other = {} if first else dict(cluster_size=1, threads=768)
    got = []
    for kw in (first, other):
        s = system(c, R=R, **kw)
        t = s.autotune(probe_steps=20, use_cache=True)
        assert t["from_cache"] == len(got)
        got.append([s.info()[q] for q in SHAPE])
        s.close()
    assert got[0] == got[1]


def run(s):
    s.step(30)
    assert s.status()[0] == 0
    st = s.get_state()
    s.close()
    return [st[q] for q in ("x", "v", "zm", "T")]


@pytest.mark.parametrize("n,R", [(560, 1), (560, 24), (304, 6)])
def test_a_reported_shape_can_be_asked_for(torch_cuda, n, R):  # noqa: F811
    c = cut(synth.make_chain(35, seed=1), n)
    a = system(c, R=R)
    info = a.info()
    assert info["cluster_size"] >= 4
    b = system(c, R=R, cluster_size=info["cluster_size"], threads=info["threads"])
    assert [b.info()[q] for q in SHAPE] == [info[q] for q in SHAPE]
    for x, y in zip(run(a), run(b)):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("n", [17, 64, 129])
def test_more_ctas_than_tiles(torch_cuda, n):  # noqa: F811
    c = cut(synth.make_chain(35, seed=1), n)
    runs = [run(system(c, R=3, cluster_size=k)) for k in (1, 4, 8)]
    for r in runs[1:]:
        for x, y in zip(runs[0], r):
            assert np.array_equal(x, y)


def test_shapes_that_are_refused(torch_cuda):  # noqa: F811
    import paper_1705_02180_gb300 as pkg
    c = cut(synth.make_chain(35, seed=1), 64)
    for kw, code in ((dict(cluster_size=3), -7), (dict(cluster_size=16), -7), (dict(cluster_size=-1), -7),
                     (dict(cluster_size=8, threads=1024), -1),
                     (dict(cluster_size=4, exec_form=pkg.EXEC_PLAIN), -7),
                     (dict(cluster_size=4, box=9.0, elec=pkg.ELEC_RF), -7)):
        with pytest.raises(pkg.ScpsError) as e:
            system(c, **kw)
        assert e.value.code == code, kw


@pytest.mark.parametrize("n", [65, 100, 128, 300])
def test_shared_rows_of_hessian_vector_products(torch_cuda, n):  # noqa: F811
    # the warps of a cluster share the rows of small chains chunk by chunk: the same sums
    torch = torch_cuda
    c = cut(synth.make_chain(35, seed=1), n)
    s = system(c)
    g = np.random.default_rng(6)
    X = torch.from_numpy((c.x_unfolded[None] + g.normal(0, 0.01, (180, n, 3))).astype(np.float32)).cuda()
    V = torch.from_numpy(g.normal(0, 1, (180, n, 3)).astype(np.float32)).cuda()
    whole = torch.empty_like(X)
    s.hvp(0, X, V, whole)  # one CTA per frame
    for m in (152, 60, 20, 3):  # one with more threads, two, four, eight
        part = torch.empty_like(X[:m])
        s.hvp(0, X[:m].contiguous(), V[:m].contiguous(), part)
        assert torch.equal(whole[:m], part)
    s.close()
