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
