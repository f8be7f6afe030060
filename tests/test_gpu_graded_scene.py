"""A scene whose triangles get smaller cluster by cluster, over up to thirty
orders of magnitude: the tree peels one cluster off per level, and a ray along
the axis enters every node's remainder before the cluster's pieces, which then
wait on the stack. Each closest-hit kernel gets through it, with the same
hits."""
import numpy as np
import pytest

from paper_2112_07115_gb300 import dcem, scenes

pytestmark = pytest.mark.gpu


def graded(levels, per, ratio, moving):
    """`levels` clusters of `per` triangles beside the x axis, whose boxes hold it."""
    tris = []
    for k in range(levels):
        s = 1000.0 * ratio ** k
        if s < 1e-30:
            break
        for j in range(per):
            x = s * (1.0 + (1.0 / ratio - 1.0) * (j + 0.5) / per)
            tris.append([(x, -s, -s), (x, s, -s), (x + 0.1 * s / per, s, 0.5 * s)])
    tris.append([(2500.0, -900.0, -900.0), (2500.0, 900.0, -900.0), (2500.0, 0.0, 900.0)])
    tris = np.asarray(tris, np.float32)
    return tris, np.full(len(tris), 0 if moving else -1, np.int32)


@pytest.mark.parametrize("levels,per,ratio", [(12, 8, 0.5), (40, 3, 0.5), (100, 8, 0.5), (60, 8, 0.1), (30, 64, 0.25)])
@pytest.mark.parametrize("moving", [False, True])
def test_stacks_hold_every_waiting_node(levels, per, ratio, moving):
    import torch
    tris, obj = graded(levels, per, ratio, moving)
    g = np.random.default_rng(levels * 100 + per)
    # rays about the axis, at all scales of the clusters
    y = np.exp(g.uniform(np.log(1e-12), np.log(0.5), (600, 2))) * g.choice([-1.0, 1.0], (600, 2))
    rays = np.concatenate([np.ones((600, 1)), y], 1).astype(np.float32)
    frames = []
    for kernel in (0, 1, 2):
        s = dcem.Scene(tris, np.zeros(len(tris), np.int32), [(5.0, 0.01, 0.0)], obj, int(moving),
                       torch.cuda.current_stream().cuda_stream)
        s.set_rays(rays)
        s.set_trace_config(kernel, 256, 8)  # the shortest stacks
        if moving:
            s.update_transforms(np.array([[1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0]], np.float32))
        f = s.trace((-1.0, 0.0, 0.0), np.array([[-2.0, 0.3, 0.2]], np.float32), dcem.default_params(max_refl=2))
        assert f.stats["stack_overflow"] == 0
        frames.append(s.ray_log())
        s.close()
    for a in frames[1:]:
        for x, y in zip(frames[0], a):
            assert np.array_equal(x, y, equal_nan=True)
