"""Sorted Morton keys around the sizes where the counting sort ends, with and
without ties, against the CPU twin's (whole numbers, equal), and the boxes of a
tree whose blocks are one cluster: unions of float32 boxes, exact."""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [31, 32, 33, 500, 12287, 12288, 12289])
@pytest.mark.parametrize("grid", [None, 3])
def test_keys(orc, n, grid):
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(n, 4)
    if grid:
        sc["mean"] = (np.round(sc["mean"] * grid) / grid).astype(np.float32)
    bvh = rt.rt_build_bvh(*(torch.from_numpy(np.ascontiguousarray(sc[k])).cuda()
                            for k in ("mean", "scale", "quat", "opacity")))
    ex = rt.rt_bvh_export(bvh)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(ex["keys"].cpu().numpy().view(np.uint64), orc.lbvh(sc["mean"])["keys"])


@pytest.mark.parametrize("n", [2, 3, 511, 512, 513, 1500, 2049, 3700, 4096, 4097])
def test_boxes(n):
    from paper_2311_16043_gb300 import rt
    sc = scenes.uniform_scene(n, 6)
    bvh = rt.rt_build_bvh(*(torch.from_numpy(np.ascontiguousarray(sc[k])).cuda()
                            for k in ("mean", "scale", "quat", "opacity")))
    ex = {k: v.cpu().numpy() for k, v in rt.rt_bvh_export(bvh).items()}
    boxes = ex["boxes"].reshape(n - 1, 2, 2, 3)  # side, lo / hi
    for side, refs in enumerate((ex["left"], ex["right"])):
        refs = refs.astype(np.int64) & 0xFFFFFFFF
        inner = refs < 0x80000000
        child = boxes[refs[inner]]
        np.testing.assert_array_equal(boxes[inner, side, 0], child[:, :, 0].min(1))
        np.testing.assert_array_equal(boxes[inner, side, 1], child[:, :, 1].max(1))
