"""Forward calls captured into a CUDA graph after a warm-up with more tokens:
the replay on new inputs equals the direct call, on each kernel path."""

import numpy as np
import pytest

from paper_2608_02703_gb300 import archead
from synth import HeadShape, make_head, make_hidden
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

SHAPE = HeadShape(V=1000, d=512, core_rank=16, corr_rank=16, group_size=64)


@pytest.fixture(scope="module")
def pack():
    from paper_2608_02703_gb300.build import build

    build()
    p = archead.archead_pack_create(make_head(SHAPE, seed=9), SHAPE)
    yield p
    p.close()


@pytest.mark.parametrize("M", [40, 100, 200])
def test_prefill_replays_after_a_larger_warm_up(pack, M):
    import torch

    warm = gu.to_dev(make_hidden(SHAPE.d, 300, seed=1))
    x = gu.to_dev(make_hidden(SHAPE.d, M, seed=2))
    y = torch.empty((300, SHAPE.V), dtype=torch.float32, device="cuda")
    archead.archead_forward_path(pack, warm, 300, y, archead.OUT_FP32, archead.PATH_PREFILL)
    archead.archead_forward_path(pack, x, M, y, archead.OUT_FP32, archead.PATH_PREFILL)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        archead.archead_forward_path(pack, x, M, y, archead.OUT_FP32, archead.PATH_PREFILL)
    new = make_hidden(SHAPE.d, M, seed=3)
    x.copy_(gu.to_dev(new))
    y.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    got = y[:M].cpu().numpy().astype(np.float64)
    assert np.array_equal(got, gu.forward(pack, new, archead.OUT_FP32, archead.PATH_PREFILL))
