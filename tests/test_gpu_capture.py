"""Workspace of the forward calls: a pack that has seen M tokens holds the
scratch of every call of that kind (logits; or cross entropy and greedy) with
fewer, whichever kernel it takes, so a forward captured into a CUDA graph after
a warm-up with more tokens meets no growth; the replay on new inputs equals the
direct call."""

import numpy as np
import pytest

from paper_2608_02703_gb300 import archead
from synth import HeadShape, make_head, make_hidden, make_targets
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu

SHAPES = {
    # Partials of 16 tokens (decode kernel, 8 a tile) beyond the 1 MB minimum
    # and beyond those of 24 tokens (tensor-core kernel, 4 a tile).
    "many_tiles": HeadShape(V=140000, d=256, core_rank=8, corr_rank=8, group_size=64),
    # Pre-pass sums of 128 tokens beyond 1 MB and beyond the operand of 300.
    "wide": HeadShape(V=300, d=4096, core_rank=128, corr_rank=32, group_size=64),
    "sc4_wide": HeadShape(V=300, d=4096, core_rank=128, corr_rank=32, group_size=64, fmt="sc4"),
}
_heads = {}


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2608_02703_gb300.build import build

    build()
    yield
    _heads.clear()


@pytest.fixture
def new_pack():
    """Packs without any workspace yet."""
    packs = []

    def make(name):
        if name not in _heads:
            _heads[name] = make_head(SHAPES[name], seed=9)
        packs.append(archead.archead_pack_create(_heads[name], SHAPES[name]))
        return packs[-1]

    yield make
    for p in packs:
        p.close()


class _Call:
    """One forward on buffers of its own."""

    def __init__(self, pack, op, M, path=archead.PATH_AUTO, seed=1):
        import torch

        self.pack, self.op, self.M, self.path = pack, op, M, path
        self.x = gu.to_dev(make_hidden(pack.shape.d, M, seed=seed))
        self.targets = gu.to_dev(make_targets(pack.shape.V, M, seed=seed).astype(np.int32))
        n = M * pack.shape.V if op == "logits" else M
        self.out = torch.empty(n, dtype=torch.float32, device="cuda")
        self.index = torch.empty(M, dtype=torch.int32, device="cuda")

    def run(self):
        if self.op == "logits":
            archead.archead_forward_path(self.pack, self.x, self.M, self.out, archead.OUT_FP32, self.path)
        elif self.op == "ce":
            archead.archead_forward_ce_path(self.pack, self.x, self.M, self.targets, self.out, self.path)
        else:
            archead.archead_forward_argmax_path(self.pack, self.x, self.M, self.index, self.out, self.path)


@pytest.mark.parametrize("name,warm,calls", [
    ("many_tiles", ("ce", 17), [("ce", 16), ("argmax", 16), ("logits", 9), ("ce", 1)]),
    ("many_tiles", ("argmax", 24), [("argmax", 16), ("ce", 24), ("logits", 24)]),
    ("many_tiles", ("argmax", 64), [("ce", 64), ("ce", 33), ("ce", 32)]),
    ("wide", ("logits", 300), [("logits", 128), ("ce", 128), ("logits", 64), ("logits", 16)]),
    ("wide", ("ce", 129), [("argmax", 128), ("ce", 65), ("ce", 20)]),
    ("sc4_wide", ("logits", 300), [("ce", 128), ("logits", 16)]),
], ids=lambda v: str(v))
def test_no_growth_after_more_tokens(new_pack, name, warm, calls):
    pack = new_pack(name)
    _Call(pack, *warm).run()
    held = archead.archead_device_bytes(pack)
    for op, M in calls:
        _Call(pack, op, M).run()
        assert archead.archead_device_bytes(pack) == held, f"{op} of {M} tokens grew the workspace"
    assert archead.archead_sync_status(pack) == archead.OK


@pytest.mark.parametrize("name,warm,M,op,path", [
    ("many_tiles", 24, 16, "ce", archead.PATH_AUTO),
    ("many_tiles", 24, 16, "argmax", archead.PATH_DECODE),
    ("many_tiles", 24, 20, "logits", archead.PATH_PREFILL),
    ("wide", 300, 8, "logits", archead.PATH_AUTO),
    ("wide", 300, 40, "logits", archead.PATH_PREFILL),
    ("wide", 300, 100, "ce", archead.PATH_PREFILL),
    ("wide", 300, 200, "logits", archead.PATH_PREFILL),
], ids=str)
def test_replays_after_a_warm_up_with_more_tokens(new_pack, name, warm, M, op, path):
    import torch

    # (Kernels of this output and path are loaded on another pack.)
    other = _Call(new_pack(name), op, M, path)
    other.run()
    pack = new_pack(name)
    _Call(pack, op, warm).run()
    call = _Call(pack, op, M, path)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call.run()
    new = _Call(other.pack, op, M, path, seed=3)
    call.x.copy_(new.x)
    call.targets.copy_(new.targets)
    call.out.fill_(float("nan"))
    g.replay()
    new.run()
    torch.cuda.synchronize()
    assert torch.equal(call.out, new.out)
    if op == "argmax":
        assert torch.equal(call.index, new.index)


def test_capture_of_more_tokens_that_fit(new_pack):
    """Captured with more tokens than the pack has seen, within its workspace."""
    import torch

    pack = new_pack("many_tiles")
    other = _Call(new_pack("many_tiles"), "logits", 16, seed=2)
    other.run()
    _Call(pack, "logits", 1).run()
    call = _Call(pack, "logits", 16, seed=2)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call.run()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(call.out, other.out)


def test_pack_creation_while_another_stream_is_captured(new_pack):
    """Pack creation waits for its own stream only, so it runs beside a capture."""
    import torch

    want = _Call(new_pack("wide"), "logits", 8)
    want.run()
    side = torch.cuda.Stream()
    buf = torch.zeros(16, device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="relaxed"):
        buf += 1
        pack = archead.archead_pack_create(_heads["wide"], SHAPES["wide"], stream=side)
    try:
        got = _Call(pack, "logits", 8)
        got.run()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(got.out, want.out) and bool((buf == 1).all())
    finally:
        pack.close()
