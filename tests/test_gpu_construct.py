"""Offline construction on the GPU (paper Section 3.4, Algorithm 1) against
the construction oracle (oracle/construct.py):

- the library's quantisers, packers and dequantisers bit for bit on the same
  fp32 inputs (both take every integer decision in fp32);
- the whole construction (fp64 linear algebra on the GPU, the same random
  test matrices) giving the same stored arrays as the oracle, in both packed
  formats;
- the constructed head through archead_pack_create and the forward kernels
  against the forward oracle, and its error in the activation metric.
"""

import numpy as np
import pytest

import oracle
from oracle import construct as oc
from paper_2608_02703_gb300 import archead
from synth import HeadShape, make_dense_head, make_hidden, make_test_matrix
from tests import gpu_util as gu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2608_02703_gb300.build import build

    build()


def _dev(a):
    import torch

    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _inputs(seed, shape=(96, 64)):
    rng = np.random.default_rng(seed)
    x = (rng.standard_normal(shape) * np.exp2(rng.integers(-20, 8, shape))).astype(np.float32)
    x[:4, :8] = 0.0
    x[5, 3] = 1e-30  # far below the smallest fp16 scale step
    return x


@pytest.mark.parametrize("bits", [8, 5, 4])
@pytest.mark.parametrize("groups", [(1, 64), (1, 8), (96, 1), (8, 1), (4, 4)])
def test_quantiser_bit_exact(bits, groups):
    import torch
    from paper_2608_02703_gb300 import construct as gc

    x = _inputs(bits * 7 + groups[0])
    codes, scales = gc.quantize(_dev(x), groups[0], groups[1], bits)
    rq, rs = oc.quantize_symmetric(x, groups[0], groups[1], bits)
    assert np.array_equal(codes.cpu().numpy(), rq)
    assert np.array_equal(scales.cpu().numpy().view(np.uint16), rs)
    back = gc.dequantize(codes, scales, groups[0], groups[1])
    torch.cuda.synchronize()
    ref = rq.astype(np.float64) * np.repeat(np.repeat(rs.view(np.float16).astype(np.float64), groups[0], 0),
                                            groups[1], 1)
    assert np.array_equal(back.cpu().numpy().astype(np.float64), ref)


@pytest.mark.parametrize("g", [32, 64, 128])
def test_residual_quantiser_of_the_papers_format_bit_exact(g):
    import torch

    x = _inputs(g, (80, 512))
    rc = torch.empty((80, 512), dtype=torch.int8, device="cuda")
    rq = torch.empty((80, 512 // g), dtype=torch.uint8, device="cuda")
    rs = torch.empty(80, dtype=torch.int16, device="cuda")
    archead.archead_quantize_residual_sc4(_dev(x), g, rc, rq, rs)
    c, q, s = oc.quantize_residual_sc4(x, g)
    assert np.array_equal(rc.cpu().numpy(), c)
    assert np.array_equal(rq.cpu().numpy(), q)
    assert np.array_equal(rs.cpu().numpy().view(np.uint16), s)
    out = torch.empty((80, 512), dtype=torch.float32, device="cuda")
    archead.archead_dequant_residual_sc4(rc, rq, rs, g, out)
    sg = s.view(np.float16).astype(np.float64)[:, None] * (q.astype(np.float64) + 1)
    assert np.array_equal(out.cpu().numpy().astype(np.float64), c * np.repeat(sg, g, axis=1))


def _edge_values(seed, shape):
    """Values across many scales, near half-integers of their scale, zero groups and ties of the maximum."""
    rng = np.random.default_rng(seed)
    x = rng.standard_normal(shape).astype(np.float32)
    half = rng.random(shape) < 0.3
    x[half] = (rng.integers(-7, 7, shape)[half] + 0.5).astype(np.float32) * np.float32(0.25)
    x *= np.exp2(rng.integers(-30, 12, (shape[0], 1))).astype(np.float32)  # down to fp16 subnormal scales and below
    x[shape[0] // 2] = 0.0
    return x


def _quantise_at(x, gr, gc, bits, offset):
    """The quantiser on buffers that start `offset` elements past an allocation."""
    import torch

    R, C = x.shape
    xd = torch.empty(R * C + offset, dtype=torch.float32, device="cuda")
    xd[offset:] = _dev(x).view(-1)
    codes = torch.zeros(R * C + offset, dtype=torch.int8, device="cuda")
    scales = torch.zeros((R // gr, C // gc), dtype=torch.int16, device="cuda")
    view = codes[offset:].view(R, C)
    archead.archead_quantize_symmetric(xd[offset:].view(R, C), gr, gc, bits, view, scales)
    return view.cpu().numpy(), scales.cpu().numpy().view(np.uint16)


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("shape,groups,bits", [
    ((3, 32), (1, 32), 4), ((37, 192), (1, 64), 4), ((5, 1664), (1, 128), 8), ((9, 768), (1, 256), 5),  # rows
    ((511, 3), (511, 1), 8), ((512, 7), (512, 1), 8), ((4095, 16), (4095, 1), 5), ((4096, 16), (4096, 1), 8),
    ((20011, 13), (20011, 1), 8), ((1200, 24), (600, 1), 4),
    ((5 * 1216, 180), (1216, 1), 8), ((40 * 2048, 16), (2048, 1), 8),  # several groups
    # Kernels' outer loops several times over: rows, columns in three passes
    # (one group, two), columns in strips.
    ((20011, 1056), (1, 32), 4), ((262144, 4), (262144, 1), 8), ((40013, 128), (40013, 1), 8),
    ((2 * 6000, 1024), (6000, 1), 8), ((40000, 16), (40000, 1), 8),
    ((1215, 4), (1215, 1), 8), ((1216, 4), (1216, 1), 8), ((2432, 1024), (1216, 1), 5), ((9001, 200), (9001, 1), 8),  # columns
], ids=str)
def test_quantiser_routes_bit_exact(shape, groups, bits, offset):
    x = _edge_values(shape[0] + bits, shape)
    codes, scales = _quantise_at(x, *groups, bits, offset)
    rq, rs = oc.quantize_symmetric(x, groups[0], groups[1], bits)
    assert np.array_equal(scales, rs)
    assert np.array_equal(codes, rq)


def test_quantiser_routes_agree_on_values_that_are_not_finite():
    """The 16-byte route against the general kernel (which unaligned buffers take)."""
    x = _edge_values(1, (6, 256))
    x[1, ::7] = np.nan
    x[2, 3] = np.inf
    x[3] = np.nan
    x[4, 9] = 3e38
    a, b = _quantise_at(x, 1, 64, 4, 0), _quantise_at(x, 1, 64, 4, 1)
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])


def _residual_at(x, g, offset):
    """The paper's residual quantiser on buffers that start `offset` elements past an allocation."""
    import torch

    R, C = x.shape
    xd = torch.empty(R * C + offset, dtype=torch.float32, device="cuda")
    xd[offset:] = _dev(x).view(-1)
    rc = torch.zeros(R * C + offset, dtype=torch.int8, device="cuda")
    rq = torch.zeros((R, C // g), dtype=torch.uint8, device="cuda")
    rs = torch.zeros(R, dtype=torch.int16, device="cuda")
    view = rc[offset:].view(R, C)
    archead.archead_quantize_residual_sc4(xd[offset:].view(R, C), g, view, rq, rs)
    return view.cpu().numpy(), rq.cpu().numpy(), rs.cpu().numpy().view(np.uint16)


def _not_finite(seed, shape):
    x = _edge_values(seed, shape)
    x[1, ::7] = np.nan
    x[2, 3] = np.inf
    x[3] = np.nan
    x[4, 9] = 3e38
    x[5, 2:5] = -np.inf
    x[:, 6] = np.nan
    return x


@pytest.mark.parametrize("shape", [(1300, 12), (70000, 16), (9001, 120)])  # strips, three passes
def test_column_routes_agree_on_values_that_are_not_finite(shape):
    """Against the general kernel on the transpose (one group a row)."""
    x = _not_finite(2, shape)
    codes, scales = _quantise_at(x, shape[0], 1, 8, 0)
    rc, rs = _quantise_at(np.ascontiguousarray(x.T), 1, shape[0], 8, 0)
    assert np.array_equal(codes, rc.T) and np.array_equal(scales.ravel(), rs.ravel())


@pytest.mark.parametrize("cols,g", [(512, 32), (1024, 256), (4096, 64)])
def test_residual_routes_agree_on_values_that_are_not_finite(cols, g):
    x = _not_finite(3, (9, cols))
    for a, b in zip(_residual_at(x, g, 0), _residual_at(x, g, 1)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("rows,cols,g", [(10007, 256, 32), (9731, 1056, 32), (9800, 1024, 256)])
def test_sc4_residual_blocks_of_several_rows_bit_exact(rows, cols, g):
    """More rows than blocks: the next row's loads and the shared memory of a row after another."""
    x = _edge_values(rows, (rows, cols))
    for a, b in zip(_residual_at(x, g, 0), oc.quantize_residual_sc4(x, g)):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("cols,g", [
    (32, 32), (1024, 256), (1056, 32), (2112, 64), (4096, 128), (8192, 256), (8256, 64),
    (224, 32), (256, 32), (320, 64), (384, 64), (640, 128), (768, 128), (768, 256),  # rows too short for a block, and enough
])
def test_sc4_residual_row_widths_bit_exact(cols, g):
    import torch

    x = _edge_values(cols + g, (11, cols))
    rc = torch.empty(x.shape, dtype=torch.int8, device="cuda")
    rq = torch.empty((11, cols // g), dtype=torch.uint8, device="cuda")
    rs = torch.empty(11, dtype=torch.int16, device="cuda")
    archead.archead_quantize_residual_sc4(_dev(x), g, rc, rq, rs)
    c, q, s = oc.quantize_residual_sc4(x, g)
    assert np.array_equal(rs.cpu().numpy().view(np.uint16), s)
    assert np.array_equal(rq.cpu().numpy(), q)
    assert np.array_equal(rc.cpu().numpy(), c)


@pytest.mark.parametrize("cols,g", [(128, 128), (256, 64), (768, 256), (512, 32), (1024, 128)])
def test_sc4_residual_route_is_not_the_slower_one(cols, g):
    """Against the general kernel (which unaligned buffers take); narrow rows
    took a block each, up to 4.5 times as long."""
    import torch

    rows = 32000
    x = torch.randn(rows * cols + 1, device="cuda")
    rc = torch.empty(rows * cols, dtype=torch.int8, device="cuda")
    rq = torch.empty((rows, cols // g), dtype=torch.uint8, device="cuda")
    rs = torch.empty(rows, dtype=torch.int16, device="cuda")
    t = [gu.microseconds(lambda: archead.archead_quantize_residual_sc4(
        x[o:o + rows * cols].view(rows, cols), g, rc.view(rows, cols), rq, rs)) for o in (0, 1)]
    assert t[0] <= 1.25 * t[1], f"{t[0]:.1f} us against {t[1]:.1f}"


def test_column_route_of_many_groups_is_not_the_slower_one():
    """Against the strips of eight columns (which unaligned buffers take)."""
    import torch

    gr, groups, cols = 2048, 200, 32
    n = gr * groups * cols
    x = torch.randn(n + 1, device="cuda")
    codes = torch.empty((gr * groups, cols), dtype=torch.int8, device="cuda")
    scales = torch.empty((groups, cols), dtype=torch.int16, device="cuda")
    t = [gu.microseconds(lambda: archead.archead_quantize_symmetric(x[o:o + n].view(-1, cols), gr, 1, 8, codes, scales))
         for o in (0, 1)]
    assert t[0] <= 1.25 * t[1], f"{t[0]:.1f} us against {t[1]:.1f}"


@pytest.mark.parametrize("rows,cols", [(1, 16), (3, 32), (8, 2), (129, 1040), (3, 34)])
def test_nibble_packer_routes_bit_exact(rows, cols):
    from paper_2608_02703_gb300 import construct as gc

    c = np.random.default_rng(rows).integers(-8, 8, (rows, cols)).astype(np.int8)
    assert np.array_equal(gc.pack(_dev(c), 4).cpu().numpy(), oc.pack_int4(c))


def test_packers_bit_exact():
    from paper_2608_02703_gb300 import construct as gc

    rng = np.random.default_rng(3)
    c4 = rng.integers(-8, 8, (33, 70)).astype(np.int8)
    assert np.array_equal(gc.pack(_dev(c4), 4).cpu().numpy(), oc.pack_int4(c4))
    q = rng.integers(0, 16, (33, 5)).astype(np.int8)
    assert np.array_equal(gc.pack(_dev(q), 4).cpu().numpy(), oc.pack_scale_codes(q))
    for r in (1, 3, 10, 13, 64):
        c5 = rng.integers(-16, 16, (33, r)).astype(np.int8)
        assert np.array_equal(gc.pack(_dev(c5), 5).cpu().numpy(), oc.pack_int5(c5))


CASES = [
    ("int8", 1000, 256, 16, 8, 64),
    ("sc4", 700, 320, 10, 6, 64),
    ("int8", 513, 256, 0, 8, 32),
]


@pytest.mark.parametrize("fmt,V,D,rc,rr,g", CASES, ids=[f"{c[0]}-V{c[1]}-d{c[2]}-r{c[3]}-{c[4]}" for c in CASES])
def test_construction_matches_the_oracle(fmt, V, D, rc, rr, g):
    import torch
    from paper_2608_02703_gb300 import construct as gc

    N = 1024
    W = make_dense_head(V, D, seed=11)
    Hb = make_hidden(D, N, seed=11)
    H = oracle.bf16_values(Hb)
    om_c = make_test_matrix(D, rc + 10, seed=12) if rc else None
    om_r = make_test_matrix(D, rr + 10, seed=13)
    ref = oc.construct(W.astype(np.float64), H, rc, rr, g, fmt=fmt, omega_core=om_c, omega_corr=om_r)
    Hd = torch.from_numpy(Hb.view(np.int16)).cuda().view(torch.bfloat16).float()
    got = gc.construct(_dev(W), Hd, rc, rr, g, fmt=fmt, omega_core=_dev(om_c) if rc else None, omega_corr=_dev(om_r))
    got = gc.to_numpy(got)
    can = oc.canonical(ref)
    assert set(got) == set(can)
    for k in can:
        assert got[k].shape == can[k].shape and got[k].dtype == can[k].dtype, k
        mism = int(np.sum(got[k] != can[k]))
        assert mism == 0, f"{k}: {mism} of {can[k].size} entries differ"
    # the constructed head runs through the library like any other
    shape = HeadShape(V=V, d=D, core_rank=rc, corr_rank=rr, group_size=g, fmt=fmt)
    pack = archead.archead_pack_create(got, shape)
    try:
        x = make_hidden(D, 16, seed=14)
        yref = oracle.logits(can, shape, x)
        for M, path in ((16, archead.PATH_DECODE), (16, archead.PATH_PREFILL)):
            gu.check_logits(gu.forward(pack, x[:M], archead.OUT_FP32, path), yref[:M], where=f"{fmt} constructed")
    finally:
        pack.close()
    # the correction lowers the error in the activation metric
    Wq = oracle.dequant_rows(can, shape)
    T = ref["_T"]
    assert oc.metric_error(W, Wq, T) < 0.5 * oc.metric_error(W, ref["_W_d"], T)
