"""Decode over a table in L2 at row counts that do not divide over the SMs: fewer rows than SMs, one row more, a ragged last row,
less than a chunk of columns, two slabs, layers of uneven rows that share a launch, calls back to back without a pause."""
import pytest
import torch

from oracle import oracle
from paper_2409_17066_b200 import synth

from helpers import TOL, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,B,kw", [
    (8, 40, 1, dict()),
    (1180, 515, 2, dict(k2=256)),                       # 148 rows, the last one short
    (1192, 2048, 1, dict(k2=256, x_dtype="bf16")),      # 149 rows
    (600, 33000, 1, dict()),                            # two slabs
    (2400, 16640, 2, dict(k2=256, out_dtype="fp32")),
    (1000, 8200, 4, dict(out_dtype="bf16")),
    (1300, 1000, 3, dict(k2=200, has_scale=False)),
])
def test_rows_that_do_not_divide(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("l2", M, N, v=8, k1=65536, **kw)
    d = synth.make_layer(spec, 99, B, B)
    dl = b.DeviceLayer(d)
    assert b.vptq_linear_path(dl.desc, B) == "decode_l2_fma"
    x = dl.upload_x(d["x"])
    ys = [dl.linear(x) for _ in range(3)]               # dependent launches
    y_ref = oracle.Layer.from_synth(d).linear(d["x"])
    tol = TOL if spec.out_dtype != "bf16" else 2.0 ** -8
    assert all(rel_err(y.float().cpu().numpy(), y_ref) <= tol for y in ys)


@pytest.mark.parametrize("Ms,B", [((600, 592), 1), ((1184, 16, 8), 4)])
def test_uneven_rows_share_a_launch(Ms, B):
    from paper_2409_17066_b200 import binding as b
    ds = [synth.make_layer(synth.LayerSpec("l%d" % i, M, 1000, v=8, k1=65536), 99 + i, 0, B) for i, M in enumerate(Ms)]
    dls = [b.DeviceLayer(d) for d in ds]
    fused = b.FusedLayers(dls)
    assert fused.path(B) == "fused_decode_l2_fma"
    ys = [torch.empty(B, M, dtype=torch.float16, device="cuda") for M in Ms]
    fused.linear(dls[0].upload_x(ds[0]["x"]), ys)
    for d, y in zip(ds, ys):
        assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(ds[0]["x"])) <= TOL
