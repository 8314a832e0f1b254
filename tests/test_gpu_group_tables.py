"""Decode over group-wise tables staged in shared memory by clusters: every row width of a staged table, groups that start and
end inside a lane's eight columns, more columns than one slab, a stored column order, odd table sizes, two tokens, a fused
launch of several layers."""
import pytest
import torch

from oracle import oracle
from paper_2409_17066_b200 import synth

from helpers import TOL, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,B,kw", [
    (2403, 2111, 1, dict(v=12, k1=512, k2=256, n_out=13, v0=4, k0=512, n_groups=4)),
    (2400, 1333, 2, dict(v=12, k1=513, k2=255, n_out=7, v0=3, k0=100, n_groups=8, permuted=True)),
    (3000, 1500, 1, dict(v=16, k1=600, k2=600, n_groups=2)),
    (1501, 2050, 2, dict(v=14, k1=300, n_groups=4, x_dtype="bf16", out_dtype="fp32")),
    (1600, 1030, 1, dict(v=8, k1=4096, k2=16, n_groups=2)),
    (900, 900, 2, dict(v=10, k1=256, k2=256)),                                    # one group: no cluster
    (1200, 30011, 1, dict(v=12, k1=4096, k2=4096, n_groups=2)),                   # more columns than a slab holds
])
def test_staged_group_tables(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("gs", M, N, **kw)
    d = synth.make_layer(spec, 92, B, B)
    dl = b.DeviceLayer(d)
    assert b.vptq_linear_path(dl.desc, B) == "decode_gl_fma"
    y = dl.linear(dl.upload_x(d["x"])).float().cpu().numpy()
    assert rel_err(y, oracle.Layer.from_synth(d).linear(d["x"])) <= TOL


@pytest.mark.parametrize("B", [1, 2])
def test_staged_group_tables_fused(B):
    from paper_2409_17066_b200 import binding as b
    specs = [synth.LayerSpec("gf%d" % i, M, 1100, v=12, k1=512, k2=512, n_out=9, v0=4, k0=512, n_groups=4) for i, M in enumerate((2400, 2405, 1200))]
    ds = [synth.make_layer(sp, 93 + i, 0, B) for i, sp in enumerate(specs)]
    for d in ds[1:]:
        d["x"] = ds[0]["x"]
    fused = b.FusedLayers([b.DeviceLayer(d) for d in ds])
    assert fused.path(B) == "fused_decode_gl_fma"
    outs = [torch.full((B, sp.M), float("nan"), dtype=torch.float16, device="cuda") for sp in specs]
    fused.linear(fused.dls[0].upload_x(ds[0]["x"]), outs)
    for d, y in zip(ds, outs):
        assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(d["x"])) <= TOL
