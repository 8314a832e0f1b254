"""Decode over a table in L2 at row counts that do not divide over the SMs: fewer rows than SMs, one row more, a ragged last row,
less than a chunk of columns, two slabs, layers of uneven rows that share a launch, calls back to back without a pause."""
import ctypes as C

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
    (8, 32512, 1, dict(k2=256)),                        # 127 chunks of one row: 16 warps
    (8, 32513, 1, dict(k2=256)),                        # 128: 32 warps
    (2361, 16380, 1, dict(k2=200, x_dtype="bf16", out_dtype="fp32")),
    (1192, 36000, 1, dict(k2=256, permuted=True)),      # 32 warps, two slabs
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


@pytest.mark.parametrize("M,N,B,k2,out,perm", [
    (303109, 8200, 4, 256, "fp16", False),              # 37889 rows: the sums of one CTA no longer fit; two slabs; a short last row
    (303112, 72, 4, 0, "fp32", True),
    (606300, 40, 3, 0, "bf16", False),                  # two launches over one scratch, a token short
    (1212500, 300, 1, 200, "fp32", False),
])
def test_more_rows_than_their_sums_fit_shared_memory(M, N, B, k2, out, perm):
    """Tasks dealt out regardless of rows, partial sums in the workspace, against the plain kernel."""
    from paper_2409_17066_b200 import binding as b
    g = torch.Generator(device="cuda").manual_seed(M)

    def stream(rows, k):                                # any bytes are indices (clamped where k is no power of two); N % 8 == 0
        return torch.randint(0, 256, (rows, b.vptq_packed_row_bytes(N, k)), generator=g, dtype=torch.uint8, device="cuda")

    def normal(sd, *shape):
        return (torch.randn(shape, generator=g, device="cuda") * sd).half()
    R = -(-M // 8)
    parts = [stream(R, 65536), normal(0.02, 65536, 8), stream(R, k2) if k2 else None, normal(0.005, k2, 8) if k2 else None, None, None,
             normal(0.2, N) + 1, normal(0.01, N), torch.randperm(N, generator=g, device="cuda").int() if perm else None]
    ptrs = b.LayerPtrs(*[None if t is None else t.data_ptr() for t in parts])
    flags = b.FLAG_SCALE_BIAS | (b.FLAG_COL_PERM if perm else 0)
    desc = b.make_desc(M, N, 8, 65536, k2, out_dtype=out, flags=flags)
    plain = b.make_desc(M, N, 8, 65536, k2, out_dtype="fp32", flags=flags | b.FLAG_FORCE_GENERIC)
    assert b.vptq_linear_path(desc, B) == "decode_l2_fma"
    ws = torch.full((b.vptq_linear_workspace_bytes(desc, B),), 0x7F, dtype=torch.uint8, device="cuda")
    assert ws.numel() >= 4 * (4 if B == 4 else 2 if B > 1 else 1) * M
    ws_plain = torch.empty(b.vptq_linear_workspace_bytes(plain, B), dtype=torch.uint8, device="cuda")
    for _ in range(2):                                  # the second call finds the first one's sums and counts
        x = normal(1, B, N)
        y = torch.full((B, M), float("nan"), dtype=b._TORCH_DT[desc.out_dtype], device="cuda")
        want = torch.empty((B, M), dtype=torch.float32, device="cuda")
        b.vptq_linear(desc, x, ptrs, y, ws)
        b.vptq_linear(plain, x, ptrs, want, ws_plain)
        err = (y.float() - want).abs().max() / want.abs().max()
        assert float(err) <= (TOL if out != "bf16" else 2.0 ** -8)


def test_many_tasks_a_cta_in_shared_and_deterministic_launches():
    from paper_2409_17066_b200 import binding as b
    ds = [synth.make_layer(synth.LayerSpec("m%d" % i, M, 16384, v=8, k1=65536, k2=256), 102 + i, 0, 1) for i, M in enumerate((1200, 1181))]
    dls = [b.DeviceLayer(d) for d in ds]
    x = dls[0].upload_x(ds[0]["x"])
    fused = b.FusedLayers(dls)
    assert fused.path(1) == "fused_decode_l2_fma"
    ys = [torch.empty(1, d["spec"].M, dtype=torch.float16, device="cuda") for d in ds]
    fused.linear(x, ys)
    for d, dl, y in zip(ds, dls, ys):
        y_ref = oracle.Layer.from_synth(d).linear(ds[0]["x"])
        assert rel_err(y.float().cpu().numpy(), y_ref) <= TOL
        det = dl.with_flags(dl.desc.flags | b.FLAG_DETERMINISTIC)
        zs = [det.linear(x).clone() for _ in range(3)]
        assert all(torch.equal(z, zs[0]) for z in zs) and rel_err(zs[0].float().cpu().numpy(), y_ref) <= TOL


def test_deterministic_sums_take_nothing_from_the_previous_kernel():
    """Nine tasks for sixteen warps: the slots of warps without tasks hold what the previous kernel left in shared memory, here
    the residual table of a layer that leaves large values at that place on every SM."""
    from paper_2409_17066_b200 import binding as b
    fill = synth.make_layer(synth.LayerSpec("fill", 8 * 148, 16384, v=8, k1=65536, k2=256), 100, 0, 1)
    fill["c2"][:] = 60000.0                             # as FP32 pairs: 1.1e36
    spec = synth.LayerSpec("det", 1030, 2100, v=8, k1=65536, k2=256)
    d = synth.make_layer(spec, 101, 0, 1)
    filler, dl = b.DeviceLayer(fill), b.DeviceLayer(d)
    det = dl.with_flags(dl.desc.flags | b.FLAG_DETERMINISTIC)
    x, xf = dl.upload_x(d["x"]), filler.upload_x(fill["x"])
    y_ref = oracle.Layer.from_synth(d).linear(d["x"])
    for _ in range(3):
        filler.linear(xf)
        torch.cuda.synchronize()
        assert rel_err(det.linear(x).float().cpu().numpy(), y_ref) <= TOL
