"""Decode over tables in shared memory where its staging and its outlier pass have edges: more pieces of outlier rows than a
warp asks for in advance, rows that are not 16-byte aligned, a stored column order, more columns than one pass of the CTA
stages, more than one slab, small tables with and without copies."""
import ctypes as C

import pytest

from oracle import oracle
from paper_2409_17066_b200 import synth

from helpers import TOL, rel_err

pytestmark = pytest.mark.gpu

V6 = dict(v=6, k1=4096, k2=256, v0=1, k0=300)


@pytest.mark.parametrize("M,N,B,kw", [
    (7110, 72, 1, dict(V6, n_out=33)),                      # 3 pieces of up to 16 columns in each of 49 outlier rows per CTA
    (7110, 73, 3, dict(V6, n_out=17, permuted=True)),
    (1776, 4100, 1, dict(V6, n_out=16, v0=4)),              # staged 8 columns at a time ...
    (60, 4101, 1, dict(V6, n_out=5, v0=4)),                 # ... and one by one, in more than one round
    (60, 2056, 2, dict(V6, n_out=1, permuted=True)),
    (64, 12808, 4, dict(v=8, k1=256)),                      # two slabs
    (64, 12809, 4, dict(v=8, k1=256, x_dtype="bf16")),
    (40, 264, 2, dict(v=4, k1=512, k2=17, has_scale=False)),
])
def test_smem_decode_edges(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    d = synth.make_layer(synth.LayerSpec("se", M, N, **kw), 98, B, B)
    dl = b.DeviceLayer(d)
    assert b.vptq_linear_path(dl.desc, B) == "decode_smem_fma"
    y = dl.linear(dl.upload_x(d["x"]))
    assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(d["x"])) <= TOL


@pytest.mark.parametrize("k1", [200, 256, 257, 512, 1024, 1025])
@pytest.mark.parametrize("M,N,B,kw", [
    (4800, 2300, 1, dict(v=8)),                             # eight copies of a main table of up to 256 rows, four of 512, none of more
    (4001, 2303, 4, dict(v=6, k2=256, n_out=9, v0=4, k0=64)),   # too few reads for four tokens: none
    (900, 700, 2, dict(v=4, out_dtype="fp32")),             # too few reads
    (1000, 2300, 8, dict(v=8, k2=100)),                     # the tensor-core kernel: copies
    (1000, 1003, 13, dict(v=6)),                            # ... two copies of up to 257 rows, none
    (576, 2300, 2, dict(v=8)),                              # copies where less than half of the SMs have a row
    (7000, 9000, 3, dict(v=6, k2=256)),                     # two tokens a launch
    (7001, 7111, 4, dict(v=8, x_dtype="bf16", out_dtype="bf16")),   # four
])
def test_small_tables_in_copies(k1, M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    d = synth.make_layer(synth.LayerSpec("sc", M, N, k1=k1, **kw), 102, B, B)
    dl = b.DeviceLayer(d)
    assert b.vptq_linear_path(dl.desc, B) == ("decode_smem_fma" if B <= 4 else "decode_smem_mma")
    y = dl.linear(dl.upload_x(d["x"]))
    tol = TOL if kw.get("out_dtype") != "bf16" else 2.0 ** -8
    assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(d["x"])) <= tol


@pytest.mark.parametrize("M,N,B,kw", [                      # on 148 SMs:
    (2056, 9001, 16, dict(v=8, k1=256)),                    # two slabs, eight copies
    (4096, 6600, 16, dict(v=8, k1=256, out_dtype="fp32")),  # two slabs, one of them for the sake of eight copies
    (2056, 6700, 9, dict(v=8, k1=256)),                     # one slab that is nearly full, no copies
    (4096, 13000, 13, dict(v=8, k1=256, x_dtype="bf16")),   # three slabs
    (2500, 14300, 16, dict(v=7, k1=300)),                   # three slabs, four copies
    (2056, 20000, 16, dict(v=8, k1=4096, out_dtype="bf16")),    # five slabs
    (4600, 9003, 8, dict(v=6, k1=4096, k2=256, n_out=9, v0=4, k0=300)),    # two, outlier columns, up to 8 tokens
    (4096, 19000, 5, dict(v=8, k1=200, k2=100)),
    (500, 9000, 16, dict(v=4, k1=256)),
    (1000, 14001, 8, dict(v=4, k1=1024, k2=256)),
    (2400, 13000, 12, dict(v=4, k1=4096, k2=256)),          # four slabs
])
def test_tensor_core_decode_slab_by_slab(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    d = synth.make_layer(synth.LayerSpec("sl", M, N, **kw), 104, B, B)
    dl = b.DeviceLayer(d)
    assert b.vptq_linear_path(dl.desc, B) == "decode_smem_mma" and b.vptq_linear_launches(dl.desc, B) == 2
    assert b.lib.vptq_linear_has_status(C.byref(dl.desc), B) == 0           # not the batched kernel
    y_ref = oracle.Layer.from_synth(d).linear(d["x"])
    for _ in range(2):
        y = dl.linear(dl.upload_x(d["x"]))
        assert rel_err(y.float().cpu().numpy(), y_ref) <= (TOL if kw.get("out_dtype") != "bf16" else 2.0 ** -8)
