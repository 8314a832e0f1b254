"""The batched tensor-core kernel where its tiles and pieces have edges: every vector length it takes, tables staged and in
L2, outlier columns of both kinds, groups that end inside a column group, odd index widths, split tiles in every output type,
several token tiles, few tokens (the decode families it serves from 5 tokens on)."""
import ctypes as C

import numpy as np
import pytest

from oracle import oracle
from paper_2409_17066_b200 import synth

from helpers import TOL, batched_segments, rel_err

pytestmark = pytest.mark.gpu

V6 = dict(v=6, k1=4096, k2=256, n_out=7, v0=4, k0=4096)
V12 = dict(v=12, k1=4096, k2=4096, n_out=13, v0=4, k0=8192, n_groups=4)


@pytest.mark.parametrize("M,N,B,kw", [
    (130, 700, 17, V6),                                                           # one tile and a short last row
    (721, 1003, 300, dict(V6, out_dtype="fp32")),                                 # rows of an FP32 output that are no multiple of 4
    (720, 1301, 256, dict(V6, n_out=33, v0=3, k0=100, permuted=True)),            # outlier vectors that straddle the tiles
    (1210, 2100, 49, dict(v=6, k1=5000, k2=5000, out_dtype="bf16")),              # 13-bit indices, both tables padded in the workspace
    (900, 515, 33, dict(v=6, k1=256, out_dtype="fp32")),                          # staged with copies, no residual
    (1201, 1034, 40, dict(V12, out_dtype="bf16")),                                # groups that end inside a lane's 8 columns
    (2400, 2222, 530, V12),                                                       # two token tiles, split tiles
    (600, 640, 512, dict(v=12, k1=4096, out_dtype="fp32", has_scale=False)),      # no residual, no scale
    (1100, 1000, 64, dict(v=8, k1=256, k2=256, n_out=9, v0=5, k0=37)),            # outlier vectors of 5
    (1024, 2051, 97, dict(v=8, k1=4096, k2=4096, n_groups=3, x_dtype="bf16")),    # group-wise with v = 8
    (1000, 4100, 5, dict(v=8, k1=65536, k2=256)),                                 # the decode families' batches
    (1000, 1411, 16, dict(v=8, k1=65536, x_dtype="bf16", out_dtype="fp32")),
    (1300, 1500, 6, V12),
])
def test_batched_kernel_formats_and_edges(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("bf", M, N, **kw)
    d = synth.make_layer(spec, 89, B % 5, B)
    dl = b.DeviceLayer(d)
    y_ref = oracle.Layer.from_synth(d).linear(d["x"])
    x = dl.upload_x(d["x"])
    tol = TOL if spec.out_dtype != "bf16" else 2.0 ** -8
    for _ in range(2):                                  # the workspace is reused
        y = dl.linear(x)
        assert b.vptq_workspace_status(dl.workspace(B)) == b.OK
        assert rel_err(y.float().cpu().numpy(), y_ref) <= tol
    shared = dl.with_flags(dl.desc.flags | b.FLAG_CONCURRENT)
    assert b.lib.vptq_linear_waits_between_ctas(C.byref(shared.desc), B) == 0
    assert rel_err(shared.linear(x).float().cpu().numpy(), y_ref) <= tol


@pytest.mark.parametrize("M,N,B,kw", [
    (18816, 520, 40, dict(v=8, k1=65536)),                                        # on 148 SMs: a tile less than SMs, whole ones, one CTA each
    (18944, 520, 40, dict(v=8, k1=65536, out_dtype="bf16")),                      # as many tiles as SMs: the same
    (19065, 520, 33, dict(v=8, k1=65536, out_dtype="fp32")),                      # one more; rows of 4 bytes' alignment
    (9600, 300, 600, dict(v=8, k1=65536, k2=256)),                                # two token tiles
    (25000, 130, 520, dict(v=6, k1=256)),                                         # tiles of few k blocks: some whole, some cut
    (600, 9000, 24, dict(v=12, k1=512)),                                          # few tiles, many pieces each
    (40000, 72, 16, dict(v=8, k1=65536, out_dtype="fp32")),                       # segment after segment of one staged piece
    (40032, 40, 33, dict(v=8, k1=65536, out_dtype="fp32")),                       # ... of three; a quarter without rows at the end
])
def test_split_tiles_have_scratch_of_their_own(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    d = synth.make_layer(synth.LayerSpec("sl", M, N, **kw), 96, 0, B)
    dl = b.DeviceLayer(d)
    y_ref = oracle.Layer.from_synth(d).linear(d["x"])
    x = dl.upload_x(d["x"])
    tol = TOL if kw.get("out_dtype") != "bf16" else 2.0 ** -8
    for _ in range(2):                                  # the second call finds the first one's sums and counts
        assert rel_err(dl.linear(x).float().cpu().numpy(), y_ref) <= tol


@pytest.mark.parametrize("M,N,B,kw", [
    (1000, 1100, 32, dict(v=8, k1=65536, k2=256)),                                # the last tokens of the form for few tokens,
    (1000, 1100, 33, dict(v=8, k1=65536, k2=256)),                                # the first of the other one
    (726, 1100, 64, V6), (726, 1100, 65, V6),
    (724, 1100, 17, dict(V6, out_dtype="fp32")),                                  # pieces that add up in the output
    (1450, 2100, 256, V6), (1450, 2100, 257, V6),                                 # room for two sets of accumulators, for one; a piece a CTA
    (9600, 200, 20, dict(v=6, k1=512)),                                           # whole tiles, one CTA each
    (600, 70, 20, V12),                                                           # ... of two k blocks
    (7200, 2600, 20, dict(v=6, k1=4096, k2=5000)),                                # few tokens, residual table in L2: rows of 12 bytes, padded
    (1000, 1100, 20, dict(v=8, k1=1024, k2=4096)),                                # ... of 16
    (2048, 2048, 64, dict(v=8, k1=256, n_out=40, v0=4, k0=300)),                  # outlier columns past a k block of 32
    (700, 9000, 9, dict(V6, n_out=65, k0=5000)),                                  # 13-bit outlier indices, a k block and a column of them;
    (700, 9000, 8, dict(V6, n_out=8, k0=200)),                                    # ... 8 bits, in a call of the decode family's name
    (300, 9000, 16, dict(v=8, k1=512, out_dtype="bf16")),                         # a small layer of many slabs
])
def test_few_tokens_and_cuts_within_tiles(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    d = synth.make_layer(synth.LayerSpec("ft", M, N, **kw), 101, 0, B)
    dl = b.DeviceLayer(d)
    x, y_ref = dl.upload_x(d["x"]), oracle.Layer.from_synth(d).linear(d["x"])
    for _ in range(2):
        y = dl.linear(x)
        assert b.lib.vptq_linear_has_status(C.byref(dl.desc), B) == 1 and b.vptq_workspace_status(dl.workspace(B)) == b.OK
        assert rel_err(y.float().cpu().numpy(), y_ref) <= (TOL if kw.get("out_dtype") != "bf16" else 2.0 ** -8)


FP32 = dict(out_dtype="fp32")


@pytest.mark.parametrize("M,N,B,kw,pieces,in_order", [      # on 148 SMs
    (71990, 200, 40, dict(v=6, k1=512), 5, False),                                # accumulators in turn, both phases of both sets: v = 6, few tokens
    (71996, 200, 40, dict(v=6, k1=512, **FP32), 5, True),
    (71990, 130, 200, dict(v=6, k1=512, out_dtype="bf16"), 5, False),             # ... the other form
    (71996, 130, 200, dict(v=6, k1=512, **FP32), 5, True),
    (71990, 130, 200, dict(v=12, k1=512), 5, False),
    (71996, 130, 200, dict(v=12, k1=512, **FP32), 5, True),
    (76780, 66, 16, dict(v=8, k1=65536), 5, False),
    (76780, 66, 100, dict(v=8, k1=65536, **FP32), 5, False),
    (12797, 1500, 16, dict(v=8, k1=65536), 2, False),                             # fewer tiles than SMs, shares across their boundaries: a CTA ends one cut
    (12797, 1500, 40, dict(v=8, k1=65536, out_dtype="bf16"), 2, False),           # tile and begins the next, a slot per tile
    (11990, 1500, 16, V6, 2, False), (11989, 1900, 100, dict(V6, out_dtype="bf16"), 2, False),
    (9000, 1700, 100, dict(v=12, k1=4096), 2, False),
    (1300, 13000, 40, dict(v=6, k1=4096, **FP32), 2, True),                       # flag order, tiles of 120 rows: the last one ends in its quarter of 24
    (1300, 13000, 100, dict(v=6, k1=4096, **FP32), 2, True),
    (1304, 13000, 40, dict(v=12, k1=4096, **FP32), 2, True),
    (10550, 878, 256, dict(v=8, k1=4096, k2=256), 1, False),                      # whole tiles, one CTA each
])
def test_pieces_that_a_cta_takes_in_turn(M, N, B, kw, pieces, in_order):
    import torch
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("pt", M, N, **kw)
    d = synth.make_layer(spec, 105, 0, B)
    dl = b.DeviceLayer(d)
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    ctas, kb, tile_n, flags = batched_segments(spec, B, n_sm)
    assert b.lib.vptq_linear_waits_between_ctas(C.byref(dl.desc), B) == int(flags)
    if n_sm == 148:
        assert max(map(len, ctas)) == pieces and flags == in_order and (pieces < 5 or tile_n <= 256)
        assert pieces != 2 or any(len(c) == 2 and c[0][1] > 0 and c[1][2] < kb for c in ctas)
    y_ref = oracle.Layer.from_synth(d).linear(d["x"])
    x, tol = dl.upload_x(d["x"]), TOL if kw.get("out_dtype") != "bf16" else 2.0 ** -8
    for _ in range(2):
        y = dl.linear(x)
        assert b.vptq_workspace_status(dl.workspace(B)) == b.OK and rel_err(y.float().cpu().numpy(), y_ref) <= tol
    shared = dl.with_flags(dl.desc.flags | b.FLAG_CONCURRENT)
    assert b.lib.vptq_linear_waits_between_ctas(C.byref(shared.desc), B) == 0
    assert rel_err(shared.linear(x).float().cpu().numpy(), y_ref) <= tol


ANY = dict(V6, k1=1100, out_dtype="fp32")


@pytest.mark.parametrize("Ms,N,B,kw", [                     # staged tables of sizes that are no multiple of 128 bytes, FP32 results
    ((720,), 12000, 8, ANY), ((724,), 9000, 16, ANY),                             # calls of the decode family's name
    ((724,), 1003, 40, dict(ANY, k1=4096, k2=300)), ((720,), 1100, 100, dict(ANY, k1=1001)),
    ((1000,), 1100, 20, dict(v=8, k1=1100, k2=300, out_dtype="fp32")),
    ((1000,), 1100, 70, dict(v=8, k1=4095, out_dtype="fp32")), ((264,), 1003, 40, dict(v=8, k1=65536, k2=300, out_dtype="fp32")),
    ((520, 132), 1003, 17, ANY), ((520, 136), 1003, 70, dict(v=8, k1=1001, k2=75, out_dtype="fp32")),
])
def test_fp32_pieces_are_staged_where_the_copy_engine_can_read(Ms, N, B, kw):
    import torch
    from paper_2409_17066_b200 import binding as b
    ds = [synth.make_layer(synth.LayerSpec("al%d" % i, M, N, **kw), 103 + i, 0, B) for i, M in enumerate(Ms)]
    dls = [b.DeviceLayer(d) for d in ds]
    x, ys = dls[0].upload_x(ds[0]["x"]), [torch.empty(B, M, dtype=torch.float32, device="cuda") for M in Ms]
    if len(Ms) == 1:
        assert b.lib.vptq_linear_has_status(C.byref(dls[0].desc), B) == 1
        dls[0].linear(x, ys[0])
    else:
        fused = b.FusedLayers(dls)
        assert fused.path(B) == "fused_gemm_tcgen05"
        fused.linear(x, ys)
    for d, y in zip(ds, ys):
        assert rel_err(y.cpu().numpy(), oracle.Layer.from_synth(d).linear(ds[0]["x"])) <= TOL


@pytest.mark.parametrize("M,N,B,kw", [
    (1000, 1003, 40, dict(k1=40000, k2=129)),                                     # 16 and 8 bits, indices that need the clamp
    (136, 33, 17, dict(k1=32769)),                                                # 16 bits, one k block and a column more
    (130, 31, 300, dict(k1=65536, k2=256, out_dtype="fp32")),                     # fewer columns than a k block, fewer k blocks than producers
    (2056, 1411, 513, dict(k1=65536, k2=256, permuted=True, x_dtype="bf16")),
    (1000, 1003, 40, dict(k1=32768, k2=256)),                                     # just outside: 15 bits,
    (1000, 1003, 40, dict(k1=65536, k2=128, out_dtype="fp32")),                   # 7 bits,
    (1000, 1003, 40, dict(k1=65536, k2=257)),                                     # 9 bits,
    (1000, 1003, 40, dict(k1=65536, k2=256, n_out=9, v0=4, k0=37)),               # outlier columns,
    (1000, 1003, 40, dict(k1=65536, k2=256, n_groups=2)),                         # groups
])
def test_v8_kernel_for_16_and_8_bit_indices_and_its_neighbours(M, N, B, kw):
    from paper_2409_17066_b200 import binding as b
    d = synth.make_layer(synth.LayerSpec("v8", M, N, v=8, **kw), 99, 0, B)
    dl = b.DeviceLayer(d)
    y = dl.linear(dl.upload_x(d["x"]))
    assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(d["x"])) <= TOL


def test_batched_kernel_repeats_bit_for_bit_when_asked():
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("bd", 1210, 2100, **V6)
    d = synth.make_layer(spec, 90, 0, 100)
    dl = b.DeviceLayer(d)
    det = dl.with_flags(dl.desc.flags | b.FLAG_DETERMINISTIC)
    x = dl.upload_x(d["x"])
    ys = [det.linear(x).clone() for _ in range(3)]
    assert all(np.array_equal(y.cpu().numpy().view(np.uint16), ys[0].cpu().numpy().view(np.uint16)) for y in ys)
    assert rel_err(ys[0].float().cpu().numpy(), oracle.Layer.from_synth(d).linear(d["x"])) <= TOL


@pytest.mark.parametrize("Ms,N,B,kw,outs", [
    ((130, 2100, 721), 1003, 65, dict(V6), ("fp16", "fp32", "bf16")),             # the fewest tokens that share a launch
    ((1024, 8), 2056, 513, dict(v=8, k1=65536, permuted=True), ("fp16", "fp32")),  # two token tiles; a layer of one tile
    ((600, 1800, 600, 600), 1034, 130, dict(V12, permuted=True), ("fp32",) * 4),
    ((2048, 2048), 1000, 300, dict(v=8, k1=65536, k2=256), ("fp32", "fp32")),
    ((520, 130), 1003, 17, dict(V6), ("fp16", "fp32")),                           # small layers at few tokens
    ((520, 130), 1003, 5, dict(V6), ("fp16", "bf16")),
    ((1024, 264), 1411, 9, dict(v=8, k1=65536), ("fp16", "fp16")),
    ((600, 1300), 1034, 3, dict(V12), ("fp32", "bf16")),
])
def test_layers_that_share_a_batched_launch(Ms, N, B, kw, outs):
    import torch
    from paper_2409_17066_b200 import binding as b
    ds = [synth.make_layer(synth.LayerSpec("bl%d" % i, M, N, out_dtype=o, **kw), 91 + i, 0, B) for i, (M, o) in enumerate(zip(Ms, outs))]
    dls = [b.DeviceLayer(d) for d in ds]
    fused = b.FusedLayers(dls)
    assert fused.path(B) == "fused_gemm_tcgen05"
    assert b.vptq_linear_fused_launches([dl.desc for dl in dls], B) == 2
    types = dict(fp16=torch.float16, fp32=torch.float32, bf16=torch.bfloat16)
    ys = [torch.empty(B, M, dtype=types[o], device="cuda") for M, o in zip(Ms, outs)]
    for _ in range(2):
        fused.linear(dls[0].upload_x(ds[0]["x"]), ys)
    for d, y, o in zip(ds, ys, outs):
        y_ref = oracle.Layer.from_synth(d).linear(ds[0]["x"])
        assert rel_err(y.float().cpu().numpy(), y_ref) <= (TOL if o != "bf16" else 2.0 ** -8)


@pytest.mark.parametrize("N,B", [(512, 64), (1003, 257), (12800, 100), (12808, 70), (51201, 66)])
def test_column_orders_gathered_from_staged_rows(N, B):
    """4 rows of 12800 columns are the most that fit twice, 2 rows of 51200 the most that fit at all."""
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("cr", 24, N, v=8, k1=4096, n_out=5, v0=4, k0=64, permuted=True)
    d = synth.make_layer(spec, 97, 0, B)
    dl = b.DeviceLayer(d)
    y = dl.linear(dl.upload_x(d["x"]))
    assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(d["x"])) <= TOL


@pytest.mark.parametrize("Ms,B,kw", [((1000,), 5, dict(v=8, k1=65536)), ((1000,), 16, dict(v=8, k1=65536, out_dtype="fp32")), ((600,), 3, V12),
                                     ((1024, 264), 6, dict(v=8, k1=65536)), ((600, 1300), 3, V12)])
def test_calls_that_keep_a_status_word_set_it(Ms, B, kw):
    """What vptq_linear_has_status promises: the word an earlier error left behind is gone after a healthy call."""
    import torch
    from paper_2409_17066_b200 import binding as b
    ds = [synth.make_layer(synth.LayerSpec("st%d" % i, M, 1100, **kw), 98 + i, 0, B) for i, M in enumerate(Ms)]
    dls = [b.DeviceLayer(d) for d in ds]
    call = dls[0] if len(Ms) == 1 else b.FusedLayers(dls)
    if len(Ms) == 1:
        assert b.lib.vptq_linear_has_status(C.byref(call.desc), B) == 1
    else:
        assert b.lib.vptq_linear_fused_has_status(call.descs, call.n, B) == 1
    ws = call.workspace(B)
    ws.view(torch.int32)[0] = b.E_TIMEOUT
    assert b.vptq_workspace_status(ws) == b.E_TIMEOUT
    x = dls[0].upload_x(ds[0]["x"])
    outs = [torch.empty(B, M, dtype=b._TORCH_DT[dl.desc.out_dtype], device="cuda") for M, dl in zip(Ms, dls)]
    call.linear(x, outs[0] if len(Ms) == 1 else outs)
    assert call.workspace(B) is ws and b.vptq_workspace_status(ws) == b.OK
    for d, y in zip(ds, outs):
        assert rel_err(y.float().cpu().numpy(), oracle.Layer.from_synth(d).linear(ds[0]["x"])) <= TOL
