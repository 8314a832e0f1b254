"""Argument marshalling of the extension module: what binding.py checked in Python is still checked, with the same exceptions."""
import pytest
import torch

from paper_2409_17066_b200 import synth


@pytest.fixture(scope="module")
def b():
    from paper_2409_17066_b200 import build as vbuild
    vbuild.build()
    from paper_2409_17066_b200 import binding
    return binding


def test_host_tensors_and_wrong_arguments_are_refused(b):
    d, p = b.make_desc(64, 64, 8, 256), b.LayerPtrs()
    x, out = torch.zeros((1, 64), dtype=torch.float16), torch.zeros((1, 64), dtype=torch.float16)
    with pytest.raises(AssertionError):
        b.vptq_linear(d, x, p, out, None)
    with pytest.raises(TypeError):
        b.vptq_linear(d, [0.0] * 64, p, out, None)
    with pytest.raises(TypeError):
        b.vptq_linear(bytearray(8), x, p, out, None)


@pytest.mark.gpu
def test_checks_on_the_device(b):
    spec = synth.small_specs()[0]
    d = synth.make_layer(spec, 91, 0, 2)
    dl = b.DeviceLayer(d)
    x = dl.upload_x(d["x"])
    y = dl.linear(x)
    assert y.shape == (2, spec.M) and y.dtype == torch.float16
    out = torch.empty_like(y)
    assert dl.linear(x, out) is out and torch.equal(out, y)
    for bad_x, bad_out in ((x.float(), None), (x[:, :-1].contiguous(), None), (x, out[:1]), (x, out.float()), (x.t().contiguous().t(), None)):
        with pytest.raises(AssertionError):
            dl.linear(bad_x, bad_out)
    fused = b.FusedLayers([dl, dl])
    with pytest.raises(ValueError):
        fused.linear(x, [out])
    with pytest.raises(b.VptqError) as e:
        b.vptq_linear(dl.with_flags(1 << 20).desc, x, dl.ptrs, out, None)
    assert e.value.code == b.E_UNSUPPORTED
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):                          # the call goes to the current stream
        z = dl.linear(x)
    side.synchronize()
    assert torch.equal(z, y)
