"""vptq_dequant where its tasks have edges: columns per store (8 or 4, 2, 1), ragged last chunks and rows, outlier
columns that misalign the main ones, staged and unstaged tables, a group boundary inside a chunk."""
import numpy as np
import pytest

from oracle import oracle
from paper_2409_17066_b200 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,kw", [
    (8, 8, dict(v=8, k1=65536, k2=256)),                                                # one lane's columns
    (1203, 264, dict(v=8, k1=256)),                                                     # staged table, 16-byte stores, short last row
    (1200, 1022, dict(v=8, k1=4096, k2=300)),                                           # staged, 4-byte stores, residual without copies
    (131, 2051, dict(v=8, k1=65536, k2=256)),                                           # 2-byte stores
    (1501, 1000, dict(v=6, k1=4096, k2=256, n_out=9, v0=4, k0=4096)),                   # odd number of columns in front
    (4100, 1604, dict(v=12, k1=1000, k2=4096, n_out=13, v0=4, k0=8192, n_groups=3)),    # staged per group, 4 columns a lane
    (121, 1030, dict(v=12, k1=4096, n_out=2, v0=4, k0=64, n_groups=4)),                 # groups out of global memory
    (3000, 904, dict(v=6, k1=5000, k2=5000)),                                           # 13-bit indices
    (264, 520, dict(v=8, k1=65536, k2=256, has_scale=False)),
])
def test_restored_weight_is_bit_exact_at_the_edges_of_its_tasks(M, N, kw):
    from paper_2409_17066_b200 import binding as b
    spec = synth.LayerSpec("r", M, N, **kw)
    d = synth.make_layer(spec, 88, M % 7, 1)
    W = b.DeviceLayer(d).dequant().cpu().numpy()
    assert np.array_equal(W.view(np.uint16), oracle.Layer.from_synth(d).dequant().view(np.uint16))
