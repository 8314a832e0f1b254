"""The tensor-core assignment where its tiles and lists have edges: the widest vectors (13 components, and 14 without the low half of
the norm), codebooks that end inside a stage, vectors that end inside a step, candidate lists that overflow, a workspace of the
centroid update that starts off a 16-byte boundary."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,v,k,sigma", [
    (26, 2050, 13, 1500, 0.02),
    (28, 2100, 14, 1024, 0.02),
    (14, 4097, 14, 3001, 1.0),
    (8, 4096, 8, 1025, 0.02),        # 16 steps exactly
    (4, 4099, 1, 1024, 1.0),
    (16, 2100, 4, 4097, 1.0),
])
def test_assign_tiles(M, N, v, k, sigma):
    from paper_2409_17066_b200 import binding as b
    rng = np.random.default_rng(k + v)
    W = rng.normal(0, sigma, (M, N)).astype(np.float16)
    Cb = rng.normal(0, sigma, (k, v)).astype(np.float16)
    assert b.vptq_assign_path(M, N, v, k) == "assign_tcgen05"
    assert np.array_equal(b.vptq_assign(torch.from_numpy(W).cuda(), v, torch.from_numpy(Cb).cuda()).cpu().numpy(), oracle.assign(W, v, Cb))


@pytest.mark.parametrize("k", [16383, 16384])                 # a warp a group, a lane a group
@pytest.mark.parametrize("copies,noise", [(1, 0.02), (3, 0.02), (8, 0.0)])
def test_assign_with_several_candidate_groups_a_vector(k, copies, noise):
    # centroids that come more than once, far apart in the table, and vectors that are centroids: ties and near ties across groups
    from paper_2409_17066_b200 import binding as b
    rng = np.random.default_rng(k + copies)
    base = rng.normal(0, 1, (k // copies + 1, 8))
    Cb = np.tile(base, (copies, 1))[rng.permutation((k // copies + 1) * copies)[:k]].astype(np.float16)
    W = (Cb[rng.integers(0, k, 4100)].astype(np.float64) + noise * rng.normal(0, 1, (4100, 8))).T.astype(np.float16)
    assert b.vptq_assign_path(8, 4100, 8, k) == "assign_tcgen05"
    assert np.array_equal(b.vptq_assign(torch.from_numpy(W.copy()).cuda(), 8, torch.from_numpy(Cb).cuda()).cpu().numpy(), oracle.assign(W.copy(), 8, Cb))


@pytest.mark.parametrize("spread", [0.0, 1e-3])
def test_assign_with_more_candidates_than_a_list_holds(spread):
    # all centroids (nearly) equal: every group stays within the filter's error of the best one
    from paper_2409_17066_b200 import binding as b
    rng = np.random.default_rng(7)
    W = rng.normal(0, 1, (16, 2100)).astype(np.float16)
    Cb = (rng.normal(0, 1, (1, 8)) + spread * rng.normal(0, 1, (8192, 8))).astype(np.float16)
    assert np.array_equal(b.vptq_assign(torch.from_numpy(W).cuda(), 8, torch.from_numpy(Cb).cuda()).cpu().numpy(), oracle.assign(W, 8, Cb))


def test_kmeans_update_with_an_unaligned_workspace():
    from paper_2409_17066_b200 import binding as b
    rng = np.random.default_rng(3)
    M, N, v, k = 50, 300, 6, 5000
    W = rng.normal(0, 1, (M, N)).astype(np.float16)
    Cb = rng.normal(0, 1, (k, v)).astype(np.float16)
    idx = rng.integers(0, 60, (9, N)).astype(np.int32)
    want = oracle.kmeans_update(W, v, idx, Cb, None).astype(np.float64)
    Wd, Id, Cd = torch.from_numpy(W).cuda(), torch.from_numpy(idx).cuda(), torch.from_numpy(Cb).cuda()
    need = b.lib.vptq_kmeans_update_workspace_bytes(v, k)
    ws = torch.empty(need + 4, dtype=torch.uint8, device="cuda")
    assert b.lib.vptq_kmeans_update(Wd.data_ptr(), M, N, v, Id.data_ptr(), None, k, Cd.data_ptr(), ws.data_ptr() + 4, C.c_size_t(need),
                                    torch.cuda.current_stream().cuda_stream) == b.OK
    got = Cd.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - want) <= 2.0 ** -10 * np.abs(want) + 1e-6)
