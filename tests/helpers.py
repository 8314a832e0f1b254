"""Helpers shared by the GPU parity tests: build the same layer for the oracle (host) and for
the CUDA library (device) from one seeded synth dict, and the acceptance metric."""
import numpy as np

from oracle import oracle
from paper_2409_17066_b200 import synth

TOL = 2e-3   # acceptance bound on max|y_gpu - y_ref| / max|y_ref| over a call's whole output


def rel_err(y_gpu: np.ndarray, y_ref: np.ndarray) -> float:
    return float(np.max(np.abs(y_gpu.astype(np.float64) - y_ref)) / np.max(np.abs(y_ref)))


def sample_rows(M: int, n: int, seed: int = 0) -> np.ndarray:
    """Rows to check one by one: first, last, tile boundaries and random ones."""
    rng = np.random.default_rng(seed)
    fixed = [0, 1, M - 1, M - 2, M // 2, 127, 128, 129, 255, 256]
    fixed = [m for m in fixed if 0 <= m < M]
    rnd = rng.integers(0, M, size=max(0, n - len(fixed))).tolist()
    return np.array(sorted(set(fixed + rnd)), dtype=np.int32)


def x_as_float64(spec, x_np):
    if spec.x_dtype == "bf16":
        return synth.bf16_bits_to_f32(x_np).astype(np.float64)
    return x_np.astype(np.float64)


def batched_segments(spec, B: int, n_sm: int, concurrent: bool = False):
    """How the batched kernel deals out a layer, restated: for every CTA its pieces (tile, first and end k block); k blocks of a tile,
    tokens of a tile, whether tiles that are cut meet by flag order.  A test that is about pieces says with it what it reaches."""
    up = lambda a, b: -(-a // b)
    vecs, ks = {8: (16, 32), 6: (20, 64), 12: (10, 64)}[spec.v]
    token_tiles = up(B, 512)
    tile_n = up(up(B, token_tiles), 16) * 16
    kb = up(spec.N - spec.n_out, ks) + up(spec.n_out, ks)
    tiles = up(up(spec.M, spec.v), vecs) * token_tiles
    sums = spec.out_dtype == "fp32" and spec.M % 4 == 0                 # pieces add up in the output
    workers = min(n_sm, up(tiles * kb * ks, 128))
    share = tiles * kb * ks // workers
    in_order = sums and share >= 768 and not concurrent
    per_tile = 0
    if not in_order and tiles < workers:
        n = workers // tiles
        if up(kb, n) * ks - share <= (400 + tile_n * 5 // 4 if n == 1 else 96 if sums else 128 + tile_n // 8):
            per_tile, workers = n, tiles * n
    length = kb + (160 * tile_n // 512 + (0 if sums else 128 if spec.v == 8 else 224)) // ks
    each, rest = divmod(kb, per_tile) if per_tile else divmod(tiles * length, workers)

    def begin(w):
        if per_tile:
            tile, part = divmod(w, per_tile)
            return tile * kb + part * each + min(part, rest)
        tile, off = divmod(w * each + min(w, rest), length)
        return tile * kb + min(off, kb)

    ctas = []
    for w in range(workers):
        u, end, pieces = begin(w), begin(w + 1), []
        while u < end:
            stop = min(end, (u // kb + 1) * kb)
            pieces.append((u // kb, u % kb, stop - u // kb * kb))
            u = stop
        ctas.append(pieces)
    cut = any(begin(w) % kb for w in range(1, workers))
    return ctas, kb, tile_n, cut and in_order
