"""Kernel variants and dispatch rules at the sizes where they change: edges of tiles, remainders, the ends of a range.
Every comparison is bit for bit against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import assert_same_bits, dev, empty, host, ws

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.fixture(scope="module")
def det():
    import paper_2609_17380_b200 as d
    d.load()
    return d


def _sync():
    import torch
    torch.cuda.synchronize()


# chunk counts of a launch around the rule between the two hash kernels (a warp of eight chains per scheduler: 8 * 4 * SMs),
# tensors of one, two and three levels, an empty one, byte counts off the 4- and 64-byte grid, more tensors than one
# launch takes
@pytest.mark.parametrize("sizes", [
    [16, 0, 4096, 4095, 4097, 61, 64, 55, 56, 128 * 4096, 128 * 4096 + 1, 0],
    "edge", "edge+1", [128 * 128 * 4096 + 4096 + 48, 5000, 129 * 4096 + 3],
    [(37 * i) % 9000 for i in range(300)],
])
def test_hash_batch(det, sizes):
    if isinstance(sizes, str):
        edge = 8 * 4 * det.det_device_sm_count()
        sizes = [4096 * (edge - 200) + 4096 * (sizes != "edge"), 4096 * 199 + 777]
    rng = np.random.default_rng(len(sizes))
    blobs = [rng.integers(0, 256, n).astype(np.uint8) for n in sizes]
    tensors = [dev(b) for b in blobs]
    roots = empty((32 * len(sizes),), np.uint8)
    det.det_tensor_hash_batch(tensors, roots, ws(det.det_tensor_hash_batch_ws_bytes(tensors)))
    _sync()
    raw = host(roots).tobytes()
    for i, b in enumerate(blobs):
        assert raw[32 * i:32 * i + 32].hex() == oracle.tensor_hash(b), (i, sizes[i])
