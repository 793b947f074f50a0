"""Run detection after the multi-kernel sort (129 workers: more than the resident sort takes): strips and steps of 256 keys
that lie inside a strip, begin or end one, or hold a segment's first key; runs of all lengths, up to one over many steps, and
keys that are all different.  Against the CPU checker."""
import numpy as np
import pytest

from tests.test_gpu_parity import _check_bwd

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,seed", [(3, 0), (400, 1), (1 << 22, 2)])
def test_strips_and_segments(V, seed):
    rng = np.random.default_rng(seed)
    sizes = np.array([0, 1, 127, 128, 129, 255, 256, 257, 511, 513, 4095, 4096, 4097, 8191, 33_000, 70_001] * 8 + [50_000])
    wso = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(wso[-1])
    ids = rng.integers(0, V, size=n).astype(np.int32)
    for w in range(0, len(sizes), 3):                  # runs of every length up to a whole list
        a, b = wso[w], wso[w + 1]
        ids[a:b] = np.sort(rng.choice([0, V - 1, int(V // 2)], size=b - a)) if w % 2 else V - 1
    off = np.arange(n + 1, dtype=np.int64)
    dY = rng.normal(size=(n, 4)).astype(np.float32)
    _check_bwd(ids, off, 1, dY, V, wso)
