"""The rounding of the warm-start network's forward pass stays what it was, at image
sides that the GEMMs' boxes of positions do not divide: a pre-activation whose rounding
changes its sign switches a ReLU, and gradient entries jump there.  (Channel counts
that are multiples of 16: the others pad the operands' rows differently.)

``golden/warmstart_bits.json`` holds checksums of predictions; ``python -m
tests.test_gpu_warmstart_bits`` prints those of the built library."""
import json
import os
import zlib

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "warmstart_bits.json")
CASES = [(72, 16, 1), (72, 32, 5), (104, 16, 3), (104, 32, 20), (136, 32, 1), (136, 32, 3), (160, 16, 1), (160, 32, 2),
         (128, 32, 1), (64, 16, 8)]          # image side, channels, batch


def _values(n, seed):
    """24-bit values in [-1, 1), the same on every machine."""
    x = (np.arange(n, dtype=np.uint64) + np.uint64(977 * seed + 1)) * np.uint64(0x9E3779B97F4A7C15)
    x ^= x >> np.uint64(29)
    x *= np.uint64(0xBF58476D1CE4E5B9)
    i = (x >> np.uint64(40)).astype(np.int64) - (1 << 23)
    return torch.from_numpy((i * 2.0 ** -23).astype(np.float32))


def _predict(m, c, B):
    from paper_1703_04446_gb300 import lgnk
    net = lgnk.WarmStart(m, c, B, 0.0625)
    net.set_params(_values(net.num_params, 1) * 0.125)
    T, R = (_values(B * m * m, s).reshape(B, m, m).cuda() for s in (2, 3))
    v = net.predict(T, R).cpu().numpy()
    net.close()
    return zlib.crc32(v.tobytes())


@pytest.mark.parametrize("m,c,B", CASES)
def test_predictions_keep_their_rounding(m, c, B):
    with open(GOLDEN) as f:
        assert _predict(m, c, B) == json.load(f)["%d %d %d" % (m, c, B)]


if __name__ == "__main__":
    print(json.dumps({"%d %d %d" % a: _predict(*a) for a in CASES}, indent=1))
