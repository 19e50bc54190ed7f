"""The top-B buckets of the calibration kernel on rows with an attention sink, as a
model of their arithmetic in fp32 with the source's own constants.  CPU only.

A bucket with more tokens than the kernel ranks pairwise costs two more passes and
two more cluster barriers, so the B-th score has to fall into a small one also
where five pooled sink tokens hold most of a row's mass."""
import re
from pathlib import Path

import numpy as np
import pytest

SRC = (Path(__file__).resolve().parents[1] / "paper_2606_01790_gb300" / "csrc" / "select.cu").read_text()


def _constant(name):
    return int(re.search(rf"constexpr int {name} = (-?\d+);", SRC).group(1))


def _tokens_in_the_bucket(x, shi, G, B, w, lam=0.5):
    """Tokens that share the bucket of the B-th largest of the scores x."""
    buckets, key_max = _constant("kBuckets"), 0x7FFFFFFF
    xhi = np.float32(shi) * np.float32((1 - lam) + lam * G)
    xlo = min(xhi * np.float32(2.0 ** -_constant("kTopOctaves")), np.float32(w / x.size) * np.float32(2.0 ** -_constant("kMeanOctaves")))
    bits = lambda v: np.asarray(v, np.float32).view(np.uint32).astype(np.int64)
    scale = np.float32(buckets) / (np.float32(bits(xhi) - bits(xlo)) + np.float32(1))
    u = key_max - bits(x)
    b = np.trunc((u - (key_max - bits(xhi))).astype(np.float32) * scale).clip(0, buckets - 1).astype(int)
    return int((b == b[np.argsort(u, kind="stable")[B - 1]]).sum())


@pytest.mark.parametrize("mass", [0.0, 0.5, 0.9, 0.99])
@pytest.mark.parametrize("G", [1, 4, 28])
@pytest.mark.parametrize("lp", [576, 5504, 14000, 56096])
def test_the_bth_score_has_a_small_bucket(lp, G, mass):
    w = 32
    rng = np.random.default_rng([lp, G])
    S = rng.lognormal(0.0, 1.0, (G, lp))
    S *= w * (1 - mass) / S.sum(1, keepdims=True)
    if mass:
        S[:, :5] = w * mass / 5
    S = S.astype(np.float32)
    x = S.mean(0, dtype=np.float32)   # beta = D = 1
    for pct in (10, 20, 40):
        assert _tokens_in_the_bucket(x, S.max(), G, lp * pct // 100, w) <= _constant("kCandMax")
