"""The FP64 deviate's table at the edges of its segments (gen_erfcinv_f64.py):
the words whose m = 2 s + 1 or 2^32 - m are the first and last of each segment,
in the tails and around u = 1/2 and u = 1, against the oracle.  Tolerance: the
nine terms leave 2^-59, their evaluation and the oracle's Newton steps a few
units of 2^-53; 1e-18 absolute for the oracle near u = 1."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _edge_words():
    m = []
    for lz in range(1, 32):
        for j in range(33):
            n = (32 + j) << 26
            m += [(n >> lz) + d for d in (-3, -2, -1, 0, 1, 2, 3)]
    for j in range(65):
        m += [(1 << 32) - (j << 25) + d for d in (-3, -2, -1, 0, 1, 2, 3)]
    s = np.unique([v >> 1 for v in m if v > 0 and (v >> 1) < 2**31])
    return np.concatenate([s, 2**32 - 1 - s]).astype(np.uint32)


@pytest.mark.parametrize("half", [0, 1])
def test_fp64_deviate_at_segment_edges(orc, half):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1403_0711_gb300 import _build, coulps
    _build.build()
    w = np.array_split(_edge_words(), 2)[half]
    ref = np.array([orc.heatbath_noise(int(v)) for v in w])
    got = coulps.heatbath_noise(torch.from_numpy(w.view(np.int32)).cuda(), coulps.F64).cpu().numpy()
    assert np.all(np.abs(got - ref) <= 1e-14 * np.abs(ref) + 1e-18)
    assert np.all((got < 0) == (w < 2**31))
