"""The rescore's ring transforms against the FP32 path's.

Both report the correlation coefficient of the winning pose in FP32, from
different ring-FFT code.  Each is off by at most
u (log2 N + rings + log2 M + 10) |A| |B|, u = 6e-8: under 1.5 x 5.2e-6 |A| |B| for
both together, and a particle of signal-to-noise ratio 50 has a coefficient of
more than 0.9 |A| |B|: 2e-5 of it holds.  The ring sets have every length from 8
(4 complex points) to the longest of M = 256 and M = 512, and the longest alone.
"""
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module")
def mra():
    import __graft_entry__ as entry
    entry.build()
    import paper_2011_05755_gb300 as m
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need CUDA")
    return m


@pytest.mark.parametrize("L,r1,r2,M", [(64, 1, 28, 256), (76, 33, 35, 256), (100, 1, 45, 512), (128, 41, 60, 512)])
def test_rescored_cc_equals_the_fp32_path(mra, L, r1, r2, M):
    refs, blob = synth.make_refs(4, L, blobs=12, sigma=(L / 24, L / 12), disc=L / 2.5, seed=710)
    imgs, _ = synth.make_particles(blob, 40, shift_range=1, mirror=True, snr=50.0, seed=711, noise_seed=712)
    refs, imgs = refs.float().contiguous().to(DEV), imgs.float().contiguous().to(DEV)
    got = []
    for precision in (mra.MRA_FP32, mra.MRA_BF16_RESCORE):
        al = mra.Aligner(L, r1, r2, 1, 1.0, 1.0, 1, precision)
        assert al.info["M"] == M
        al.set_refs(refs)
        got.append(mra.decode_poses(al.align(imgs)))
        al.close()
    a, b = got
    assert (abs(a["cc"] - b["cc"]) <= 2e-5 * abs(a["cc"])).all()
