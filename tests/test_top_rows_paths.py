"""Row selection of the 16-bit paths by a warp or by a CTA per image: the same rows, so the same poses.

450 rows per image: a CTA each in a short call, a warp each in a call of more
images than CTAs fit on the GPU.  150 rows: a warp in both.  Zero images tie in every row.
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
    return m


@pytest.mark.parametrize("K,mirror", [(9, 1), (9, 0), (3, 1), (1, 0)])
def test_long_and_short_calls_pick_the_same_rows(mra, K, mirror):
    L, n = 32, 2000
    refs, blob = synth.make_refs(K, L, blobs=8, sigma=(2.0, 4.0), disc=8.0, seed=710)
    imgs, _ = synth.make_particles(blob, n, shift_range=2, mirror=bool(mirror), snr=0.3, seed=711, noise_seed=712)
    imgs = imgs.float().contiguous().to(DEV)
    imgs[1::500] = 0.0
    al = mra.Aligner(L, 1, 12, 1, 2.0, 1.0, mirror, mra.MRA_BF16_RESCORE, chunk_images=n)
    al.set_refs(refs.float().contiguous().to(DEV))
    whole = al.align(imgs)
    for at in (0, 700, 1400, 1900):
        assert torch.equal(al.align(imgs[at:at + 100].contiguous()), whole[at:at + 100]), at
    zero = mra.decode_poses(whole[1::500])
    for field in ("k", "shift_idx", "mirror", "ang_idx", "cc"):
        assert (zero[field] == 0).all(), field
    al.close()
