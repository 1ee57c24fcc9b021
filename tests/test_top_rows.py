"""Row selection of the 16-bit paths where row maxima tie.

An image of zeros has the value 0 in every cell of its table: all rows tie,
more of them than the selection's list holds, and the smallest (reference,
shift, mirror, angle) wins.  Two copies of one reference tie row by row; the
first copy wins.
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


@pytest.mark.parametrize("L,r2,K,mirror", [(32, 12, 9, 1), (76, 35, 3, 0), (32, 12, 1, 0)])
def test_ties_keep_the_smallest_row(mra, L, r2, K, mirror):
    refs, blob = synth.make_refs(K, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=700)
    imgs, _ = synth.make_particles(blob, 4, shift_range=2, mirror=bool(mirror), snr=2.0, seed=701, noise_seed=702)
    refs, imgs = refs.float().contiguous().to(DEV), imgs.float().contiguous().to(DEV)
    al = mra.Aligner(L, 1, r2, 1, 2.0, 1.0, mirror, mra.MRA_BF16_RESCORE)
    al.set_refs(refs)
    zeros = mra.decode_poses(al.align(torch.zeros_like(imgs)))
    for field in ("k", "shift_idx", "mirror", "ang_idx", "cc"):
        assert (zeros[field] == 0).all(), field
    once = al.align(imgs)
    al.set_refs(torch.cat([refs, refs]))
    assert torch.equal(al.align(imgs), once)
    al.close()
