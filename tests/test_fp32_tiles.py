"""Reference tiles of the FP32 contraction (M = 256).

The number of references picks tiles of 4 or of 8; both add a pair's bins in
the same order, so a reference's table does not depend on how many others
there are.
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


@pytest.mark.parametrize("K", [1, 4, 5, 8, 9, 12])
def test_tables_do_not_depend_on_the_tile(mra, K):
    refs, blob = synth.make_refs(13, 64, blobs=8, sigma=(3.0, 6.0), disc=16.0, seed=800)
    imgs, _ = synth.make_particles(blob, 3, shift_range=1, mirror=True, snr=1.0, seed=801, noise_seed=802)
    refs, imgs = refs.float().contiguous().to(DEV), imgs.float().contiguous().to(DEV)
    al = mra.Aligner(64, 1, 28, 1, 1.0, 1.0, 1, mra.MRA_FP32)
    al.set_refs(refs)
    want = al.debug_cc(imgs)[:, :K]
    al.set_refs(refs[:K].contiguous())
    assert torch.equal(al.debug_cc(imgs), want)
    al.close()
