"""Reference tiles of the FP32 contraction (M = 256): tiles of 8 in short calls, of 4 in long ones at some K.

An image by itself fills no pass of the GPU and takes tiles of 8 references
whatever their number; a stack of 400 images takes tiles of 4 at K = 1, 4, 9
and 12.  A pair's bins are added in the same order in both.
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


@pytest.mark.parametrize("K", [1, 4, 5, 9, 12, 13])
def test_table_of_a_stack_equals_that_of_its_images(mra, K):
    n = 400
    refs, blob = synth.make_refs(K, 62, blobs=8, sigma=(3.0, 6.0), disc=16.0, seed=810)
    imgs, _ = synth.make_particles(blob, n, shift_range=1, mirror=True, snr=1.0, seed=811, noise_seed=812)
    imgs = imgs.float().contiguous().to(DEV)
    al = mra.Aligner(62, 1, 26, 1, 1.0, 1.0, 1, mra.MRA_FP32)
    al.set_refs(refs.float().contiguous().to(DEV))
    whole, poses = al.debug_cc(imgs), al.align(imgs)
    for i in (0, 1, 200, n - 1):
        one = imgs[i:i + 1].contiguous()
        assert torch.equal(al.debug_cc(one)[0], whole[i]), i
        assert torch.equal(al.align(one), poses[i:i + 1]), i
    al.close()
