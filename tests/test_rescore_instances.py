"""A pose's last bits do not depend on which rescore instantiation an image's call takes.

Calls of a few images split an image's candidates over CTAs and use the plain
ring transform, larger ones (M >= 256) the transform with two stages per pass;
both kernels sample and transform with the same operations in the same order.
The stack sizes below take 8, 4, 2 and 1 CTAs per image.
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


@pytest.mark.parametrize("L,r2,R,step,prec", [(76, 35, 2.0, 1.0, "bf16"), (84, 40, 1.0, 1.0, "fp16"),
                                              (62, 26, 1.5, 0.5, "bf16"), (96, 44, 1.0, 1.0, "fp16")])
def test_parts_of_a_stack_equal_the_stack(mra, L, r2, R, step, prec):
    n = 1300
    refs, blob = synth.make_refs(5, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=510)
    imgs, _ = synth.make_particles(blob, n, shift_range=int(R), mirror=True, snr=0.5, seed=511, noise_seed=512)
    imgs = imgs.float().contiguous().to(DEV)
    al = mra.Aligner(L, 1, r2, 1, R, step, 1, mra.MRA_BF16_RESCORE if prec == "bf16" else mra.MRA_FP16_RESCORE)
    al.set_refs(refs.float().contiguous().to(DEV))
    whole = al.align(imgs)
    for size in (1, 60, 130, 280, 600):
        for at in (0, n - size):
            assert torch.equal(al.align(imgs[at:at + size].contiguous()), whole[at:at + size]), (size, at)
    al.close()
