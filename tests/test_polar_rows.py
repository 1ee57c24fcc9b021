"""Rows per CTA of the polar kernel: an image's result does not depend on the call it is part of.

One image by itself runs with one row (shift) per CTA; a stack that fills the
GPU with as many rows as fit, groups that straddle the rows of the shift grid
and a ragged last group.  The arithmetic of a sample, a ring FFT and a pose
is the same in both, so the poses are equal bit for bit.
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


# (L, first, last ring, shift range, step, precision): integer grids with steps 1 and 2, a fractional
# grid, rows that are no multiple of 16 bytes, rings of every length class, one row per SM
CASES = [(32, 1, 12, 3.0, 1.0, "fp32"), (48, 1, 20, 4.0, 2.0, "bf16"), (32, 1, 12, 1.5, 0.5, "fp32"),
         (30, 1, 11, 2.0, 1.0, "bf16"), (96, 1, 44, 1.0, 1.0, "fp32"), (128, 1, 60, 1.0, 1.0, "bf16")]


@pytest.mark.parametrize("L,r1,r2,R,step,prec", CASES)
def test_alone_equals_in_a_stack(mra, L, r1, r2, R, step, prec):
    n = 600 if L < 90 else 320
    refs, blob = synth.make_refs(3, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=500)
    imgs, _ = synth.make_particles(blob, n, shift_range=int(R), mirror=True, snr=1.0, seed=501, noise_seed=502)
    imgs = imgs.float().contiguous().to(DEV)
    al = mra.Aligner(L, r1, r2, 1, R, step, 1, mra.MRA_FP32 if prec == "fp32" else mra.MRA_BF16_RESCORE)
    al.set_refs(refs.float().contiguous().to(DEV))
    whole = al.align(imgs)
    for i in (0, 1, n // 2, n - 1):
        assert torch.equal(al.align(imgs[i:i + 1].contiguous()), whole[i:i + 1]), i
    if prec == "fp32":
        assert torch.equal(al.debug_spectra(imgs[:400].contiguous())[:1], al.debug_spectra(imgs[:1].contiguous()))
    al.close()
