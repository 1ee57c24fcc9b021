"""CTAs of 8 or 16 warps in the polar kernel: the same spectra and poses.

Images with one row (no shifts) and small boxes take CTAs of 8 warps, the
others one of 16.  The row of an image without shifts is the centre row of the
same image on a shift grid; small boxes in long and short calls, and images
with 4 shifts, sit on either side of the rule.
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


# L, last ring: 56, 312, 696, 1,976, 5,560 and 17,080 samples a row
BOXES = [(12, 3), (24, 8), (32, 12), (60, 21), (76, 35), (128, 60)]


def _stack(L, n, seed):
    refs, blob = synth.make_refs(3, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=seed)
    imgs, _ = synth.make_particles(blob, n, shift_range=1, mirror=True, snr=1.0, seed=seed + 1, noise_seed=seed + 2)
    return refs.float().contiguous().to(DEV), imgs.float().contiguous().to(DEV)


@pytest.mark.parametrize("L,r2", BOXES)
def test_one_row_per_image_equals_the_centre_row(mra, L, r2):
    _, imgs = _stack(L, 40, 540)
    spectra = {}
    for R, step in ((0.0, 1.0), (2.0, 1.0), (3.0, 1.5), (6.0, 1.0)):  # 1, 25, 25 (fractional) and 169 rows
        al = mra.Aligner(L, 1, r2, 1, R, step, 1, mra.MRA_FP32)
        s = al.debug_spectra(imgs)
        spectra[R] = s[:, s.shape[1] // 2].clone()
        al.close()
    assert torch.equal(spectra[2.0], spectra[0.0])
    assert torch.equal(spectra[6.0], spectra[0.0])
    assert torch.equal(spectra[3.0], spectra[0.0])


@pytest.mark.parametrize("prec", ["fp32", "bf16"])
@pytest.mark.parametrize("L,r2,R,step", [(12, 3, 0.0, 1.0), (24, 8, 2.0, 1.0), (32, 12, 2.0, 1.0), (32, 12, 0.25, 0.5),
                                         (32, 12, 1.5, 0.5), (60, 21, 0.0, 1.0), (30, 11, 0.0, 1.0)])
def test_parts_of_a_stack_equal_the_stack(mra, L, r2, R, step, prec):
    n = 1500
    refs, imgs = _stack(L, n, 550)
    al = mra.Aligner(L, 1, r2, 1, R, step, 1, mra.MRA_FP32 if prec == "fp32" else mra.MRA_BF16_RESCORE, chunk_images=n)
    al.set_refs(refs)
    whole = al.align(imgs)
    for size in (1, 7, 200, 620):
        for at in (0, n - size):
            assert torch.equal(al.align(imgs[at:at + size].contiguous()), whole[at:at + size]), (size, at)
    al.close()
