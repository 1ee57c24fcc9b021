"""mra_copy_refs between handles of every kernel choice.

The choices differ in speed and, at M = 256, in the order of the reference
fragments: a default handle and one the autotuner chose for share references
either way.
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


@pytest.mark.parametrize("L,r2,precision", [(76, 35, 1), (84, 40, 2), (76, 35, 0), (32, 12, 1), (96, 44, 1)])
def test_references_copied_between_all_kernels(mra, L, r2, precision):
    refs, blob = synth.make_refs(9, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=95)
    imgs, _ = synth.make_particles(blob, 6, shift_range=1, mirror=True, snr=1.0, seed=96, noise_seed=97)
    refs, imgs = refs.float().contiguous().to(DEV), imgs.float().contiguous().to(DEV)
    src = [mra.Aligner(L, 1, r2, 1, 1.0, 1.0, 1, precision, kernel=k) for k in (0, 1, 2)]
    dst = [mra.Aligner(L, 1, r2, 1, 1.0, 1.0, 1, precision, kernel=k) for k in (0, 1, 2)]
    for s in src:
        s.set_refs(refs)
    for i, d in enumerate(dst):
        want = src[i].debug_cc(imgs)  # the table with its own set_refs
        for s in src:
            d.copy_refs(s)
            assert torch.equal(d.debug_cc(imgs), want), (i, src.index(s))
            assert torch.equal(d.align(imgs), src[i].align(imgs))
    for h in src + dst:
        h.close()
