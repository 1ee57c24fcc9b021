"""The M = 256 kernel where a CTA walks several units of several reference tiles.

A unit is a row tile and a range of reference tiles; the barriers of the row
fragments (in shared memory for rings beyond 36) go through several phases
only when a CTA takes more than one.  120 images x 25 shifts are 375 row
tiles, which a GPU of up to 187 SMs walks as at least two or three units of three
tiles per CTA; an image by itself is four row tiles, one unit a CTA.
"""
import os

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


def _stack(L, K, n, seed):
    refs, blob = synth.make_refs(K, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=seed)
    imgs, _ = synth.make_particles(blob, n, shift_range=2, mirror=True, snr=0.5, seed=seed + 1, noise_seed=seed + 2)
    return refs.float().contiguous().to(DEV), imgs.float().contiguous().to(DEV)


@pytest.mark.parametrize("L,r2,prec", [(84, 40, "bf16"), (80, 37, "fp16"), (64, 28, "bf16")])
def test_table_of_a_stack_equals_that_of_its_images(mra, L, r2, prec):
    refs, imgs = _stack(L, 17, 120, seed=520)
    al = mra.Aligner(L, 1, r2, 1, 2.0, 1.0, 1, mra.MRA_BF16_RESCORE if prec == "bf16" else mra.MRA_FP16_RESCORE)
    al.set_refs(refs)
    whole = al.debug_cc(imgs)
    mra.mra_sync(al.h)
    for i in (0, 1, 48, 60, 97, 118, 119):
        assert torch.equal(al.debug_cc(imgs[i:i + 1].contiguous())[0], whole[i]), i
    al.close()


@pytest.mark.parametrize("L,r2", [(84, 40), (96, 44)])
def test_wait_timeout_is_reported_and_recoverable(mra, L, r2):
    """The first waits give up at once; the copies and MMAs in flight are waited for with the normal bound."""
    refs, imgs = _stack(L, 9, 4, seed=530)
    al = mra.Aligner(L, 1, r2, 1, 1.0, 1.0, 1, mra.MRA_BF16_RESCORE)
    al.set_refs(refs)
    good = al.align(imgs)
    mra.mra_sync(al.h)
    os.environ["MRA_DEBUG_FIRST_WAIT_LIMIT"] = "0"
    try:
        al.align(imgs)
        with pytest.raises(mra.MRAError) as ei:
            mra.mra_sync(al.h)
        assert ei.value.code == mra.MRA_ETIMEOUT
    finally:
        del os.environ["MRA_DEBUG_FIRST_WAIT_LIMIT"]
    again = al.align(imgs)
    mra.mra_sync(al.h)
    assert torch.equal(good, again)
    al.close()
