"""The M = 256 kernel with the tcgen05 inverse DFT at the edges of its tiles.

The full correlation table before rescoring against the FP64 oracle, at the
tolerance the 16-bit tables have for M = 256: at most 8 unit roundoffs of the
contraction operands plus, for the inverse DFT, one BF16 rounding (2^-9) of
the spectrum and one of the DFT matrix, 4 * 2^-8 of the Cauchy-Schwarz scale
covering both.
"""
import numpy as np
import pytest
import torch

import synth
from oracle import mra_oracle as O
from test_gpu_parity import _cs_scale, _oracle_table, tc_tol

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


def _stack(L, K, n, shift, seed):
    refs, blob = synth.make_refs(K, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=seed)
    imgs, _ = synth.make_particles(blob, n, shift_range=shift, mirror=True, snr=1.0, seed=seed + 1, noise_seed=seed + 2)
    return refs.float().contiguous(), imgs.float().contiguous()


# (L, first, last ring, shift range, K, n, precision): both k-step patterns and
# their boundary (rings 1..36 / 1..37), the largest ring count, a single ring,
# reference tiles of 1, 7 and 8 + 1, rows that leave the last tile ragged, one
# row tile split over many reference ranges and more row tiles than SMs
CASES = [(76, 1, 36, 0, 1, 1, "bf16"), (84, 1, 37, 1, 7, 1, "bf16"), (84, 1, 40, 1, 9, 2, "fp16"),
         (48, 21, 21, 0, 8, 3, "bf16"), (64, 1, 28, 1, 65, 1, "bf16"), (60, 1, 24, 2, 2, 50, "fp16")]


@pytest.mark.parametrize("L,r1,r2,R,K,n,prec", CASES)
def test_table_at_the_tile_edges(mra, L, r1, r2, R, K, n, prec):
    refs, imgs = _stack(L, K, n, R, seed=300 + r2 + K)
    cfg = O.MRAConfig(L, r1, r2, 1, float(R), 1.0, 1)
    al = mra.Aligner(L, r1, r2, 1, float(R), 1.0, 1, mra.MRA_BF16_RESCORE if prec == "bf16" else mra.MRA_FP16_RESCORE)
    al.set_refs(refs.to(DEV))
    table = al.debug_cc(imgs.to(DEV)).cpu().numpy()
    al.close()
    err = np.abs(table - _oracle_table(imgs, refs, cfg)) / _cs_scale(imgs, refs, cfg)[..., None]
    assert err.max() <= tc_tol(prec, 256), float(err.max())


def test_references_copied_between_the_kernels_layouts(mra):
    """The two M = 256 kernels order the fragments differently; a copy re-derives them."""
    refs, imgs = _stack(76, 9, 6, 1, seed=400)
    refs, imgs = refs.to(DEV), imgs.to(DEV)
    handles = [mra.Aligner(76, 1, 35, 1, 1.0, 1.0, 1, mra.MRA_BF16_RESCORE, kernel=k) for k in (0, 1)]
    handles[0].set_refs(refs)
    want = handles[0].align(imgs)
    handles[1].copy_refs(handles[0])
    assert torch.equal(handles[1].align(imgs), want)
    handles[1].set_refs(refs)
    handles[0].copy_refs(handles[1])
    assert torch.equal(handles[0].align(imgs), want)
    for h in handles:
        h.close()
