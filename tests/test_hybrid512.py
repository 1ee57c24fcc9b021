"""The M = 512 kernel with the tcgen05 inverse DFT at the edges of its tiles and schedules.

The full correlation table before rescoring against the FP64 oracle, at the
tolerance the 16-bit tables have for M = 512 (8 unit roundoffs of the
contraction operands plus 4 * 2^-8 for the inverse DFT's BF16 roundings).
"""
import numpy as np
import pytest
import torch

from oracle import mra_oracle as O
from test_gpu_parity import _cs_scale, _oracle_table, tc_tol
from test_hybrid256 import DEV, _stack, mra  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

# (L, first, last ring, shift range, K, n, precision): the most rings (6 k-steps per frequency), a
# single ring (one k-step everywhere), frequencies with no ring of the shorter lengths, ragged
# reference and row tiles
CASES = [(96, 1, 81, 0, 9, 1, "bf16"), (92, 41, 41, 0, 1, 1, "fp16"), (96, 1, 44, 1, 8, 2, "fp16"),
         (88, 30, 42, 0, 17, 3, "bf16")]


@pytest.mark.parametrize("L,r1,r2,R,K,n,prec", CASES)
def test_table_at_the_tile_edges(mra, L, r1, r2, R, K, n, prec):  # noqa: F811
    refs, imgs = _stack(L, K, n, R, seed=600 + r2 + K)
    cfg = O.MRAConfig(L, r1, r2, 1, float(R), 1.0, 1)
    al = mra.Aligner(L, r1, r2, 1, float(R), 1.0, 1, mra.MRA_BF16_RESCORE if prec == "bf16" else mra.MRA_FP16_RESCORE)
    al.set_refs(refs.to(DEV))
    table = al.debug_cc(imgs.to(DEV)).cpu().numpy()
    al.close()
    err = np.abs(table - _oracle_table(imgs, refs, cfg)) / _cs_scale(imgs, refs, cfg)[..., None]
    assert err.max() <= tc_tol(prec, 512), float(err.max())
