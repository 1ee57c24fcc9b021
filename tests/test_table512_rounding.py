"""Where the M = 512 table of the 16-bit paths is rounded.

The eight rows of an image that are rescored in FP32 are those with the
largest maxima in this table, so its roundings decide, now and then, which of
two close poses an image gets: 23 of 924,000 images got another pose from a
table that is rounded elsewhere.  They are pinned here by an emulation in 64
bits: q and p of the particle bins and v and u of the weighted reference bins
in the operand type, the spectrum Z of a pair in BF16, and both halves of its
inverse DFT (even and odd f) as two stages of 16-point DFTs, matrices and the
twiddled intermediate in BF16.

Tolerance: the kernel's FP32 spectra and sums differ from the emulation's by
some 2^-20 of a value, which takes a BF16 rounding (spacing 2^-8 or 2^-7 of it)
to its other neighbour in fewer than one case in 1,000.  A rounding that flips
is wrong by up to a spacing, where a rounding error is uniform over one (its
square a twelfth on average), so the flips make up at most 12 / 1000 of the
squared error: a tenth of it in the root mean square, for which 1/4 is
allowed.  A table with roundings of its own is off by the root mean square of
both errors, more than 1.
"""
import math

import numpy as np
import pytest
import torch

import synth
from oracle import mra_oracle as O

DEV = "cuda:0"
CASES = [(96, 1, 44, 3, 2), (128, 1, 60, 3, 2)]  # L, first and last ring, K, n


def _round(x, prec):
    t = torch.from_numpy(np.ascontiguousarray(x)).float()
    return t.to(torch.bfloat16 if prec == "bf16" else torch.float16).double().numpy()


def _stack(L, K, n):
    refs, blob = synth.make_refs(K, L, blobs=8, sigma=(L / 20, L / 10), disc=L / 4, seed=900 + L)
    imgs, _ = synth.make_particles(blob, n, shift_range=0, mirror=True, snr=0.5, seed=901 + L, noise_seed=902 + L)
    return refs.float().contiguous(), imgs.float().contiguous()


def _spectrum(imgs, refs, cfg, prec):
    """Z(f) of every (image, reference) pair, [n, K, 512]; prec None: operands not rounded."""
    rings = O.ring_table(cfg.first_ring, cfg.last_ring, cfg.ring_step)
    M = O.angle_count(rings)
    rnd = (lambda x: x) if prec is None else (lambda x: _round(x, prec))
    d = [np.zeros((len(imgs), len(refs), M // 2 + 1)) for _ in range(4)]
    X = [O.ring_dft(np.stack(s))[:, -(len(s[0]) // 2 + 1):] for s in
         zip(*(O.polar_samples(im.double().numpy(), rings) for im in imgs))]
    Y = [O.ring_dft(np.stack(s))[:, -(len(s[0]) // 2 + 1):] for s in
         zip(*(O.polar_samples(r.double().numpy(), rings) for r in refs))]
    for (r, N), x, y in zip(rings, X, Y):
        w = np.full(N // 2 + 1, 2 * math.pi * r * cfg.ring_step / N ** 2)
        if N < M:
            w[-1] *= 0.5
        y = y * w
        q, p, v, u = rnd(x.real - x.imag), rnd(x.real + x.imag), rnd(y.real - y.imag), rnd(y.real + y.imag)
        for i, (a, b) in enumerate(((q, v), (q, u), (p, v), (p, u))):
            d[i][..., :N // 2 + 1] += a[:, None] * b[None]
    Z = np.zeros((len(imgs), len(refs), M), dtype=np.complex128)
    Z[..., :M // 2 + 1] = d[0] + 1j * d[1]
    Z[..., M // 2 + 1:] = (d[3] + 1j * d[2])[..., M // 2 - 1:0:-1]
    return Z


def _bf16(z):
    return _round(z.real, "bf16") + 1j * _round(z.imag, "bf16")


def _idft256(z):
    """sum_m z(m) exp(2 pi i m n / 256), [..., 256], rounded like idft256_core."""
    k = np.arange(16)
    W = _bf16(np.exp(2j * math.pi * np.outer(k, k) / 16))
    a = z.reshape(z.shape[:-1] + (16, 16))                           # [a, t]: m = t + 16 a
    y = np.einsum("ka,...at->...kt", W, a) * np.exp(2j * math.pi * np.outer(k, k) / 256)
    c = np.einsum("...kt,tj->...kj", _bf16(y), W)                    # angle k + 16 j
    return np.swapaxes(c, -1, -2).reshape(z.shape)


def _table(c):
    """[n, K, 2, 512] of c(j): its real part, and its imaginary part half a turn on."""
    return np.stack([c.real, np.roll(c.imag, 256, axis=-1)], axis=2)


def _rounded_table(Z):
    Z = _bf16(Z)
    e, o = _idft256(Z[..., 0::2]), _idft256(Z[..., 1::2]) * np.exp(2j * math.pi * np.arange(256) / 512)
    return _table(np.concatenate([e + o, e - o], axis=-1))


@pytest.mark.parametrize("L,r1,r2,K,n", CASES[:1])
def test_the_emulation_without_rounding_is_the_oracle_table(L, r1, r2, K, n):
    refs, imgs = _stack(L, K, n)
    cfg = O.MRAConfig(L, r1, r2, 1, 0.0, 1.0, 1)
    spec = O.reference_spectra(refs.double().numpy(), cfg)
    want = np.stack([O.cc_table(im.double().numpy(), spec, cfg)[:, 0] for im in imgs])
    Z = _spectrum(imgs, refs, cfg, None)
    got = _table(np.fft.ifft(Z, axis=-1) * 512)
    assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max()
    # and with its roundings it is near it
    assert 1e-5 < np.abs(_rounded_table(Z) - want).max() / np.abs(want).max() < 2e-2


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["bf16", "fp16"])
@pytest.mark.parametrize("L,r1,r2,K,n", CASES)
def test_table_rounds_where_it_did(L, r1, r2, K, n, prec):
    import __graft_entry__ as entry
    entry.build()
    import paper_2011_05755_gb300 as mra
    refs, imgs = _stack(L, K, n)
    cfg = O.MRAConfig(L, r1, r2, 1, 0.0, 1.0, 1)
    al = mra.Aligner(L, r1, r2, 1, 0.0, 1.0, 1, mra.MRA_BF16_RESCORE if prec == "bf16" else mra.MRA_FP16_RESCORE)
    al.set_refs(refs.to(DEV))
    got = al.debug_cc(imgs.to(DEV)).cpu().double().numpy()[:, :, 0]
    al.close()
    Z = _spectrum(imgs, refs, cfg, prec)
    want, exact = _rounded_table(Z), _table(np.fft.ifft(Z, axis=-1) * 512)
    off, error = np.sqrt(np.mean((got - want) ** 2)), np.sqrt(np.mean((want - exact) ** 2))
    print(f"off {off:.3g}, rounding error {error:.3g}")
    assert off <= error / 4
