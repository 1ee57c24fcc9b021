"""mra_run_graph after other calls on the handle have replaced its own buffers.

A captured pass holds the addresses of the handle's references and workspaces.
Calls with another number of references or a longer stack reallocate them; the
next graph call has to run eagerly and be captured anew, with the same results.
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


L, K, N = 48, 11, 150


def _other_refs(al, refs, imgs):      # 8 padded references instead of 16
    al.set_refs(refs[:3])


def _more_refs(al, refs, imgs):       # 32 padded references, more row maxima
    al.set_refs(torch.cat([refs, refs, refs])[:30].contiguous())
    al.align(imgs)


def _longer_stack(al, refs, imgs):    # a larger averaging workspace
    many = torch.cat([imgs] * 9)
    al.average(many, al.align(many))


def _copied_refs(al, refs, imgs):
    import paper_2011_05755_gb300 as m
    other = m.Aligner(L, 1, 22, 1, 1.0, 1.0, 1, al.precision_used)
    other.set_refs(refs[:2])
    al.copy_refs(other)
    other.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("change", [_other_refs, _more_refs, _longer_stack, _copied_refs])
def test_graph_after_the_handles_buffers_moved(mra, change, precision):
    refs64, blob = synth.make_refs(K, L, blobs=8, sigma=(2.5, 5.0), disc=12.0, seed=81)
    imgs64, _ = synth.make_particles(blob, N, shift_range=1, mirror=True, snr=0.5, seed=82, noise_seed=83)
    refs, imgs = refs64.float().contiguous().to(DEV), imgs64.float().contiguous().to(DEV)
    al = mra.Aligner(L, 1, 22, 1, 1.0, 1.0, 1, precision)
    al.set_refs(refs)
    want_p = al.align(imgs)
    want_a, want_c = al.average(imgs, want_p)
    torch.cuda.synchronize()
    al.close()

    g = mra.Aligner(L, 1, 22, 1, 1.0, 1.0, 1, precision)
    g.precision_used = precision
    poses = torch.zeros((N, 8), dtype=torch.int32, device=DEV)
    avg = torch.zeros((K, L, L), device=DEV)
    cnt = torch.zeros((K,), dtype=torch.int32, device=DEV)

    def call(captured):
        poses.zero_()
        avg.zero_()
        mra.mra_run_graph(g.h, refs, imgs, poses, avg, cnt)
        torch.cuda.synchronize()
        assert bool(mra.mra_graph_info(g.h)) == captured
        assert torch.equal(poses, want_p) and torch.equal(cnt, want_c) and torch.equal(avg, want_a)
        assert g.info["K"] == K

    call(False)
    change(g, refs, imgs)     # between the eager pass and the capture
    call(False)
    call(True)
    change(g, refs, imgs)     # with a graph in hand
    torch.cuda.synchronize()
    if change is _longer_stack:  # already that large: the graph stays
        call(True)
    else:
        assert not mra.mra_graph_info(g.h)
        call(False)
        call(True)
    call(True)
    g.set_refs(refs[:9])      # the same padded count: the graph stays, and sets its own K
    assert mra.mra_graph_info(g.h)
    call(True)
    g.close()


def test_a_longer_stack_drops_the_graph(mra):
    refs64, blob = synth.make_refs(K, L, blobs=8, sigma=(2.5, 5.0), disc=12.0, seed=84)
    imgs64, _ = synth.make_particles(blob, N, shift_range=1, mirror=True, snr=0.5, seed=85, noise_seed=86)
    refs, imgs = refs64.float().contiguous().to(DEV), imgs64.float().contiguous().to(DEV)
    g = mra.Aligner(L, 1, 22, 1, 1.0, 1.0, 1, mra.MRA_BF16_RESCORE)
    poses = torch.zeros((N, 8), dtype=torch.int32, device=DEV)
    avg = torch.zeros((K, L, L), device=DEV)
    cnt = torch.zeros((K,), dtype=torch.int32, device=DEV)
    got = []
    for i in range(4):
        if i == 2:
            g.set_refs(refs)
            _longer_stack(g, refs, imgs)
            assert not mra.mra_graph_info(g.h)
        mra.mra_run_graph(g.h, refs, imgs, poses, avg, cnt)
        torch.cuda.synchronize()
        got.append((poses.clone(), avg.clone(), cnt.clone()))
        assert bool(mra.mra_graph_info(g.h)) == (i in (1, 3))
    for p, a, c in got[1:]:
        assert torch.equal(p, got[0][0]) and torch.equal(a, got[0][1]) and torch.equal(c, got[0][2])
    g.close()
