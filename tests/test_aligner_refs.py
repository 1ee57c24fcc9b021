"""Aligner's buffers follow the references of its handle, whichever call set them."""
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


@pytest.mark.parametrize("call", ["graph", "host"])
def test_average_after_a_pass_on_the_handle(mra, call):
    L, K, n = 32, 11, 40
    refs, blob = synth.make_refs(K, L, blobs=8, sigma=(2.0, 4.0), disc=8.0, seed=91)
    imgs, _ = synth.make_particles(blob, n, shift_range=1, mirror=True, snr=1.0, seed=92, noise_seed=93)
    dev = "cpu" if call == "host" else DEV
    refs, imgs = refs.float().contiguous(), imgs.float().contiguous()
    al = mra.Aligner(L, 1, 12, 1, 1.0, 1.0, 1)
    al.set_refs(refs[:9].contiguous().to(DEV))
    assert al.K == 9
    poses = torch.zeros((n, 8), dtype=torch.int32, device=dev)
    avg = torch.zeros((K, L, L), device=dev)
    cnt = torch.zeros((K,), dtype=torch.int32, device=dev)
    (mra.mra_run_graph if call == "graph" else mra.mra_run_host)(al.h, refs.to(dev), imgs.to(dev), poses, avg, cnt)
    assert al.K == K  # before any buffer is sized by it
    got_a, got_c = al.average(imgs.to(DEV), poses.to(DEV))
    torch.cuda.synchronize()
    assert torch.equal(got_a.cpu(), avg.cpu()) and torch.equal(got_c.cpu(), cnt.cpu())
    assert al.debug_cc(imgs[:2].to(DEV)).shape[1] == K
    al.close()
