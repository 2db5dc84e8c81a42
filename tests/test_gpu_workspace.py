"""Workspaces smaller than hf_workspace_size: a window-form lattice takes the band buffers it is
given, in more launches, with the same results; below the smallest accepted size nothing is set up."""
import numpy as np
import pytest

from paper_1006_2716_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

GIB = 1 << 30
# radius-30 disc: 500 frequencies take 2.5 GiB of band buffers in one launch, three launches of 1 GiB
CFG = dict(wl.CONFIGS["square6"], geometry=1, Lx=30, Ly=30, V0=0.02, chains_per_site=1, n_matsubara=500,
           bin_size=1, max_bins=1)


def test_smaller_workspaces_take_more_launches_and_give_the_same():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1006_2716_gb300 import build as B

    B.build()
    from paper_1006_2716_gb300 import hf

    p = hf.make_params(CFG)
    p.cuda_stream = torch.cuda.current_stream().cuda_stream
    full = hf.hf_workspace_size(p)
    N, _, band, spins = hf.hf_lattice_info(p)[:4]
    per = N * (band + 1) * 16
    nq = spins * CFG["n_matsubara"]
    assert nq * per > 2.2 * GIB
    buf = torch.zeros(full + 512, dtype=torch.uint8, device="cuda")
    base = (buf.data_ptr() + 255) & ~255
    rest = full - nq * per                      # all but the band buffers (to alignment)
    ref = None
    # all; one matrix fewer: two launches of half the matrices; 1 GiB: the smallest accepted
    for matrices, launches in ((nq, 1), (nq - 1, 2), (GIB // per, -(-nq // (GIB // per)))):
        h = hf.hf_init(p, base, rest + matrices * per)
        assert hf.hf_get_lattice_plan(h)[1] == launches
        hf.hf_compute_baths(h)
        sites, _, L, _ = hf.hf_get_sizes(h)
        out = hf.hf_get_gloc(h, sites, CFG["n_matsubara"]), hf.hf_get_g0(h, sites, L)
        hf.hf_free(h)
        if ref is None:
            ref = out
        assert all(np.array_equal(a, b) for a, b in zip(ref, out))
    least = -(-nq // -(-nq // (GIB // per)))    # matrices of an even split at 1 GiB
    with pytest.raises(hf.HFError) as e:
        hf.hf_init(p, base, rest + (least - 1) * per)
    assert e.value.status == hf.HF_ENOMEM
