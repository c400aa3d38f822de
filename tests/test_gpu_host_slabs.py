"""Host transfers of grids above 128^3, which go by slabs of z-planes through several staging slots:
asynchronous and synchronous gets, gets in flight while the context works on, and sets queued behind
steps, in every precision (each has row kernels of its own)."""
import numpy as np
import pytest
import torch

from paper_1810_12707_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu

N = 256


def pinned():
    return [torch.empty(s, dtype=torch.float64, pin_memory=True).numpy() for s in ((N, N, N), (3, N, N, N), (3, N, N, N))]


@pytest.fixture(scope="module")
def states():
    return [inputs.orszag_tang(N, seed=s, mach=0.2, nu=1e-2, eta=1e-2) for s in (120, 121, 122)]


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_slabs_give_the_device_paths_values(states, precision):
    ctx = mhd.mhd_init(N, [(ic.nu, ic.eta, ic.cs) for ic in states[:2]], precision=precision)
    ic = states[0]
    mhd.mhd_set_state(ctx, 0, ic.rho, ic.u, ic.b)
    mhd.mhd_set_state(ctx, 1, *[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (ic.rho, ic.u, ic.b)])
    ref = [t.cpu().numpy() for t in mhd.mhd_get_state(ctx, 0, device=True)]
    out = pinned()
    mhd.mhd_get_state_async(ctx, 0, *out)
    assert mhd.mhd_synchronize(ctx) == mhd.MHD_OK
    for got in (out, mhd.mhd_get_state(ctx, 0), mhd.mhd_get_state(ctx, 1)):
        for g, r in zip(got, ref):
            assert np.array_equal(g, r)
    mhd.mhd_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1, 2])
def test_slab_transfers_in_order_with_queued_work(states, precision):
    """get(0) in flight behind steps while instance 1 is set and both step, then get(1) and get(0) again,
    with and without waiting between the calls."""
    def run(wait):
        ctx = mhd.mhd_init(N, [(ic.nu, ic.eta, ic.cs) for ic in states[:2]], precision=precision)
        for i in range(2):
            mhd.mhd_set_state(ctx, i, states[i].rho, states[i].u, states[i].b)
        outs = [pinned() for _ in range(3)]
        sync = (lambda: mhd.mhd_synchronize(ctx)) if wait else (lambda: None)
        mhd.mhd_step(ctx, 3)
        sync()
        mhd.mhd_get_state_async(ctx, 0, *outs[0])
        sync()
        mhd.mhd_set_state(ctx, 1, states[2].rho, states[2].u, states[2].b)
        mhd.mhd_step(ctx, 2)
        sync()
        for i, o in ((1, outs[1]), (0, outs[2])):
            mhd.mhd_get_state_async(ctx, i, *o)
            sync()
        assert mhd.mhd_synchronize(ctx) == mhd.MHD_OK
        mhd.mhd_destroy(ctx)
        return [a for o in outs for a in o]

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b)
