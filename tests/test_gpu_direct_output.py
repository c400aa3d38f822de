"""mhd_get_state, mhd_rhs and mhd_rhs_noalloc into device arrays at an address that is no multiple of 8
and into page-locked host memory passed as a device pointer: the bytes of an ordinary device output."""
import ctypes

import pytest
import torch

from paper_1810_12707_gb300 import inputs, mhd

pytestmark = pytest.mark.gpu


def places(count, kind):
    """(address, read) of room for `count` doubles."""
    if kind == "odd":
        raw = torch.zeros(8 * count + 16, dtype=torch.uint8, device="cuda")
        return raw.data_ptr() + 4, lambda: raw[4:4 + 8 * count].clone().view(torch.float64).cpu()
    raw = torch.zeros(count, dtype=torch.float64).pin_memory()
    return raw.data_ptr(), lambda: raw.clone()


@pytest.mark.parametrize("kind", ["odd", "page-locked"])
@pytest.mark.parametrize("n,precision", [(16, 0), (32, 0), (32, 1), (32, 2), (256, 0)])
def test_outputs_that_take_a_copy(n, precision, kind):
    ic = inputs.orszag_tang(n, seed=3, mach=0.3, nu=1e-2, eta=1e-2)
    phys = (ic.nu, ic.eta, ic.cs)
    ctx = mhd.mhd_init(n, [phys], precision=precision)
    mhd.mhd_set_state(ctx, 0, ic.rho, ic.u, ic.b)
    lib = mhd.load_library()
    counts = [n ** 3, 3 * n ** 3, 3 * n ** 3]
    for call, ref in ((lib.mhd_get_state, mhd.mhd_get_state(ctx, 0, device=True)),
                      (lib.mhd_rhs, mhd.mhd_rhs(ctx, 0, device=True))):
        for odd in (range(3) if n == 32 else (0,)):  # one such output among ordinary ones, too
            out = [places(c, kind if i == odd or n != 32 else "page-locked") for i, c in enumerate(counts)]
            assert call(ctx.handle, 0, *[p for p, _ in out], 1) == mhd.MHD_OK
            for (_, read), r in zip(out, ref):
                assert torch.equal(read(), r.cpu().reshape(-1))
    mhd.mhd_destroy(ctx)
    if n <= 32 and precision == 0:
        dev = [torch.from_numpy(a).cuda().contiguous() for a in (ic.rho, ic.u, ic.b)]
        ref = mhd.mhd_rhs_noalloc(n, phys, *dev)
        out = [places(c, kind) for c in counts]
        ph = mhd.MhdPhys(*phys)
        assert lib.mhd_rhs_noalloc(n, ctypes.byref(ph), *[t.data_ptr() for t in dev], *[p for p, _ in out],
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == mhd.MHD_OK
        torch.cuda.synchronize()
        for (_, read), r in zip(out, ref):
            assert torch.equal(read(), r.cpu().reshape(-1))


def test_rhs_noalloc_in_a_captured_graph():
    n = 32
    ic = inputs.orszag_tang(n, seed=4, mach=0.3, nu=1e-2, eta=1e-2)
    ph = mhd.MhdPhys(ic.nu, ic.eta, ic.cs)
    lib = mhd.load_library()
    dev = [torch.from_numpy(a).cuda().contiguous() for a in (ic.rho, ic.u, ic.b)]
    ref = mhd.mhd_rhs_noalloc(n, (ic.nu, ic.eta, ic.cs), *dev)
    out = [torch.zeros_like(t) for t in dev]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        assert lib.mhd_rhs_noalloc(n, ctypes.byref(ph), *[t.data_ptr() for t in dev], *[o.data_ptr() for o in out],
                                   ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)) == mhd.MHD_OK
    assert all(not o.any() for o in out)
    graph.replay()
    torch.cuda.synchronize()
    for o, r in zip(out, ref):
        assert torch.equal(o, r)
