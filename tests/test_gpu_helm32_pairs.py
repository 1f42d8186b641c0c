"""The Helmholtz solves by FP32 transforms carry two fields in one complex one: what is not finite in one
must stay there."""

import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def built(cuda_ok):
    from paper_2606_15035_gb300 import build
    build.build()


@pytest.mark.parametrize("n", [(32, 32, 32), (12, 10, 14)])
@pytest.mark.parametrize("name,index", [("phi", 0), ("A", 1)])
def test_static_update_keeps_a_nan_in_its_field(built, n, name, index):
    """phi and A_x, and A_y and A_z, travel in pairs through the transforms: a NaN in one must not reach
    the other, whose values are those of the call without it, to rounding."""
    import torch
    from paper_2606_15035_gb300 import _lib
    N = int(np.prod(n))
    gen = torch.Generator(device="cuda").manual_seed(3)
    ins = {k: torch.randn(c * N, generator=gen, device="cuda", dtype=torch.float64)
           for k, c in (("phi", 1), ("psi", 1), ("A", 3), ("U", 3), ("rho", 1), ("J", 3))}
    stream = torch.cuda.current_stream().cuda_stream

    def update():
        outs = [torch.empty(c * N, device="cuda", dtype=torch.float64) for c in (1, 1, 3, 3)]
        assert _lib.lib().pic_cn_update_static((C.c_int32 * 3)(*n), (C.c_double * 3)(1.3, 1.1, 0.9), 0.1, 1.0, 1.0, 1.0,
                                               1e-17, *[ins[k].data_ptr() for k in ("phi", "psi", "A", "U", "rho", "J")],
                                               *[o.data_ptr() for o in outs], C.c_void_p(stream)) == 0
        torch.cuda.synchronize()
        phi, psi, A, U = (o.cpu().numpy() for o in outs)
        return [phi, *A.reshape(3, N)], [psi, *U.reshape(3, N)]

    F, W = update()
    field = 0 if name == "phi" else 1 + index
    ins[name][index * N + 5] = float("nan")
    Fn, Wn = update()
    for f in range(4):
        if f == field:
            assert np.isnan(Fn[f]).any() and np.isnan(Wn[f]).any()
        else:
            assert np.abs(Fn[f] - F[f]).max() <= 1e-14 * np.abs(F[f]).max(), f
            assert np.abs(Wn[f] - W[f]).max() <= 1e-13 * np.abs(W[f]).max(), f
