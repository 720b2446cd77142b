"""Reciprocals and square roots of the eigenvalue kernels' dependent chains (Newton's method on the hardware's
approximations), against numbers with eleven more bits: half a unit in the last place and the rounding of the correction."""
import ctypes as C

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _newton(x):
    from paper_2410_03090_b200 import build
    lib = C.CDLL(build.build(debug=True))
    recip, root = torch.empty_like(x), torch.empty_like(x)
    rc = lib.uncomp_debug_newton(C.c_void_p(x.data_ptr()), C.c_void_p(recip.data_ptr()), C.c_void_p(root.data_ptr()),
                                 C.c_int(x.numel()), C.c_int(int(x.dtype == torch.float64)),
                                 C.c_void_p(torch.cuda.current_stream().cuda_stream))
    torch.cuda.synchronize()
    assert rc == 0
    return recip.cpu().numpy(), root.cpu().numpy()


def _units_off(got, x, wide):
    """Largest error in units of the last place of the result."""
    x = x.cpu().numpy().astype(wide)
    return [float((np.abs(g.astype(wide) - ref) / np.spacing(g).astype(wide)).max())
            for g, ref in zip(got, (1 / x, np.sqrt(x)))]


@pytest.mark.parametrize("exponent", [-100, -1, 0, 1, 31, 98])
def test_every_fp32_mantissa(exponent):
    x = torch.ldexp(1.0 + torch.arange(1 << 23, device="cuda", dtype=torch.float32) * 2.0 ** -23, torch.tensor(exponent, device="cuda"))
    assert max(_units_off(_newton(x), x, np.float64)) <= 0.51


@pytest.mark.parametrize("decades", [(-1, 1), (-299, 299), (-20, 20)])
def test_fp64(decades):
    rng = np.random.default_rng(decades[1])
    x = 10.0 ** rng.uniform(*decades, 1 << 20)
    x[:64] = 2.0 ** np.arange(-32, 32)
    x[64:128] = np.nextafter(x[:64], np.inf)
    x[128:192] = np.nextafter(x[:64], 0)
    x = torch.from_numpy(x).cuda()
    assert max(_units_off(_newton(x), x, np.longdouble)) <= 0.51
