"""Which route the wide entropy takes (host rule, no GPU)."""
import ctypes as C

import pytest


@pytest.mark.parametrize("n,k,ctas,lanczos", [
    (4096, 32, 148, 1),      # the whole device
    (4096, 32, 128, 1),      # just room for its 128 CTAs
    (4096, 32, 127, 0),      # fewer SMs than CTAs that wait for one another: the full reduction, which takes any number
    (1024, 64, 32, 1),
    (1024, 64, 31, 0),
    (4096, 32, 0, 0),
    (384, 32, 148, 1),       # the smallest matrix
    (320, 32, 148, 0),
    (4096, 64, 148, 1),      # the largest k
    (4096, 65, 148, 0),
    (384, 33, 148, 0),       # too few blocks for the ten steps of k > 32
    (448, 33, 148, 1),
])
def test_lanczos_only_where_its_ctas_fit_together(n, k, ctas, lanczos):
    from paper_2410_03090_b200 import build
    lib = C.CDLL(build.build(debug=True))
    assert lib.uncomp_debug_krylov_applies(n, k, ctas) == lanczos
