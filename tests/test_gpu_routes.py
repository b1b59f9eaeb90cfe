"""Calls on either side of the lines between the FP64 pipes and the digit products, against torch in
FP64 on the same device. Bounds: both sides sum K terms (a relative error of K 2^-53 each on the
absolute values) in every product of the chain."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
U = 2.0 ** -53


@pytest.fixture(scope="module")
def api():
    import __graft_entry__ as g
    g.build()
    from paper_2502_17683_gb300 import api as a
    return a


def _rnd(seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)


# a Gram of 8192 terms is the longest that one digit launch sums
@pytest.mark.parametrize("o,v", [(5, 8192), (5, 8193), (8200, 7)])
def test_norm_of_long_factors(api, o, v):
    rnd, Rt = _rnd(o + v), 220
    Xo, Xv, Z = rnd(o, Rt), rnd(v, Rt), rnd(Rt, Rt)

    def norm2(Xo, Xv, Z):
        S = (Xo.T @ Xo) * (Xv.T @ Xv)
        return float((Z * (S @ Z @ S)).sum())

    lim = 2 * U * (2 * (o + v) + 2 * Rt + Rt * Rt) * norm2(Xo.abs(), Xv.abs(), Z.abs())
    assert abs(api.thc_cpd_thc_norm2(Xo, Xv, Z) - norm2(Xo, Xv, Z)) <= lim
