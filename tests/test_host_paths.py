"""The host side of the entry points, on the CPU, against a CUDA runtime that runs no kernel
(tests/_fake_cuda.py): which kernels are launched, and what becomes of a call whose launch,
tensor map or allocation fails."""
import shutil

import pytest

from tests import _fake_cuda

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _fake_cuda.load(tmp_path_factory.mktemp("fake_cuda"))


@pytest.fixture
def calls(lib):
    lib.fake_reset()
    yield _fake_cuda.Calls(lib)
    lib.fake_reset()


LAUNCHES = {
    "mttkrp": lambda c: c.mttkrp(20, 100, 300, 400),
    "split": lambda c: c.mttkrp(20, 100, 300, 400, precision=1),
    "loss": lambda c: c.loss(20, 100, 300, 400, normG2=0.0),
    "sweep": lambda c: c.sweep(20, 100, 300, 400),
    "emulated": lambda c: c.sweep(20, 100, 300, 1100, ldl=3),
    "batched": lambda c: c.batched([(12, 60, 200, 420), (3, 9, 30, 40)]),
    "exchange": lambda c: c.exchange(10, 50, 200, 300, 4),
    "core fit": lambda c: c.core_fit(10, 50, 200, 220, loss=True),
    "DF": lambda c: c.df_als(10, 50, 200, 220),
    "order 4": lambda c: c.nd_als((5, 15, 7, 9), 2, 40, 60),
    "order 3": lambda c: c.nd_mttkrp((10, 50, 30), 1, 200, 300),
    "solve": lambda c: c.solve(1100, 140),
}


# kernel attributes (the shared memory a launch may ask for) belong to one device
@pytest.mark.parametrize("what", LAUNCHES)
def test_second_device_launches_what_the_first_does(calls, what):
    counts = []
    for dev in (0, 1):
        calls.lib.fake_reset()
        calls.lib.fake_device(dev)
        assert LAUNCHES[what](calls) == 0, calls.lib.thc_cpd_last_error()
        counts.append({k: calls.lib.fake_launches(k) for k in (b"k_oz_update", b"k_oz_split", b"k_fix", b"k_tc_gemm",
                                                               b"k_ldl_flow", b"")})
    assert counts[0] == counts[1] and counts[0][b""] > 0


# every kernel of a call, its first launch and its last: the call has to report the failure
@pytest.mark.parametrize("what", LAUNCHES)
def test_failed_launch_is_reported(calls, what):
    from paper_2502_17683_gb300._lib import ERR_CUDA
    assert LAUNCHES[what](calls) == 0, calls.lib.thc_cpd_last_error()
    kernels = {n: calls.lib.fake_launches(n) for n in calls.launched()}
    for name, n in kernels.items():
        for after in {0, n - 1}:
            calls.lib.fake_reset()
            calls.lib.fake_fail_launch(name, after)
            assert LAUNCHES[what](calls) == ERR_CUDA, (name, after)


# (the solve of this size and the small order-4 run use no tensor map)
@pytest.mark.parametrize("what", [w for w in LAUNCHES if w not in ("solve", "order 4")])
def test_failed_tensor_map_is_reported(calls, what):
    from paper_2502_17683_gb300._lib import ERR_CUDA
    calls.lib.fake_fail_encode(1)
    assert LAUNCHES[what](calls) == ERR_CUDA


# a Gram of more terms than one digit launch sums (8192) beside products that run from digits
@pytest.mark.parametrize("o,v", [(5, 8192), (5, 8193), (8193, 5)])
def test_long_factors_run(calls, o, v):
    assert calls.norm2(o, v, 220) == 0, calls.lib.thc_cpd_last_error()
    assert calls.loss(o, v, 220, 40, normG2=0.0) == 0, calls.lib.thc_cpd_last_error()
    assert calls.lib.fake_launches(b"k_oz_update") > 0


# a block that does not fit is asked for with fewer points, at last without digits: one point's needs on
# the FP64 pipes are enough (five Rt x R, three R x R, the scaled factors, partial sums)
@pytest.mark.parametrize("ldl", [0, 3])
def test_exchange_makes_do_with_one_point(calls, ldl):
    from paper_2502_17683_gb300._lib import ERR_ALLOC
    o, v, Rt, R, na = 10, 50, 400, 600, 12
    run = lambda: calls.exchange(o, v, Rt, R, na, ldl=ldl)
    assert run() == 0
    sizes = [calls.lib.fake_largest_alloc()]
    while True:
        calls.lib.fake_reset()
        calls.lib.fake_alloc_limit(sizes[-1] - 1)
        s = run()
        if s != 0:
            break
        sizes.append(calls.lib.fake_largest_alloc())
    assert s == ERR_ALLOC
    # 16 split-K partial sums of the largest product at most, 256 bytes of padding a piece
    one = 8 * ((o + v) * Rt + 5 * Rt * R + (2 * o + v) * R + 3 * R * R + 16 * Rt * R) + 65536
    assert len(sizes) > 3 and sizes[-1] <= one
    calls.lib.fake_alloc_limit(1 << 62)
    assert run() == 0  # the failure leaves nothing behind


ALLOCS = {
    "mttkrp": lambda c: c.mttkrp(20, 100, 300, 400),
    "loss": lambda c: c.loss(20, 100, 300, 400, normG2=0.0),
    "norm": lambda c: c.norm2(20, 100, 300),
    "sweep": lambda c: c.sweep(20, 100, 300, 400, normG2=0.0),
    "split": lambda c: c.sweep(20, 100, 300, 400, precision=1),
    "batched": lambda c: c.batched([(12, 60, 200, 420), (3, 9, 30, 40)]),
    "core fit": lambda c: c.core_fit(10, 50, 200, 220, loss=True),
    "DF": lambda c: c.df_als(10, 50, 200, 220),
    "order 3": lambda c: c.nd_mttkrp((10, 50, 30), 1, 200, 300),
}


# a call whose digits do not fit runs on the FP64 pipes; what those need is refused as before
@pytest.mark.parametrize("what", ALLOCS)
def test_call_makes_do_without_digits(calls, what):
    from paper_2502_17683_gb300._lib import ERR_ALLOC
    assert ALLOCS[what](calls) == 0, calls.lib.thc_cpd_last_error()
    sizes = [calls.lib.fake_largest_alloc()]
    for expect in (0, ERR_ALLOC):
        calls.lib.fake_reset()
        calls.lib.fake_alloc_limit(sizes[-1] - 1)
        assert ALLOCS[what](calls) == expect, calls.lib.thc_cpd_last_error()
        sizes.append(calls.lib.fake_largest_alloc())
        assert what == "batched" or calls.lib.fake_launches(b"k_oz_update") == 0
    calls.lib.fake_alloc_limit(1 << 62)
    assert ALLOCS[what](calls) == 0, calls.lib.thc_cpd_last_error()  # the failure leaves nothing behind


# the digits of one operand take 256 MB at most, however long or many its rows, beside what the call
# takes without them
@pytest.mark.parametrize("what", [lambda c: c.core_fit(200, 1000, 100, 160), lambda c: c.df_als(60, 70, 4000, 20),
                                  lambda c: c.norm2(5, 200000, 250)], ids=["core fit", "DF", "norm"])
def test_digit_workspace_is_bounded(calls, what):
    assert what(calls) == 0 and calls.lib.fake_launches(b"k_oz_update") > 0
    full = calls.lib.fake_largest_alloc()
    calls.lib.fake_reset()
    calls.lib.fake_alloc_limit(full - 1)
    assert what(calls) == 0 and calls.lib.fake_launches(b"k_oz_update") == 0
    assert full - calls.lib.fake_largest_alloc() <= 2 * ((1 << 28) + (1 << 20))


def test_products_option_took_padding():
    from paper_2502_17683_gb300._lib import Opts
    assert Opts.products.offset == Opts.ldl.offset + 4 and Opts.wait_limit_s.offset == Opts.ldl.offset + 8


# products = 1: nothing of an FP64 call leaves the FP64 pipes, the factorisation included
PIPES = {
    "mttkrp": lambda c, **k: c.mttkrp(20, 100, 300, 400, **k),
    "norm": lambda c, **k: c.norm2(20, 100, 300, **k),
    "loss": lambda c, **k: c.loss(20, 100, 300, 400, normG2=0.0, **k),
    "sweep": lambda c, **k: c.sweep(20, 100, 300, 1100, **k),
    "batched": lambda c, **k: c.batched([(12, 60, 200, 420), (20, 100, 300, 1100)], **k),
    "exchange": lambda c, **k: c.exchange(10, 50, 200, 300, 4, **k),
    "core fit": lambda c, **k: c.core_fit(10, 50, 200, 220, loss=True, **k),
    "DF": lambda c, **k: c.df_als(10, 50, 200, 220, **k),
    "order 3": lambda c, **k: c.nd_mttkrp((10, 50, 30), 1, 200, 300, **k),
    "solve": lambda c, **k: c.solve(1100, 140, **k),
}


@pytest.mark.parametrize("what", PIPES)
@pytest.mark.parametrize("products", [0, 1])
def test_products_on_the_fp64_pipes(calls, what, products):
    assert PIPES[what](calls, products=products) == 0, calls.lib.thc_cpd_last_error()
    digits = calls.lib.fake_launches(b"k_oz_") + calls.lib.fake_launches(b"k_fix_")
    assert (digits == 0) == (products == 1)


# Every digit cut and every tensor map stays inside its block, at the sizes of the other tests and where the
# operands are long, wide or many: as many chunks as a launch sums, more rows than 256 MB of digits hold.
EXTENTS = {
    **LAUNCHES, **{"alloc " + k: f for k, f in ALLOCS.items()},
    "norm R_thc 8000": lambda c: c.norm2(3, 5, 8000),
    "norm R_thc 8192": lambda c: c.norm2(8192, 5, 8192),
    "norm R_thc 8193": lambda c: c.norm2(3, 5, 8193),
    "loss wide": lambda c: c.loss(1, 1, 8000, 700, normG2=0.0),
    "loss many columns": lambda c: c.loss(1, 1, 300, 8000, normG2=0.0),
    "mttkrp long": lambda c: c.mttkrp(4000, 8, 700, 900, mode=1),
    "mttkrp long factors": lambda c: c.mttkrp(9000, 8, 300, 200),
    "mttkrp many columns": lambda c: c.mttkrp(30, 200, 400, 8192),
    "sweep two-level": lambda c: c.sweep(50, 250, 1200, 1800, normG2=0.0),
    "sweep of 2048": lambda c: c.sweep(5, 2100, 300, 2049),
    "sweep split": lambda c: c.sweep(20, 100, 480, 720, precision=1, normG2=0.0),
    "trial points": lambda c: c.trajectory(20, 100, 480, 720),
    "trial points split": lambda c: c.trajectory(30, 150, 720, 1080, precision=1),
    "batch": lambda c: c.batched([(30, 150, 720, 1080), (20, 100, 480, 720), (5, 15, 60, 80)]),
    "exchange groups": lambda c: c.exchange(20, 60, 203, 261, 500),
    "exchange large": lambda c: c.exchange(50, 250, 1200, 1800, 12),
    "exchange wide": lambda c: c.exchange(3, 4, 5000, 2000, 5),
    "core fit long": lambda c: c.core_fit(200, 1000, 100, 160, loss=True),
    "core fit 2048": lambda c: c.core_fit(20, 100, 2048, 300, loss=True),
    "core fit emulated": lambda c: c.core_fit(40, 300, 128, 2000, ldl=3),
    "DF long": lambda c: c.df_als(60, 70, 4000, 20),
    "DF emulated": lambda c: c.df_als(30, 300, 600, 300, ldl=3),
    "order 4 large": lambda c: c.nd_als((20, 100, 20, 100), 2, 480, 720),
    "order 2 long": lambda c: c.nd_mttkrp((4096, 4096), 1, 500, 700),
    "solve 1800": lambda c: c.solve(1800, 250),
}


@pytest.mark.parametrize("what", EXTENTS)
def test_digits_and_maps_stay_inside_their_blocks(calls, what):
    assert EXTENTS[what](calls) == 0, calls.lib.thc_cpd_last_error()
    assert calls.lib.fake_outside() == 0


# only a run with trial points reserves the workspace of their products, and those run from digits
def test_trial_points_run_from_digits(calls):
    assert calls.sweep(20, 100, 480, 720, normG2=0.0) == 0
    plain, n = calls.lib.fake_largest_alloc(), calls.lib.fake_launches(b"k_oz_update")
    calls.lib.fake_reset()
    assert calls.trajectory(20, 100, 480, 720, sweeps=1) == 0
    # the start point's loss and the one of alpha = 1.5: four projections, four Grams and Z each, of which the
    # occupied Grams (1.04e7 flops) count, too
    assert calls.lib.fake_launches(b"k_oz_update") == n + 2 * 9
    assert calls.lib.fake_largest_alloc() > plain
