"""What atkm_plan_tuning reports of the binary64 passes: the shared-memory engine
with compile-time radices and the generic one are told apart, only lengths that
the former is built for report it, and the DF32 form, which runs the same passes,
has the binary64 entries."""
import pytest

pytestmark = pytest.mark.gpu
COMPILED = {18, 20, 24, 30, 36, 40, 48, 60, 72, 80, 90, 96, 100, 108, 120, 144, 150, 160, 180, 192, 200, 216, 240, 288, 320, 384}


@pytest.mark.parametrize("N", [(144, 144, 36), (96, 90, 20), (54, 50, 12)])
@pytest.mark.parametrize("generic", [False, True])
def test_reported_engines(lib, N, generic):
    plan = lib.Plan(N, (8.0, 7.0, 2.0), (0.0, 0.0, 1.0), f32=True, df32=True, generic_fft=generic, autotune=True)
    tun = {(t["precision"], t["length"], t["line_major"]): t for t in plan.tuning()}
    for (r, L, lm), t in tun.items():
        if r == 1:
            assert t["compiled"] == 0
            continue
        assert t["engine"] == 2
        if t["compiled"]:
            assert L in COMPILED and not generic and t["tile_shift"] == 0
        same = tun[(2 - r, L, lm)]
        assert all(t[k] == same[k] for k in ("engine", "compiled", "tile_shift", "ms_default", "ms_best"))
    if N[0] == 144 and not generic:  # the generic engine takes half as long again on these passes
        assert all(tun[(0, L, lm)]["compiled"] for L, lm in ((144, 1), (288, 0), (144, 0)))
    plan.close()
