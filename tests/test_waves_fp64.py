"""The wave planner takes an FP64 q that fits its budget with the smallest workspace only, in a wave of its
own, and still refuses one that does not fit at all."""
import pytest

torch = pytest.importorskip("torch")


def test_fp64_q_without_room_for_the_slices():
    try:
        import paper_1003_0316_gb300 as gw
    except ImportError as e:      # library not built here
        pytest.skip(str(e))
    Ks, nbs, nw = [102400, 102400, 2000], [600, 600, 64], 4
    data = [K * nb * 16 + nw * nb * nb * 16 for K, nb in zip(Ks, nbs)]
    assert gw.polarization_workspace(Ks[:1], nbs[:1], nw, "fp64") > 2 ** 30
    waves = gw.plan_waves(Ks, nbs, nw, "fp64", data[0] + 2 ** 29)
    assert sorted(q for w in waves for q in w) == [0, 1, 2]
    assert all(len(w) == 1 for w in waves if w != [2])
    assert len(gw.plan_waves(Ks, nbs, nw, "fp64", 2 ** 34)) == 1
    with pytest.raises(gw.GWError) as e:
        gw.plan_waves(Ks, nbs, nw, "fp64", data[0])
    assert e.value.code == gw.GW_EINVAL
