"""The autotuner's candidates include the library's own choice of the knobs."""
from paper_2404_16517_gb300 import autotune


def test_the_librarys_defaults_are_a_candidate():
    c = autotune.candidates()
    assert c[0] == {k: 0 for k in autotune.DEFAULT_GRID}
    # what the size rules choose is in the grid's reach, each by itself
    assert {256, 2048} <= {x["cta_cap"] for x in c} and {4352, 8192} <= {x["direct_cap"] for x in c}
    assert any(x["cta_cap"] == 0 and x["direct_cap"] == 8192 for x in c)


def test_zero_is_valid_beside_any_value():
    got = autotune.candidates({"cta_cap": [0, 512, 2048], "direct_cap": [0, 1024]})
    pairs = sorted((x["cta_cap"], x["direct_cap"]) for x in got)
    assert pairs == [(0, 0), (0, 1024), (512, 0), (512, 1024), (2048, 0)]
    assert autotune.candidates({"direct_cap": [0, 1024]}) == [{"direct_cap": 0}, {"direct_cap": 1024}]


def test_defaults_leave_the_params_as_they_are():
    import paper_2404_16517_gb300 as sss
    from paper_2404_16517_gb300 import _build
    _build.build()
    base, prm = sss.params(), autotune._with(None, autotune.DEFAULTS)
    assert all(getattr(base, f) == getattr(prm, f) for f in autotune.DEFAULTS)
