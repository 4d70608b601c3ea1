"""bench.py's rooflines follow the kernels that ran (Operator.form): counts and names of the stored and the
factorised products at the production size, on times measured there."""
import pytest

from paper_2512_21697_gb300 import binding as B, workloads as W


@pytest.fixture(scope="module")
def production():
    from paper_2512_21697_gb300 import build
    build.build()
    return B.Basis(W.PRODUCTION)


def _roof(bas, forms, ms, precision, tol=1e-10):
    import bench
    cfg = dict(W.PRODUCTION, tol=tol)
    return bench.roofline(bas, cfg, ms, {k: 1 for k in ms}, precision, 6800.0, forms)


# 6.4e9 multiply-adds against the stored form's 8.5e9 (plus the diagonal's 0.4e9 in both)
def test_fp64_roofline_counts_the_form_that_ran(production):
    ang, _ = _roof(production, {"residual": "angular"}, {"apply": 12.1}, 0)
    rows, _ = _roof(production, {"residual": "rows"}, {"apply": 15.6}, 0)
    assert "k_ang" in ang["kernel"] and "k_apply<double>" in rows["kernel"]
    assert sum(ang["fma_per_apply"].values()) == pytest.approx(6.4e9 + 0.39e9, rel=0.02)
    assert rows["flops_per_apply"] == pytest.approx(2 * (8.5e9 + 0.39e9), rel=0.06)
    for r in (ang, rows):
        assert 0.5 < r["frac"] <= 1.0
    assert ang["bytes_per_apply"] < 0.02 * rows["bytes_per_apply"]
    split, _ = _roof(production, {"residual": "split"}, {"apply": 15.6}, 0)
    assert "k_apply_split" in split["kernel"]


def test_mixed_roofline_counts_the_form_that_ran(production):
    ms = {"apply": 2.6, "owner": 2.43, "apply32": 0.57}
    own, inner = _roof(production, {"residual": "angular", "apply32": "angular"}, ms, 2, tol=1e-12)
    assert "k_ang" in own["kernel"] and "k_ang" in inner["kernel"] and own["bound"] == inner["bound"] == "alu"
    assert own["traffic"] is None and inner["traffic"] is None
    assert own["ops_per_apply"] == 10 * own["df_fma_per_apply"]
    assert 0 < own["frac"] <= 1.0 and 0 < inner["frac"] <= 1.0
    ms = {"apply": 3.8, "owner": 3.12, "apply32": 1.06}
    own, inner = _roof(production, {"residual": "owner", "apply32": "subgroup"}, ms, 2)
    assert "k_residual_own_df" in own["kernel"] and own["bound"] == "hbm" and own["traffic"] > 17e9
    assert "k_fact_tile32" in inner["kernel"]
    _, inner = _roof(production, {"residual": "owner", "apply32": "owner"}, ms, 2)
    assert "k_apply_own32" in inner["kernel"] and inner["unit"] == "GB/s"


def test_l2_note_names_coupling_values_only_where_they_are_streamed(production):
    import bench
    cfg = W.PRODUCTION
    assert "coupling values streamed" in bench.l2_note(production, cfg, {"residual": "owner", "apply32": "subgroup"})
    assert "no coupling values stored" in bench.l2_note(production, cfg, {"residual": "angular"})
