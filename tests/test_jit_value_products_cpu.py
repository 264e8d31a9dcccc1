"""The generated kernels form a sample's value from the same statements in every Monte Carlo kind, with
the same products flushing values below 2^-1022, so that the fused pass's per-sample outputs equal the
separate calls' there too; tables above 256 pole-DAG ops and the energy input flush none."""
import re

import pytest

import paper_2311_17189_gb300 as T
from paper_2311_17189_gb300 import workloads as W

VALUE = re.compile(r"exp_neg<|t2 =|rD =|pv\d+ =|RR_\d+ |W1_\d+ |W2_\d+ (?:=|\+=) W1")


def tables():
    out = [("order2_bosonic", T.Diagram(W.ORDER2["alpha"], var_is_boson=W.ORDER2["var_is_boson"])),
           ("quadruple_pole", T.Diagram([[1, 0], [1, 0], [1, 0], [1, 0], [1, 1]],
                                        eps=[[1, 0, 0, 0, 0]] * 4 + [[0, 0, 0, 0, 1]], var_is_boson=[0, 1]))]
    for m in (2, 3, 4, 5):
        for i, d in list(enumerate(T.enumerate_sigma(m)))[::1 if m < 5 else 7]:
            out.append((f"order{m}_{i}", T.Diagram(d["alpha"], eps=d["eps"])))
    return out


def value_statements(src):
    body = src[src.index("tami_seg_"):src.index("if (xr_zero) {")]
    return [l.strip() for l in body.splitlines() if VALUE.search(l)]


@pytest.mark.parametrize("name,D", tables(), ids=[t[0] for t in tables()])
def test_kinds_share_their_value_products(name, D):
    fused, forward, adjoint, energy = (value_statements(D.jit_source(k)) for k in ("fused", "forward", "adjoint", "energy"))
    assert fused == forward == adjoint and len(fused) > 4
    assert not any("imul_ftz" in l for l in energy)
    if D.info()["n_dag_ops"] > 256:
        assert not any("imul_ftz" in l for l in fused)
        # and a weight's product is never contracted into the sum it enters
        if any(" * RR_" in l for l in fused):
            assert "struct Factor" in D.jit_source("fused") and "Factor RR_" in D.jit_source("forward")
