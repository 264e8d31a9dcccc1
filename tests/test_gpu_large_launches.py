"""The 128-sample forward kernel with its program streamed, and its staging waits running out, in
launches above two tiles per SM (smaller ones take the 32-sample tile) and in energy input above
256 frequencies."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import paper_2311_17189_gb300 as T
from paper_2311_17189_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LAT = (1.0, -0.2, 0.1, np.pi / 2, np.pi / 3)


@pytest.fixture(autouse=True)
def modes():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    T.set_jit("never")
    yield
    T.set_table_staging("auto", 512)
    T.set_jit("auto")
    T.debug_set_wait_limit(-1)


def largest(order, code):
    d = next(x for x in O.enumerate_sigma(order) if x["code"] == tuple(code))
    return T.Diagram(d["alpha"], eps=d["eps"]).upload(0)


def large():
    return 3 * 128 * torch.cuda.get_device_properties(0).multi_processor_count + 37   # a ragged last tile


@pytest.mark.parametrize("order,code", [(4, W.ORDER4["code"]), (5, W.ORDER5["code"])])
def test_streamed_program_gives_resident_bits(order, code):
    D, n = largest(order, code), large()
    X, wide = W.matsubara(5.0, 3), W.matsubara(5.0, 257)
    E = torch.as_tensor(W.random_energies(3 * 128 + 37, D.n_lines, a=4.0, seed=3), device="cuda")

    def run():
        sv = D.saved_buffer(n)
        m, v, p = D.forward(LAT, 7, 11, n, X, 5.0, per_sample=True, save=sv)
        out = (m, v, p, sv, D.forward(LAT, 7, 11, n, X, 5.0)[0], D.eval_energies(E, wide, 5.0))
        torch.cuda.synchronize()
        return out

    resident = run()
    assert torch.isfinite(torch.view_as_real(resident[0])).all()
    for chunk in (16, 512):
        T.set_table_staging("streamed", chunk)
        for a, b in zip(run(), resident):
            assert torch.equal(a, b), chunk


def test_late_staging_gives_nan_means():
    """Every wait 'runs out' on a valid copy: NaN sums, the samples' values as they are."""
    c = W.ORDER2
    D, n = T.Diagram(c["alpha"], var_is_boson=c["var_is_boson"]).upload(0), large()
    lat, beta = W.lattice(c), c["beta"]
    X = W.matsubara(beta, 2)
    m0, v0, p0 = D.forward(lat, c["seed"], 0, n, X, beta, per_sample=True)
    for mode in ("auto", "streamed"):
        T.debug_set_wait_limit(0)
        T.set_table_staging(mode, 16)
        m, v, p = D.forward(lat, c["seed"], 0, n, X, beta, per_sample=True)
        torch.cuda.synchronize()
        assert torch.isnan(torch.view_as_real(m)).all() and torch.isnan(v).all(), mode
        assert torch.equal(p, p0), mode
        T.debug_set_wait_limit(-1)
        m, v, p = D.forward(lat, c["seed"], 0, n, X, beta, per_sample=True)
        torch.cuda.synchronize()
        assert torch.equal(m, m0) and torch.equal(v, v0) and torch.equal(p, p0), mode
