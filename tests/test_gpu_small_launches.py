"""The kernels of small launches, at the edges of their tiles.

Forward and energy input: the tile of 32 samples (coop_tile) keeps the 128-sample tile's
operations in their order, so per-sample values, saved rows and energy-input values equal, bit for
bit, those of launches too large (or with too many frequencies) for it.
Adjoint: where lanes share a sample's frequencies, per-sample gradients stay within the oracle's
bounds and everything that one lane computes keeps its bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import paper_2311_17189_gb300 as T
from paper_2311_17189_gb300 import workloads as W

import bounds as B

pytestmark = pytest.mark.gpu

LAT = (1.0, -0.3, -0.5, np.pi / 2, np.pi / 2)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    T.set_jit("never")
    yield
    T.set_jit("auto")


def diagram(order, index=0):
    d = O.enumerate_sigma(order)[index]
    return T.Diagram(d["alpha"], eps=d["eps"]).upload(0), d


@pytest.mark.parametrize("n_f", [1, 5, 16])
@pytest.mark.parametrize("order,index", [(2, 0), (4, 2), (5, 12)])
def test_small_forward_equals_the_slice_of_a_large_one(order, index, n_f):
    D, _ = diagram(order, index)
    X = W.matsubara(5.0, n_f)
    big_n = 3 * 128 * torch.cuda.get_device_properties(0).multi_processor_count + 5
    rows = D.saved_buffer(big_n)
    _, _, big = D.forward(LAT, 11, 3, big_n, X, 5.0, per_sample=True, save=rows)
    for n in (1, 31, 32, 33, 129):
        sv = D.saved_buffer(n)
        m, v, p = D.forward(LAT, 11, 3, n, X, 5.0, per_sample=True, save=sv)
        assert torch.equal(p, big[:, :n]) and torch.equal(sv, rows[:, :n]), n
        scale = p.abs().mean(dim=1)
        assert torch.all((m - p.mean(dim=1)).abs() <= 1e-13 * scale), n


@pytest.mark.parametrize("order,index", [(3, 0), (4, 2), (4, 9), (5, 12), (5, 44)])
def test_small_forward_off_the_axis(order, index):
    """Both forms of the small tile's frequency loop (tries of fewer products than denominators, and
    larger ones) off the imaginary axis, against the 128-sample tile's bits."""
    D, _ = diagram(order, index)
    X = W.real_axis(-3.0, 3.0, 7, 0.1)
    big_n = 3 * 128 * torch.cuda.get_device_properties(0).multi_processor_count
    _, _, big = D.forward(LAT, 5, 0, big_n, X, 4.0, per_sample=True)
    for n in (1, 33, 1000):
        assert torch.equal(D.forward(LAT, 5, 0, n, X, 4.0, per_sample=True)[2], big[:, :n]), n


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1000])
def test_energy_input_equals_the_rows_of_more_frequencies(n):
    """257 frequencies are above the small tile's limit and take the 128-sample one."""
    D, d = diagram(4, 2)
    E = torch.as_tensor(W.random_energies(n, D.n_lines, a=4.0, seed=9), device="cuda")
    X = W.matsubara(2.0, 257)
    wide = D.eval_energies(E, X, 2.0)
    for n_f in (1, 3, 256):
        assert torch.equal(D.eval_energies(E, X[:n_f], 2.0), wide[:n_f]), n_f


@pytest.mark.parametrize("n_f", [8, 17, 37])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 65])
def test_lanes_sharing_a_sample(n, n_f):
    """2, 4 and 8 lanes a sample (8, 17 and 37 frequencies), ragged shares and ragged tiles."""
    D, d = diagram(3, 0)
    S = O.Solution(d["alpha"], eps=d["eps"])
    lat, beta, seed, off = (1.0, 0.0, 0.0, np.pi / 2, np.pi / 2), 10.0, 21, 5
    X = W.real_axis(-4.0, 4.0, n_f, 0.05)
    r = np.random.default_rng(3)
    g = r.normal(size=n_f) + 1j * r.normal(size=n_f)
    fb = D.forward_backward(lat, seed, off, n, X, beta, g, per_sample=True)
    _, _, p = D.forward(lat, seed, off, n, X, beta, per_sample=True)
    sv = D.saved_buffer(n)
    D.forward(lat, seed, off, n, X, beta, save=sv)
    b = D.backward(lat, seed, off, n, X, beta, g, per_sample=True, saved=sv)
    assert torch.equal(fb["values"], p) and torch.equal(fb["dX"], b["dX"]) and torch.equal(fb["grads"], b["grads"])
    ref, bound = B.oracle_deriv(S, lat, seed, off, n, X, beta, "omega")
    assert np.all(np.abs(fb["dX"].cpu().numpy() - ref) <= bound)
    assert np.all(np.abs(fb["dSigma_dX"].cpu().numpy() - ref.mean(axis=1)) <= bound.mean(axis=1))
    grads = fb["grads"].cpu().numpy()
    for k, which in enumerate(("mu", "kx", "ky")):
        der, dbd = B.oracle_deriv(S, lat, seed, off, n, X, beta, which)
        want = np.real(np.conj(g)[:, None] * der).sum(axis=0)
        assert np.all(np.abs(grads[:, k] - want) <= (np.abs(g)[:, None] * dbd).sum(axis=0)), which
    assert np.all(np.abs(fb["grad_params"].cpu().numpy() - grads.mean(axis=0)) <= 1e-13 * np.abs(grads).mean(axis=0))
    assert torch.allclose(fb["mean"], p.mean(dim=1), rtol=0, atol=float(1e-13 * p.abs().mean()))
