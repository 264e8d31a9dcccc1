"""What the evaluating calls accept: limits that hold at every sample count, and workspaces."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle as O
import paper_2311_17189_gb300 as T
from paper_2311_17189_gb300 import _lib as L
from paper_2311_17189_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LAT = (1.0, -0.3, -0.5, np.pi / 2, np.pi / 3)


@pytest.fixture(autouse=True)
def generic():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    T.set_jit("never")
    yield
    T.set_jit("auto")


def sigma(order, index):
    d = O.enumerate_sigma(order)[index]
    return T.Diagram(d["alpha"], eps=d["eps"]).upload(0)


def test_table_that_only_the_small_tile_could_hold():
    """Order-6 diagram 105: at 243 frequencies its table does not fit beside the 128-sample tile (of
    232 448 bytes), beside the smaller buffers of the 32-sample tile it would.  Refused at every size;
    one frequency less runs, and its mean is that of its samples."""
    if torch.cuda.get_device_properties(0).shared_memory_per_block_optin != 232448:
        pytest.skip("stated for 232 448 bytes of shared memory per block")
    D = sigma(6, 105)
    X = torch.as_tensor(W.matsubara(5.0, 243), device="cuda")
    E = torch.as_tensor(W.random_energies(33, D.n_lines, a=4.0, seed=3), device="cuda")
    for call in [lambda n=n: D.forward(LAT, 7, 0, n, X, 5.0) for n in (33, 30000, 38912, 50000)] + [
            lambda: D.eval_energies(E, X, 5.0)]:
        with pytest.raises(L.TamiError) as e:
            call()
        assert e.value.code == L.TAMI_EUNSUPPORTED
    m, _, p = D.forward(LAT, 7, 0, 30000, X[:242], 5.0, per_sample=True)
    assert torch.all((m - p.mean(dim=1)).abs() <= 1e-13 * p.abs().mean(dim=1))
