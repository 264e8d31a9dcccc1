"""What the evaluating calls accept: limits that hold at every sample count, and workspaces."""
import ctypes

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


def test_many_denominators_at_many_frequencies():
    """7 lines nu and 8 lines nu + X, 56 complex denominators: at 243 frequencies the constants of the
    specialised forward leave less than 8 KB, and the generic kernels cannot stage the table.  The
    call runs in every mode that compiles, as with fewer frequencies.  (Lines of one momentum have one
    energy, so every denominator of the two groups vanishes and the values are NaN.)"""
    if torch.cuda.get_device_properties(0).shared_memory_per_block_optin != 232448:
        pytest.skip("stated for 232 448 bytes of shared memory per block")
    D = T.Diagram([[1, 0]] * 7 + [[1, 1]] * 8).upload(0)
    assert D.info()["n_cplx_dens"] == 56
    X = torch.as_tensor(W.matsubara(5.0, 243), device="cuda")
    T.set_jit("always")
    few = D.forward(LAT, 7, 0, 1000, X[:100], 5.0, per_sample=True)[2]
    for mode in ("always", "auto"):
        T.set_jit(mode)
        m, _, p = D.forward(LAT, 7, 0, 1000, X, 5.0, per_sample=True)
        assert torch.equal(torch.view_as_real(p[:100]).isnan(), torch.view_as_real(few).isnan())
        assert torch.equal(torch.view_as_real(m).isnan(), torch.view_as_real(p.mean(dim=1)).isnan())


# ------------------------------------------------------------------------------- workspaces
def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def queried(D, call, n, n_f):
    b = ctypes.c_size_t()
    L.check(getattr(L.lib(), f"tami_{call}_workspace")(D._h, n, n_f, ctypes.byref(b)))
    return b.value


def run(D, call, n, X, nbytes):
    """The call in a workspace of nbytes; its reduced outputs."""
    n_f, lib = len(X), L.lib()
    ws = torch.empty((nbytes + 255) // 256 * 256, dtype=torch.uint8, device="cuda")
    Xp = torch.view_as_real(X).contiguous()
    g = torch.view_as_real(torch.full((n_f,), 0.5 + 0.25j, dtype=torch.complex128, device="cuda")).contiguous()
    out = [torch.zeros((n_f, 2), dtype=torch.float64, device="cuda") for _ in range(3)] + [
        torch.zeros(n_f, dtype=torch.float64, device="cuda"), torch.zeros(3, dtype=torch.float64, device="cuda")]
    mean, var, dX, gX, gp = out
    lat, st = L.Lattice(*LAT), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    head = (D._h, ctypes.byref(lat), 7, 11, n, ptr(Xp), n_f, 5.0)
    if call == "forward":
        L.check(lib.tami_forward(*head, ptr(mean), ptr(var), None, None, ptr(ws), nbytes, st))
    elif call == "backward":
        L.check(lib.tami_backward(*head, ptr(g), ptr(dX), ptr(gX), ptr(gp), None, None, None, ptr(ws), nbytes, st))
    else:
        L.check(lib.tami_forward_backward(*head, ptr(g), ptr(mean), ptr(var), None, ptr(dX), ptr(gX), ptr(gp), None, None,
                                          ptr(ws), nbytes, st))
    torch.cuda.synchronize()
    return out


CALLS = ["forward", "backward", "forward_backward"]


@pytest.mark.parametrize("n_f", [5, 16, 64])
@pytest.mark.parametrize("call", CALLS)
def test_workspace_for_more_samples_serves_fewer(call, n_f):
    """Around the sample counts where the small tile and the lanes that share a sample come in."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    X = torch.as_tensor(W.matsubara(5.0, n_f), device="cuda")
    edges = [128 * sms, 256 * sms, 96 * sms, 192 * sms, 384 * sms]
    ns = sorted({1, 33, 4000} | {e + d for e in edges for d in (-1, 0, 1)} | {100000})
    for D in (sigma(2, 0), sigma(4, 2)):
        sizes = [queried(D, call, n, n_f) for n in ns]
        assert sizes == sorted(sizes)
        for e in edges:
            for a, b in zip(run(D, call, e, X, queried(D, call, e, n_f)), run(D, call, e, X, queried(D, call, e + 1, n_f))):
                assert torch.equal(a, b)          # the same grid, so the same sums


@pytest.mark.parametrize("call", CALLS)
def test_workspace_of_one_row_per_128_samples(call):
    """The rows that one block per 128 samples fills are enough (a workspace queried for more
    frequencies holds no more): only the sums' grouping changes.  One row less is refused."""
    n, n_f = 5000, 16
    X = torch.as_tensor(W.matsubara(5.0, n_f), device="cuda")
    D = sigma(4, 2)
    row = 8 * {"forward": 4 * n_f, "backward": 2 * n_f + 3, "forward_backward": 6 * n_f + 3}[call]
    least = 256 + row * -(-n // 128)
    assert queried(D, call, n, n_f) > least
    for a, b in zip(run(D, call, n, X, least), run(D, call, n, X, queried(D, call, n, n_f))):
        assert torch.all((a - b).abs() <= 1e-12 * b.abs().max())
    with pytest.raises(L.TamiError) as e:
        run(D, call, n, X, least - 1)
    assert e.value.code == L.TAMI_EINVAL


# ------------------------------------------------------------------------------- where the tiles change
@pytest.mark.parametrize("n_f", [8, 64])
@pytest.mark.parametrize("order,index", [(2, 0), (3, 0), (4, 2)])
def test_samples_around_the_small_tiles_line(order, index, n_f):
    """Either side of one and two 128-sample tiles per SM, where the choice of the tile changes with the
    table and n_f: the same per-sample bits, and the mean of the samples."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    D = sigma(order, index)
    X = torch.as_tensor(W.matsubara(5.0, n_f), device="cuda")
    big = D.forward(LAT, 3, 9, 3 * 128 * sms + 5, X, 5.0, per_sample=True)[2]
    for n in (32 * sms, 128 * sms, 128 * sms + 1, 192 * sms, 256 * sms, 256 * sms + 1):
        m, _, p = D.forward(LAT, 3, 9, n, X, 5.0, per_sample=True)
        assert torch.equal(p, big[:, :n]), n
        assert torch.all((m - p.mean(dim=1)).abs() <= 1e-13 * p.abs().mean(dim=1)), n


@pytest.mark.parametrize("order,index", [(2, 0), (5, 12)])
def test_rows_around_the_small_tiles_line(order, index):
    """Energy input: either side of the rows at which the tile changes, for a small and a large pole DAG,
    with few and many frequencies: the same bits as 257 frequencies, which only the large tile takes."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    D = sigma(order, index)
    assert (D.info()["n_dag_ops"] > 256) == (order == 5)
    X = torch.as_tensor(W.matsubara(2.0, 257), device="cuda")
    E = torch.as_tensor(W.random_energies(18 * 128 * sms + 1, D.n_lines, a=4.0, seed=9), device="cuda")
    for rows in (256 * sms, 256 * sms + 1, 768 * sms, 768 * sms + 1, 18 * 128 * sms, 18 * 128 * sms + 1):
        e = E[:rows].contiguous()
        few = D.eval_energies(e, X[:1], 2.0)
        for n_f in (15, 16, 65):
            assert torch.equal(D.eval_energies(e, X[:n_f], 2.0)[:1], few), (rows, n_f)
        tail = e[-33:].contiguous()
        assert torch.equal(D.eval_energies(tail, X, 2.0)[:1], few[:, -33:]), rows
