"""Kernel-level deposits where their routes change: warps whose particles lie in
one, four (summed across the warp) or more cells (added lane by lane), arrays
that start off a 16-byte boundary, absorbed particles, ragged counts, and blocks
that add enough particles to empty their 32-bit sums on the way.  Bit-exact
against the oracle's fixed-point rules."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_13092_gb300 import ecpic
    ecpic.lib()
    return ecpic


def _case(N, n, span, seed):
    rng = np.random.default_rng(seed)
    base = np.sort(rng.integers(0, max(1, N - span + 1), n)) if span < N else np.zeros(n, np.int64)
    cell = np.minimum(base + rng.integers(0, span, n), N - 1).astype(np.int32)
    xi = rng.random(n, dtype=np.float32)
    k = min(n, 60)
    xi[:k // 3] = 0.0
    xi[k // 3: 2 * k // 3] = np.float32(1) - np.float32(2 ** -24)
    xi[2 * k // 3: k] = np.float32(2 ** -31)
    cell[rng.random(n) < 0.02] = -1
    return cell, xi


def _run(E, name, N, bc, cell, xi, shift):
    dc = torch.zeros(cell.size + shift, dtype=torch.int32, device="cuda")
    dx = torch.zeros(xi.size + shift, dtype=torch.float32, device="cuda")
    dc[shift:] = torch.from_numpy(cell)
    dx[shift:] = torch.from_numpy(xi)
    S = torch.zeros(N + 1, dtype=torch.int64, device="cuda")
    p = (cell.size, dc.data_ptr() + 4 * shift, dx.data_ptr() + 4 * shift, S.data_ptr())
    if name == "quadratic":
        E.ecpic_deposit_device2(N, bc, *p)
    elif name == "noalloc":
        E.ecpic_deposit_device_noalloc(N, *p)
    else:
        E.ecpic_deposit_device(N, *p)
    torch.cuda.synchronize()
    got = S.cpu().numpy().view(np.uint64)
    keep = cell >= 0
    want = (oracle.deposit_fixed2(N, bc, cell[keep], xi[keep]) if name == "quadratic"
            else oracle.deposit_fixed(N, cell[keep], xi[keep]))
    assert np.array_equal(got, want)


@pytest.mark.parametrize("name,bc", [("linear", 0), ("noalloc", 0), ("quadratic", 0), ("quadratic", 1)])
@pytest.mark.parametrize("N,n,span", [(1, 3, 1), (2, 129, 2), (5, 1000, 4), (300, 40001, 1), (300, 40002, 4),
                                      (300, 40003, 5), (2048, 70001, 2048)])
@pytest.mark.parametrize("shift", [0, 1])
def test_deposit_routes(E, name, bc, N, n, span, shift):
    if name == "quadratic" and N < 2:
        pytest.skip("the oracle's quadratic shares need two cells")
    cell, xi = _case(N, n, span, N + n)
    _run(E, name, N, bc, cell, xi, shift)


@pytest.mark.parametrize("name,N,n", [("linear", 700, (1 << 26) + 3), ("noalloc", 2048, (1 << 24) + 70001),
                                      ("quadratic", 700, (1 << 24) + 5)])
def test_deposit_empties_its_sums(E, name, N, n):
    cell, xi = _case(N, n, 3, n % 1000)
    _run(E, name, N, 0, cell, xi, 0)
