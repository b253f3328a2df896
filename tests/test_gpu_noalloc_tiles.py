"""ebit_fraction_noalloc at the edges of its strips (128 columns x 4 rows a
warp, 32 rows a block) on random colours and fractions: every kind of cell,
many of them with four markers, in buffers that start at odd addresses.

The oracle computes the same double area of each cell, so float fractions are
equal and double ones agree to 1e-12 (the path's tolerance); marker counts are
whole numbers; the area is a sum of at most 4e4 doubles in another order,
within 4e4 * 2^-53 relative, far below the 1e-10 asked for."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2309_00338_gb300 import ebit  # noqa: E402


def _at_odd_address(a, dtype):
    """The array's elements in a device tensor that starts one element into its buffer."""
    t = torch.empty(a.size + 1, dtype=dtype, device="cuda")[1:]
    return t.copy_(torch.from_numpy(np.ascontiguousarray(a).reshape(-1)))


@pytest.mark.parametrize("prec", [0, 1], ids=["fp64", "fp32"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (31, 8), (32, 7), (127, 31), (128, 32), (129, 33), (1, 257), (300, 1),
                                   (255, 64), (257, 95)])
def test_noalloc_random_states(nx, ny, prec):
    rng = np.random.default_rng(nx * 1000 + ny)
    S = oracle.State(nx, ny, 1.0 / nx, prec)
    S.K[...] = rng.random(S.K.shape) < 0.5
    S.Z[...] = rng.random(S.Z.shape) < 0.5
    for a in (S.sH, S.sV):
        a[...] = rng.random(a.shape)
        a.flat[:: 7] = 0.0
        a.flat[3:: 11] *= 2.0 ** -40
        if prec == 1:
            a[...] = np.minimum(a.astype(np.float32), np.float32(1 - 2.0 ** -24))
    want, area_want = oracle.fraction(S)
    dt = torch.float64 if prec == 0 else torch.float32
    C = _at_odd_address(np.full(nx * ny, np.nan), dt)
    area = torch.zeros(1, dtype=torch.float64, device="cuda")
    counts = torch.zeros(2, dtype=torch.int64, device="cuda")
    K = _at_odd_address(S.K * 255, torch.uint8)   # any non-zero byte is the reference phase
    ebit.ebit_fraction_noalloc(nx, ny, S.dx, prec, K, _at_odd_address(S.Z, torch.uint8), _at_odd_address(S.sH, dt),
                               _at_odd_address(S.sV, dt), C, area, counts)
    torch.cuda.synchronize()
    got = C.double().cpu().numpy().reshape(ny, nx)
    if prec == 1:
        assert np.array_equal(got, want)
    else:
        assert np.max(np.abs(got - want)) <= 1e-12
    assert abs(area.item() - area_want) <= 1e-10 * max(abs(area_want), 1e-30)
    assert counts.tolist() == [int(S.hasH.sum()), int(S.hasV.sum())]
