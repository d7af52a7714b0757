"""FP64 forces of two particles over the whole range of separations: the
reciprocal square root's fast path and the arguments outside it (subnormal,
zero and overflowing squared distances, which take the library function)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEPARATIONS = [0.0, 1e-170, 1e-160, 3e-155, 1.6e-154, 1e-150, 1e-77, 7e-9, 0.3, 1.0, 123456.789, 1e77, 1e150, 1.3e154,
               1.4e154, 1e155]


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("r", SEPARATIONS)
def test_fp64_pair_over_all_separations(order, r):
    import torch

    from paper_1510_04068_gb300 import sp2
    dev = lambda q, t=torch.float64: torch.tensor(q, dtype=t, device="cuda")  # noqa: E731
    m = np.array([1.0, 0.75])
    z = [[0.0] * 3] * 2
    with sp2.Context(order=order, precision=sp2.SP2_FP64, n_max=2, eps2=0.0) as c:
        c.set_j(0, dev([5, 7], torch.int32), dev(m), dev([[0.0, 0.0, 0.0], [r, 0.0, 0.0]]), dev(z), dev(z), dev(z),
                dev(z) if order == 6 else None, dev([0.0, 0.0]))
        c.predict(0.0)
        acc, pot = torch.empty((2, 3), dtype=torch.float64, device="cuda"), dev([0.0, 0.0])
        nn, r2 = dev([0, 0], torch.int32), dev([0.0, 0.0])
        c.compute(dev([0, 1], torch.int32), acc=acc, pot=pot, nn_id=nn, nn_r2=r2)
        c.sync()
    with np.errstate(all="ignore"):
        d2 = np.float64(r) * np.float64(r)
        rinv = np.float64(1.0) / np.sqrt(d2)
        want_pot = -m[::-1] * rinv
        want_acc = m[::-1] * rinv * (rinv * rinv) * np.array([r, -r])
    # reciprocal square root within two units in the last place, one rounding each
    # for its square and the products: below 8 x 2^-53
    tol = 8 * 2.0 ** -53
    np.testing.assert_allclose(pot.cpu().numpy(), want_pot, rtol=tol, atol=0)
    np.testing.assert_allclose(acc.cpu().numpy()[:, 0], want_acc, rtol=tol, atol=1e-320)
    if np.isfinite(d2):
        assert nn.cpu().tolist() == [7, 5]
        np.testing.assert_array_equal(r2.cpu().numpy(), [d2, d2])
    else:
        assert nn.cpu().tolist() == [-1, -1]
