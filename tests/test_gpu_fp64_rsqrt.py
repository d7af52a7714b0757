"""The reciprocal square root of the FP64 pass over random mantissas and both
parities of the exponent: the potential of two unit masses is -1 / r."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(0, 2), (-500, 500)])
def test_potential_of_pairs_is_rounded_once(lo, hi):
    import torch

    from paper_1510_04068_gb300 import sp2
    n_sys = 20000
    rng = np.random.default_rng(hi)
    r = np.ldexp(rng.uniform(0.5, 1.0, n_sys), rng.integers(lo, hi, n_sys))
    x = np.zeros((2 * n_sys, 3))
    x[1::2, 0] = r
    dev = lambda q: torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    z = dev(np.zeros((2 * n_sys, 3)))
    with sp2.Context(order=4, precision=sp2.SP2_FP64, n_max=2 * n_sys, eps2=0.0) as c:
        c.set_j(0, dev(np.arange(2 * n_sys, dtype=np.int32)), dev(np.ones(2 * n_sys)), dev(x), z, z, z, None,
                dev(np.zeros(2 * n_sys)))
        plan = c.batch_plan(np.arange(0, 2 * n_sys + 1, 2))
        c.predict(0.0)
        pot = dev(np.zeros(2 * n_sys))
        c.compute_batched(plan, pot=pot)
        c.sync()
        sp2.sp2_batch_plan_destroy(plan)
    got = pot.cpu().numpy().reshape(n_sys, 2)
    np.testing.assert_array_equal(got[:, 0], got[:, 1])
    exact = -1.0 / np.sqrt((r * r).astype(np.longdouble))
    # half a unit of the last rounding, (5/16) e^3 with e below 2^-19 (2^-58.6 is below
    # 0.021 units), and the reference's own rounding (64 bits or more: 2^-9 units)
    ulp = np.spacing(np.abs(got[:, 0]))
    assert (np.abs(got[:, 0] - exact) / ulp).max() <= 0.5 + 0.021 + 0.002
