"""Neighbour lists around the lengths where their sort changes form: up to 256
entries ranked in shared memory, longer ones by the in-place network."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("length", [1, 31, 32, 33, 255, 256, 257, 511, 1000, 4095])
def test_lists_are_sorted_whatever_their_length(length):
    """`length` neighbours inside the radius of slot 0, all others far outside:
    the ids, ascending, are known exactly."""
    import torch

    from paper_1510_04068_gb300 import sp2
    n = length + 1 + 300
    rng = np.random.default_rng(length)
    x = rng.uniform(-0.5, 0.5, (n, 3))
    x[length + 1:] += 50.0
    x[0] = 0.0
    ids = rng.permutation(n).astype(np.int32)
    dev = lambda q: torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    z = np.zeros((n, 3))
    for prec in (sp2.SP2_MIXED, sp2.SP2_FP64):
        with sp2.Context(order=4, precision=prec, n_max=n, eps2=1e-6) as c:
            c.set_j(0, dev(ids), dev(np.ones(n)), dev(x), dev(z), dev(z), dev(z), None, dev(np.zeros(n)))
            c.predict(0.0)
            cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
            lst = torch.full((1, 4096), -1, dtype=torch.int32, device="cuda")
            c.compute_nb(dev(np.zeros(1, np.int32)), dev(np.array([4.0])), 4096, cnt, lst,
                         acc=torch.empty((1, 3), dtype=torch.float64, device="cuda"))
            c.sync()
        assert int(cnt[0]) == length
        got = lst.cpu().numpy()[0]
        np.testing.assert_array_equal(got[:length], np.sort(ids[1:length + 1]))
        assert (got[length:] == -1).all()
