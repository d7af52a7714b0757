"""Host-pointer calls through the packed staging buffer and beyond its size,
against the same calls on device arrays; block sizes around the rounding of
the staging slots, and the caller's arrays overwritten right after a call."""
import numpy as np
import pytest

from _parity import state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_i", [1, 15, 16, 17, 32, 33, 317, 900, 2000])
def test_host_block_steps_equal_device_block_steps(n_i):
    import torch

    from paper_1510_04068_gb300 import sp2
    n = 3000
    s = state(n, 3, order=4)
    rng = np.random.default_rng(n_i)
    dev = lambda q: torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    with sp2.Context(order=4, n_max=n, eps2=1e-6) as a, sp2.Context(order=4, n_max=n, eps2=1e-6) as b:
        for c in (a, b):
            c.set_j(0, dev(s["ids"]), dev(s["m"]), dev(s["x"]), dev(s["v"]), dev(s["a"]), dev(s["jerk"]), None, dev(s["tj"]))
        for _ in range(3):
            slots = np.sort(rng.permutation(n)[:n_i]).astype(np.int32)
            new = dict(id=s["ids"][slots], m=rng.uniform(0.5, 1.5, n_i) / n, x=rng.standard_normal((n_i, 3)),
                       v=rng.standard_normal((n_i, 3)), a=rng.standard_normal((n_i, 3)),
                       jerk=rng.standard_normal((n_i, 3)), snap=None, t=np.full(n_i, 0.75))
            out = dict(acc=(n_i, 3), jerk=(n_i, 3), pot=(n_i,), nn_id=(n_i,), nn_r2=(n_i,))
            host = {k: np.zeros(q, np.int32 if k == "nn_id" else np.float64) for k, q in out.items()}
            gpu = {k: dev(q) for k, q in host.items()}
            b.set_j(0, **{k: None if q is None else dev(q) for k, q in new.items()}, slots=dev(slots))
            a.set_j(0, **new, slots=slots)
            for q in new.values():
                if q is not None:
                    q[...] = 0  # the call has taken its inputs
            for c, o, i in ((a, host, slots), (b, gpu, dev(slots))):
                c.predict(1.0)
                c.compute(i, **o)
            b.sync()
            for k in host:
                np.testing.assert_array_equal(host[k], gpu[k].cpu().numpy(), err_msg=k)
