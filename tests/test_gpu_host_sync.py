"""Host-pointer calls return when their work is done, below and above the limit
of the packed staging buffer, and read pinned inputs in stream order."""
import numpy as np
import pytest

from _parity import state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_i", [1, 317, 2500])
def test_host_set_j_of_slots_has_stored_the_particles_on_return(n_i):
    import torch

    from paper_1510_04068_gb300 import sp2
    n = 3000
    s = state(n, 4, order=4)
    slots = np.arange(n_i, dtype=np.int32)
    part = {k: s[k][:n_i] for k in ("ids", "m", "x", "v", "a", "jerk", "tj")}
    stream = torch.cuda.current_stream()
    with sp2.Context(order=4, n_max=n, eps2=1e-6) as c:
        c.set_j(0, s["ids"], s["m"], s["x"], s["v"], s["a"], s["jerk"], None, s["tj"])
        torch.cuda._sleep(100_000_000)  # some 50 ms in front of the call's own work
        c.set_j(0, part["ids"], part["m"], part["x"], part["v"], part["a"], part["jerk"], None, part["tj"], slots=slots)
        assert stream.query()


def _pinned(torch, q):
    return torch.as_tensor(np.ascontiguousarray(q)).pin_memory()


def test_pinned_inputs_are_read_in_stream_order():
    """Pinned arrays that a queued copy out of the device still has to fill: new
    particles of set_j, explicit sinks and the radii of the neighbour lists."""
    import torch

    from paper_1510_04068_gb300 import sp2
    n, n_i = 3000, 200
    s = state(n, 6, order=4)
    rng = np.random.default_rng(6)
    slots = np.sort(rng.permutation(n)[:n_i]).astype(np.int32)
    h2 = np.full(n_i, 0.02)
    x = rng.standard_normal((n_i, 3))

    def run(late):
        def give(q):  # the array itself, or a pinned one that the stream fills after a delay
            p = _pinned(torch, np.zeros_like(q))
            src = torch.as_tensor(q).cuda()
            if late:
                torch.cuda._sleep(20_000_000)
                p.copy_(src, non_blocking=True)
            else:
                p.copy_(torch.as_tensor(q))
            return p

        res = []
        part = [_pinned(torch, s[k][slots]) for k in ("ids", "m", "v", "a", "jerk", "tj")]
        with sp2.Context(order=4, n_max=n, eps2=1e-6) as c:
            c.set_j(0, s["ids"], s["m"], s["x"], s["v"], s["a"], s["jerk"], None, s["tj"])
            c.set_j(0, part[0], part[1], give(x), part[2], part[3], part[4], None, part[5], slots=_pinned(torch, slots))
            got = np.empty((n, 3))
            c.get_j(0, n, x=got)
            res.append(got)
            c.predict(s["t"])
            acc = torch.empty((n_i, 3), dtype=torch.float64).pin_memory()
            c.compute_ext(give(x), _pinned(torch, np.zeros((n_i, 3))), acc=acc)
            res.append(acc.numpy().copy())
            cnt = torch.zeros(n_i, dtype=torch.int32).pin_memory()
            lst = torch.zeros((n_i, 64), dtype=torch.int32).pin_memory()
            c.compute_nb(_pinned(torch, slots), give(h2), 64, cnt, lst, acc=acc)
            res.append(cnt.numpy().copy())
        return res

    for a, b in zip(run(False), run(True)):
        np.testing.assert_array_equal(a, b)
