"""Host-pointer calls return when their work is done, whatever the size of the
arrays: below and above the limit of the packed staging buffer."""
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
