"""Default launch shapes under an allocator with a budget: where the partial sums
of the fastest split do not fit, the pass runs with fewer slices."""
import numpy as np
import pytest

from _parity import check, oracle_ref, state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("budget", [0, 100_000])
def test_fewer_slices_when_scratch_is_refused(oracle_mod, budget, mixed):
    import torch

    from paper_1510_04068_gb300 import sp2
    live, refused, spare = {}, [], [None]

    @sp2.ALLOC_FN
    def alloc(nbytes, user):
        if spare[0] is not None and int(nbytes) > spare[0]:
            refused.append(int(nbytes))
            return None
        buf = torch.empty(max(int(nbytes), 16), dtype=torch.uint8, device="cuda")
        live[buf.data_ptr()] = buf
        return buf.data_ptr()

    @sp2.FREE_FN
    def free(ptr, user):
        del live[ptr]

    n, n_i, eps2 = 4000, 700, 1e-6
    s = state(n, 41, order=4)
    idx = np.sort(np.random.default_rng(7).permutation(n)[:n_i]).astype(np.int32)
    dev = lambda q: torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    out = dict(acc=torch.zeros((n_i, 3), dtype=torch.float64, device="cuda"),
               jerk=torch.zeros((n_i, 3), dtype=torch.float64, device="cuda"),
               pot=torch.zeros(n_i, dtype=torch.float64, device="cuda"),
               nn_id=torch.zeros(n_i, dtype=torch.int32, device="cuda"),
               nn_r2=torch.zeros(n_i, dtype=torch.float64, device="cuda"))
    c = sp2.Context(order=4, precision=sp2.SP2_MIXED if mixed else sp2.SP2_FP64, n_max=n, eps2=eps2, alloc=alloc, free=free)
    c.set_j(0, dev(s["ids"]), dev(s["m"]), dev(s["x"]), dev(s["v"]), dev(s["a"]), dev(s["jerk"]), None, dev(s["tj"]))
    c.predict(s["t"])
    spare[0] = budget  # bytes that a single further allocation may have
    for _ in range(2):
        c.compute(dev(idx), **out)
    c.sync()
    first = len(refused)
    c.compute(dev(idx), **out)
    c.sync()
    assert 0 < first == len(refused)  # what was refused is not asked for again
    r = oracle_ref(oracle_mod, s, idx, order=4, eps2=eps2)
    check({k: v.cpu().numpy() for k, v in out.items()}, r, order=4, mixed=mixed, s=s, i_idx=idx, label=f"budget {budget}")
    c.set_launch(n_i, dict(threads=64, i_per_thread=1, j_lanes=1, j_tile=64, split_j=60, ctas_per_sm=0))
    with pytest.raises(sp2.SP2Error) as e:  # a shape that was asked for is not changed
        c.compute(dev(idx), **out)
    assert e.value.status == -3
    c.close()
    assert not live
