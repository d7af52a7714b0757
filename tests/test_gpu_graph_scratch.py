"""A captured graph keeps working after an eager call that needed larger scratch:
the outgrown buffers stay allocated while a graph exists and are given back after."""
import numpy as np
import pytest

from _parity import state

pytestmark = pytest.mark.gpu


def test_replay_after_the_scratch_has_grown():
    import torch

    from paper_1510_04068_gb300 import sp2
    live, freed = {}, []

    @sp2.ALLOC_FN
    def alloc(nbytes, user):
        buf = torch.empty(max(int(nbytes), 16), dtype=torch.uint8, device="cuda")
        live[buf.data_ptr()] = buf  # the buffer lives as long as it is in here
        return buf.data_ptr()

    @sp2.FREE_FN
    def free(ptr, user):
        freed.append(ptr)
        del live[ptr]

    n, n_i = 6000, 40
    s = state(n, 31, order=4)
    dev = lambda q: torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    outputs = lambda k: dict(acc=torch.zeros((k, 3), dtype=torch.float64, device="cuda"),  # noqa: E731
                             pot=torch.zeros(k, dtype=torch.float64, device="cuda"),
                             nn_id=torch.zeros(k, dtype=torch.int32, device="cuda"))
    stream = torch.cuda.Stream()  # a capture takes no legacy default stream
    with torch.cuda.stream(stream):
        c = sp2.Context(order=4, n_max=n, eps2=1e-6, alloc=alloc, free=free)
        c.set_j(0, dev(s["ids"]), dev(s["m"]), dev(s["x"]), dev(s["v"]), dev(s["a"]), dev(s["jerk"]), None, dev(s["tj"]))
        small, big = dev(np.arange(n_i, dtype=np.int32)), dev(np.arange(n, dtype=np.int32))
        xs = dev(s["x"][:n_i])
        o, e, ob = outputs(n_i), outputs(n_i), outputs(n)

        def step():
            c.predict(s["t"])
            c.compute(small, **o)
            c.compute_ext(xs, xs, **e)

        step()
        c.sync()
        want = {k: v.cpu().numpy().copy() for k, v in o.items()}
        want_e = {k: v.cpu().numpy().copy() for k, v in e.items()}
        sp2.sp2_graph_begin(c.ctx)
        step()
        g = sp2.sp2_graph_end(c.ctx)
        before = set(live)
        for _ in range(2):  # grows the partial sums and the sink records
            c.compute(big, **ob)
            c.compute_ext(dev(s["x"]), dev(s["v"]), **ob)
        c.sync()
        assert set(live) > before and not freed
        for q in (*o.values(), *e.values()):
            q.zero_()
        sp2.sp2_graph_launch(c.ctx, g)
        c.sync()
        for k in o:
            np.testing.assert_array_equal(o[k].cpu().numpy(), want[k], err_msg=k)
            np.testing.assert_array_equal(e[k].cpu().numpy(), want_e[k], err_msg=k)
        sp2.sp2_graph_destroy(g)
        c.sync()
        assert freed  # the outgrown buffers
        c.close()
        assert not live
