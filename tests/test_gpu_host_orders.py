"""Host-pointer calls against the same calls on device arrays in the forms that
the order-4 mixed block step leaves out: other orders and precisions, explicit sinks,
neighbour lists and all-pairs forces with their adjoint."""
import numpy as np
import pytest

from _parity import state

pytestmark = pytest.mark.gpu


def _both(call, arrays, outs):
    """call(arrays, outs) on host arrays and on device arrays; both results."""
    import torch
    dev = lambda q: None if q is None else torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    host = {k: np.zeros(sh, dt) for k, (sh, dt) in outs.items()}
    gpu = {k: dev(v) for k, v in host.items()}
    call(arrays, host)
    call({k: dev(v) for k, v in arrays.items()}, gpu)
    torch.cuda.synchronize()
    for k in host:
        np.testing.assert_array_equal(host[k], gpu[k].cpu().numpy(), err_msg=k)


@pytest.mark.parametrize("order,mixed", [(2, True), (4, False), (6, True), (6, False)])
def test_host_calls_equal_device_calls(order, mixed):
    from paper_1510_04068_gb300 import sp2
    n, n_i = 1500, 217
    s = state(n, 8, order=max(order, 4))
    slots = np.sort(np.random.default_rng(8).permutation(n)[:n_i]).astype(np.int32)
    six = order == 6
    a = dict(id=s["ids"], m=s["m"], x=s["x"], v=s["v"], a=s["a"], jerk=s["jerk"], snap=s["snap"] if six else None, t=s["tj"])
    new = {k: None if q is None else q[slots[::-1]].copy() for k, q in a.items()}
    new["id"] = s["ids"][slots]
    F = np.float64
    out = dict(acc=((n_i, 3), F), pot=((n_i,), F), nn_id=((n_i,), np.int32), nn_r2=((n_i,), F))
    if order != 2:
        out["jerk"] = ((n_i, 3), F)
    if six:
        out["snap"] = ((n_i, 3), F)
    prec = sp2.SP2_MIXED if mixed else sp2.SP2_FP64

    def step(q, o):
        with sp2.Context(order=order, precision=prec, n_max=n, eps2=1e-6) as c:
            c.set_j(0, **{k: q[k] for k in a})
            c.set_j(0, **{k: q["new_" + k] for k in a}, slots=q["slots"])
            c.predict(s["t"])
            c.compute(q["slots"], **o)
            c.sync()

    def ext(q, o):
        with sp2.Context(order=order, precision=prec, n_max=n, eps2=1e-6) as c:
            c.set_j(0, **{k: q[k] for k in a})
            c.predict(s["t"])
            c.compute_ext(q["new_x"], q["new_v"] if order != 2 else None, q["new_a"] if six else None, i_slot=q["slots"], **o)
            c.sync()

    def lists(q, o):
        o = dict(o)
        cnt, lst = o.pop("cnt"), o.pop("lst")
        with sp2.Context(order=order, precision=prec, n_max=n, eps2=1e-6) as c:
            c.set_j(0, **{k: q[k] for k in a})
            c.predict(s["t"])
            c.compute_nb(q["slots"], q["h2"], 64, cnt, lst, **o)
            c.sync()

    arrays = dict(a, **{"new_" + k: q for k, q in new.items()}, slots=slots, h2=np.full(n_i, 1e-3))
    _both(step, arrays, out)
    _both(ext, arrays, out)
    _both(lists, arrays, dict(out, cnt=((n_i,), np.int32)) | dict(lst=((n_i, 64), np.int32)))


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("accumulate", [False, True])
def test_host_forces_and_adjoint_equal_device_calls(mixed, accumulate):
    from paper_1510_04068_gb300 import sp2
    n = 333
    s = state(n, 9, order=4)
    F = np.float64

    def run(q, o):
        with sp2.Context(order=4, precision=sp2.SP2_MIXED if mixed else sp2.SP2_FP64, n_max=n, eps2=1e-6) as c:
            c.forces(q["m"], q["x"], q["v"], acc=o["acc"], jerk=o["jerk"], pot=o["pot"])
            c.force_vjp(q["m"], q["x"], q["v"], q["a"], q["jerk"], None, o["xbar"], o["vbar"], o["mbar"],
                        accumulate=accumulate)
            c.sync()

    out = dict(acc=((n, 3), F), jerk=((n, 3), F), pot=((n,), F), xbar=((n, 3), F), vbar=((n, 3), F), mbar=((n,), F))
    _both(run, {k: s[k] for k in ("m", "x", "v", "a", "jerk")}, out)
