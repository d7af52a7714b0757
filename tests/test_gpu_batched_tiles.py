"""Batched systems whose sizes lie around multiples of the 64-source tile (full
tiles are staged by a form of their own), against the oracle, every order."""
import numpy as np
import pytest

from _parity import TOL, check, state

pytestmark = pytest.mark.gpu
SIZES = [64, 63, 65, 1, 128, 127, 129, 2, 192, 320]


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("order", [2, 4, 6])
def test_systems_around_full_tiles(oracle_mod, order, mixed):
    import torch

    from paper_1510_04068_gb300 import sp2
    off = np.concatenate([[0], np.cumsum(SIZES)]).astype(np.int64)
    n, eps2 = int(off[-1]), 1e-6
    s = state(n, 13, order=max(order, 4))
    if order == 2:  # sources stay where they are
        z = np.zeros((n, 3))
        s.update(v=z, a=z, jerk=z, snap=None)
    dev = lambda q: None if q is None else torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
    out = dict(acc=dev(np.zeros((n, 3))), pot=dev(np.zeros(n)), nn_id=dev(np.zeros(n, np.int32)), nn_r2=dev(np.zeros(n)))
    if order != 2:
        out["jerk"] = dev(np.zeros((n, 3)))
    if order == 6:
        out["snap"] = dev(np.zeros((n, 3)))
    with sp2.Context(order=order, precision=sp2.SP2_MIXED if mixed else sp2.SP2_FP64, n_max=n, eps2=eps2) as c:
        c.set_j(0, dev(s["ids"]), dev(s["m"]), dev(s["x"]), dev(s["v"]), dev(s["a"]), dev(s["jerk"]), dev(s["snap"]),
                dev(s["tj"]))
        plan = c.batch_plan(off)
        c.predict(s["t"])
        c.compute_batched(plan, **out)
        c.sync()
        sp2.sp2_batch_plan_destroy(plan)
    g = {k: v.cpu().numpy() for k, v in out.items()}
    for a, b in zip(off[:-1], off[1:]):
        if b - a == 1:
            assert g["nn_id"][a] == -1 and (g["acc"][a] == 0).all() and g["pot"][a] == 0
            continue
        idx = np.arange(a, b)
        r = oracle_mod.step(s["t"], idx, s["ids"], s["m"], s["tj"], s["x"], s["v"], s["a"], s["jerk"], s["snap"],
                            eps2=eps2, order=max(order, 4), j_range=(a, b))
        gs = {k: v[a:b] for k, v in g.items()}
        if order == 2:
            err = np.linalg.norm(gs["acc"] - r["acc"], axis=1) / r["sc_acc"]
            assert err.max() <= TOL[mixed]["acc"]
            assert (np.abs(gs["pot"] - r["pot"]) <= TOL[mixed]["pot"] * np.abs(r["pot"])).all()
        else:
            check(gs, r, order=order, mixed=mixed, s=s, i_idx=idx, label=f"system of {b - a}")
