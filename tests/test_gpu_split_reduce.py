"""The split-j reduction at the edges of its forms: one thread per column below
32 slices, 8 or 32 threads per column from there on, sink counts that leave the
last block of columns ragged; against the oracle, with and without neighbours."""
import numpy as np
import pytest

from _parity import check, gpu_run, oracle_ref, state

pytestmark = pytest.mark.gpu
SHAPE = dict(threads=64, i_per_thread=1, j_lanes=2, j_tile=16, ctas_per_sm=0)


@pytest.fixture(scope="module")
def sp2():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1510_04068_gb300 import build, sp2 as mod
    build.build()
    mod.load()
    return mod


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("split", [2, 31, 32, 33, 65, 128])
@pytest.mark.parametrize("n_i", [1, 5, 33, 520])
def test_split_reduction_edges(sp2, oracle_mod, n_i, split, mixed):
    n, eps2 = 2048, 1e-6
    s = state(n, 5, order=4)
    idx = np.sort(np.random.default_rng(n_i).permutation(n)[:n_i]).astype(np.int32)
    r = oracle_ref(oracle_mod, s, idx, order=4, eps2=eps2)
    g = gpu_run(sp2, s, idx, order=4, precision=sp2.SP2_MIXED if mixed else sp2.SP2_FP64, eps2=eps2,
                launch=dict(SHAPE, split_j=split))
    check(g, r, order=4, mixed=mixed, s=s, i_idx=idx, label=f"{n_i} sinks, {split} slices")


@pytest.mark.parametrize("order", [2, 4, 6])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("n,n_i", [(3, 1), (64, 64), (257, 200), (1000, 31), (1025, 1025), (3001, 2049)])
def test_default_shapes(sp2, oracle_mod, n, n_i, order, mixed):
    """The shape that the library picks by itself, against the oracle."""
    import torch
    eps2 = 1e-6
    s = state(n, 9, order=max(order, 4))
    idx = np.sort(np.random.default_rng(n).permutation(n)[:n_i]).astype(np.int32)
    if order == 2:  # leap-frog: sources stay where they are; acc, pot and neighbours only
        z = np.zeros_like(s["v"])
        s2 = dict(s, v=z, a=z, jerk=z, snap=None)
        r = oracle_ref(oracle_mod, s2, idx, order=4, eps2=eps2)
        dev = lambda q: torch.as_tensor(np.ascontiguousarray(q)).cuda()  # noqa: E731
        with sp2.Context(order=2, precision=sp2.SP2_MIXED if mixed else sp2.SP2_FP64, n_max=n, eps2=eps2) as c:
            c.set_j(0, dev(s["ids"]), dev(s["m"]), dev(s["x"]), None, None, None, None, None)
            c.predict(s["t"])
            acc, pot = torch.empty((n_i, 3), dtype=torch.float64, device="cuda"), torch.empty(n_i, dtype=torch.float64, device="cuda")
            c.compute(dev(idx), acc=acc, pot=pot)
            c.sync()
        tol = 1e-6 if mixed else 1e-12
        err = np.linalg.norm(acc.cpu().numpy() - r["acc"], axis=1) / np.maximum(r["sc_acc"], 1e-300)
        assert err.max() <= tol
        assert (np.abs(pot.cpu().numpy() - r["pot"]) <= tol * np.abs(r["pot"])).all()
        return
    r = oracle_ref(oracle_mod, s, idx, order=order, eps2=eps2)
    g = gpu_run(sp2, s, idx, order=order, precision=sp2.SP2_MIXED if mixed else sp2.SP2_FP64, eps2=eps2)
    check(g, r, order=order, mixed=mixed, s=s, i_idx=idx, label=f"n {n}, {n_i} sinks, order {order}")
