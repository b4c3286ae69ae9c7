"""Sweep steps at orders around the widths of the kernels: the new column, row and corner of the bath
matrix share the lanes of a warp (2 k + 1 = 31, 33 .. values), its products go by 32 rows, sequences
by 128 operators. One orbital, every eigenstate kept: the chains take the oracle's decisions."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle import mlp as ref  # noqa: E402
from oracle.ctqmc import Hyb, chain, chain_da_multi  # noqa: E402
from paper_0908_0681_gb300 import engine, kt, workloads  # noqa: E402
from tests.test_sweep_gpu import model_pair  # noqa: E402


@pytest.mark.parametrize("tries", [0, 3])
def test_orders_around_the_lane_counts(tries):
    spec = workloads.ModelSpec(1, 2.0, 0.0, mu=1.0, delta=(0.0,), beta=30.0, trunc_eps=0.0)
    om, gm = model_pair(spec, kt.KT_FP64)
    table = workloads.semicircular_hybridization(spec.beta, 2, n_tau=2000)
    rng = np.random.default_rng(11)
    init = []
    for k in [(0, 0), (1, 1), (15, 2), (16, 1), (17, 15), (31, 3), (32, 32), (33, 31), (48, 16), (64, 1)]:
        ops = []
        for f in range(2):
            first = int(rng.integers(2))
            ops += [(float(t), f, (first + j) % 2) for j, t in enumerate(np.sort(rng.uniform(0, spec.beta, 2 * k[f])))]
        init.append(sorted(ops))
    nw, steps, k_cap = len(init), 40, 65
    offs = np.cumsum([0] + [len(c) for c in init]).astype(np.int32)
    cat = [o for c in init for o in c]
    sw = engine.Sweep(gm, table, spec.beta, nw, k_cap=k_cap, n_bins=10)
    sw.set_configs(workloads.Sequences(offs, np.array([o[0] for o in cat]), np.array([o[1] for o in cat], np.uint8),
                                       np.array([o[2] for o in cat], np.uint8)))
    if tries == 0:
        u = rng.random((steps, nw, 6))
        sw.run(torch.as_tensor(u, device="cuda"))
        out = chain(om, Hyb(table, spec.beta), init, u, k_cap=k_cap)
    else:
        n_in, c = ref.n_inputs(2), -0.3
        p = {k: np.zeros(s) for k, s in ref.shapes(n_in).items()}
        p["b3"] = np.array([c])
        sw.set_surrogate(engine.Surrogate(n_in, max_batch=(nw * tries + 15) // 16 * 16, params=ref.pack(p)))
        u = rng.random((steps, nw, tries, 7))
        sw.run_da_multi(torch.as_tensor(u, device="cuda"))
        cf = float(np.float32(c))
        out = chain_da_multi(om, Hyb(table, spec.beta), init, u, lambda ops, kind, *a: cf if kind == 0 else -cf,
                             k_cap=k_cap)
        assert sw.counters()["stage1_rejected"] == out["counts"]["stage1_rejected"] > 0
    assert sw.configs() == out["configs"]
    cnt = sw.counters()
    assert cnt["insert_accepted"] + cnt["remove_accepted"] == int((out["accepted"] == 1).sum()) > nw
