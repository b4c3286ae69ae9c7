"""Observables at beta/2 with a CTA per walker (csrc/kt_eig.cuh): every surviving item counts, whichever
warp finishes first.

Walkers of 0 and 2 operators finish at once, beside long ones; the workspace is filled with other
values before every call. The (n_up, n_dn) histogram is a partition of the trace, so it sums to one:
the empty and the two-operator walkers have items of one sign, at most 64 of them, whose sum in another order
agrees to 64 2^-53 with a few roundings more of each item's exponential, below 1e-13. A batch large enough for a warp per walker adds the same items in the same order: bits.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0908_0681_gb300 import engine, kt, workloads  # noqa: E402
from tests import test_eig_zero_states_gpu as ties, test_measure_gpu as measured  # noqa: E402


def _walkers(w, n_long):
    """0 operators, 2 operators (both orders) and n_long generated walkers, interleaved."""
    long = workloads.generate_sequences(w, n_long, seed=11)
    ops = []
    for i in range(n_long):
        f = i % (2 * w.model.n_orb)
        first = (i // 2) % 2
        ops += [([], [], []), ([0.2 * w.model.beta, 0.7 * w.model.beta], [f, f], [first, 1 - first]), long.walker(i)]
    offs = np.cumsum([0] + [len(o[0]) for o in ops]).astype(np.int32)
    cat = [np.concatenate([np.asarray(o[k], np.float64) for o in ops]) for k in range(3)]
    return workloads.Sequences(offs, cat[0], cat[1].astype(np.uint8), cat[2].astype(np.uint8))


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("name,trunc_eps,n_long", [("three_orbital", 0.0, 30), ("five_orbital", None, 100),
                                                  ("seven_orbital", None, 8)])
def test_every_item_counts(name, trunc_eps, n_long, prec):
    w = workloads.WORKLOADS[name]()
    if trunc_eps is not None:
        w.model.trunc_eps = trunc_eps
    m = engine.model_from_spec(w.model, precision=prec)
    seqs = _walkers(w, n_long)
    d = engine.DeviceSeqs.from_host(seqs)
    ws = torch.empty(kt.kt_measure_workspace_size(m, seqs.n), dtype=torch.uint8, device="cuda")
    sector = engine.measure_layout(w.model.n_orb)["sector"]
    first = None
    for k in range(20):
        ws.fill_((0xFF, 0x01, 0x00)[k % 3])
        s, l, obs, st = (t.cpu().numpy() for t in engine.measure(m, d, ws=ws))
        assert (st == kt.KT_OK).all() and (s[::3] == 1).all()
        short = (np.arange(seqs.n) % 3 != 2) & (s != 0)
        assert short.sum() > n_long and np.abs(obs[short][:, sector].sum(1) - 1.0).max() <= 1e-13
        first = (s, l, obs) if first is None else first
        for a, b in zip(first, (s, l, obs)):
            assert np.array_equal(a, b, equal_nan=a.dtype == np.float64)
    if name != "seven_orbital":  # blocks of 36 rows always take a CTA per walker
        many = seqs.subset(np.arange(2500) % seqs.n)
        big = [t.cpu().numpy() for t in engine.measure(m, engine.DeviceSeqs.from_host(many))]
        for a, b in zip(first, big[:3]):
            assert np.array_equal(a[np.arange(2500) % seqs.n], b, equal_nan=a.dtype == np.float64)


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("n_orb", [3, 4])
def test_halves_without_overlap(n_orb, prec):
    """An item whose halves are a singlet and a triplet adds nothing to the trace, but n_f has an element
    between them: the oracle's observables, with its tolerances. Operators at equal times project a
    kept state on one orbital's occupation and leave such halves."""
    lists = [[(0.5, 3, 0), (0.5, 3, 1), (0.9, 4, 1), (1.2, 4, 0), (2.0, 5, 1), (2.6, 5, 0)],
             [(1.15, 1, 0), (1.75, 1, 1), (2.55, 0, 0), (2.85, 0, 1), (3.25, 3, 0), (3.25, 3, 1)],
             [(0.5, 5, 0), (0.5, 5, 1), (0.9, 0, 0), (0.963, 0, 1), (0.971, 0, 0), (1.2, 0, 1), (2.0, 1, 0), (2.6, 1, 1)],
             [(1.0, 0, 0), (1.0, 0, 1)], [(3.0, 1, 1), (3.0, 1, 0)], []]
    lists += ties._batch(n_orb, 60, 13)[0]
    measured.check(ties._spec(n_orb), ties._csr(lists), prec, f"{n_orb} orbitals, ties", min_regular=40)
