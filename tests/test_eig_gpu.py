"""Traces in the block eigenbasis (csrc/kt_eig.cuh) over the forms that the route accepts.

The oracle is the reference, with the tolerances of tests/parity.py. The route with a lowered
Krylov cap (krylov_pmax below the block size) keeps the Krylov propagation and its outcomes.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0908_0681_gb300 import engine, kt, workloads  # noqa: E402
from tests import parity  # noqa: E402

PRECS = [(kt.KT_FP64, 0), (kt.KT_FP32_KRYLOV, 0), (kt.KT_FP32_KRYLOV, kt.KT_FP32_TRIDIAG64)]


def _workload(n_orb, trunc_eps, lam, beta=8.0, start="coin"):
    delta = tuple(np.linspace(-0.05, 0.07, n_orb).tolist())
    spec = workloads.ModelSpec(n_orb, 4.0, 1.0, mu=2.0 + n_orb, delta=delta, beta=beta, trunc_eps=trunc_eps)
    return workloads.Workload("eig", spec, start=start, order="poisson", lam=lam, pattern_singles=n_orb)


def _check(w, seqs, prec, flags, density=False):
    o64, ox = parity.oracle_pair(w.model, density_only=density)
    cls, sx, lx = parity.oracle_traces(o64, ox, seqs)
    m = engine.model_from_spec(w.model, precision=prec, flags=flags)
    s, l, st = (t.cpu().numpy() for t in engine.trace(m, engine.DeviceSeqs.from_host(seqs)))
    assert (st == kt.KT_OK).all()
    return m, parity.compare(cls, sx, lx, s, l, prec, ox.nkept, w.model.beta * ox.E0, "eig"), (cls, sx, lx)


@pytest.mark.parametrize("prec,flags", PRECS)
@pytest.mark.parametrize("n_orb,extra,trunc_eps,n", [
    (1, 0, 0.0, 33), (2, kt.KT_SECTOR_BLOCKS, 0.0, 40), (3, kt.KT_SECTOR_BLOCKS, 1e-10, 65),  # sectors up to 9 rows
    (4, kt.KT_SECTOR_BLOCKS, 0.0, 24),   # sectors up to 36 rows, all 256 states kept
    (4, kt.KT_DENSITY_ONLY, 1e-10, 50),  # diagonal blocks
    (5, 0, 0.0, 12),                     # 1,024 kept states: several rounds of 64
    (3, 0, 1e-10, 3000), (3, 0, 1e-10, 1),  # a warp per walker; a CTA per walker
])
def test_models_and_batches(n_orb, extra, trunc_eps, n, prec, flags):
    w = _workload(n_orb, trunc_eps, 1.5)
    _check(w, workloads.generate_sequences(w, n, seed=n_orb + n), prec, flags | extra, bool(extra & kt.KT_DENSITY_ONLY))


@pytest.mark.parametrize("prec,flags", PRECS)
@pytest.mark.parametrize("name,grid", [("three_orbital", 16), ("three_orbital", 64), ("five_orbital", 64)])
def test_operators_at_equal_times(name, grid, prec, flags):
    """Times on a coarse grid: array order decides, and exact zeros stay exact; the cache too."""
    w = workloads.WORKLOADS[name]()
    seqs = workloads.generate_sequences(w, 500 if name == "three_orbital" else 96, seed=3)
    seqs.tau[:] = np.floor(seqs.tau / w.model.beta * grid) * (w.model.beta / grid)
    m, _, (cls, sx, lx) = _check(w, seqs, prec, flags)
    moves = workloads.generate_moves(w, seqs, seed=4)
    cur = torch.as_tensor(np.where(cls == 2, sx, 0).astype(np.int8), device="cuda")
    log = torch.as_tensor(lx, device="cuda")
    d, mv = engine.DeviceSeqs.from_host(seqs), engine.DeviceMoves.from_host(moves)
    full = [t.cpu().numpy() for t in engine.trace_ratio(m, d, cur, log, mv)]
    cache = engine.RatioCache(m, seqs.n, max_ops=256)
    cache.build(d)
    part = [t.cpu().numpy() for t in cache.ratio(d, cur, log, mv)]
    assert (full[2] == part[2]).all() and (full[0] == part[0]).all()
    nz = full[0] != 0
    assert nz.sum() > 50
    assert np.abs(full[1][nz] - part[1][nz]).max() <= 2 * parity.RTOL[prec]


@pytest.mark.parametrize("prec,flags", PRECS)
def test_long_and_short_sequences(prec, flags):
    """0, 2 and 4 operators beside 1,000 in one batch, halves of every remainder modulo the lane groups."""
    w = _workload(2, 1e-10, 1.0, beta=30.0)
    rng = np.random.default_rng(7)
    lists = [[]]
    for k in [1, 1, 1, 2, 2, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 64, 125]:
        ops = []
        for f in range(4):
            first = int(rng.integers(2))
            ops += [(float(t), f, (first + j) % 2) for j, t in enumerate(np.sort(rng.uniform(0, 30.0, 2 * k if f != 3 else 2)))]
        lists.append(sorted(ops))
    offs = np.cumsum([0] + [len(x) for x in lists]).astype(np.int32)
    cat = [o for x in lists for o in x]
    seqs = workloads.Sequences(offs, np.array([o[0] for o in cat]), np.array([o[1] for o in cat], np.uint8),
                               np.array([o[2] for o in cat], np.uint8))
    _check(w, seqs, prec, flags)


def test_counted_calls_and_lowered_caps_keep_the_krylov_route():
    """kt_stats describes the Krylov propagation, and KT_ENOCONV outcomes stay: a cap of two leaves
    intervals unconverged; counted and uncounted calls agree, on the cache as well."""
    w = workloads.five_orbital()
    seqs = workloads.generate_sequences(w, 64, seed=5)
    d = engine.DeviceSeqs.from_host(seqs)
    capped = engine.model_from_spec(w.model, precision=kt.KT_FP64, krylov_pmax=2)
    assert int((engine.trace(capped, d)[2] == kt.KT_ENOCONV).sum()) > 0
    for prec in (kt.KT_FP64, kt.KT_FP32_KRYLOV):
        m = engine.model_from_spec(w.model, precision=prec)
        st = engine.new_stats()
        s, l, _ = engine.trace(m, d)
        s2, l2, _ = engine.trace(m, d, stats=st)
        wk = kt.stats_from_tensor(st)
        assert wk["krylov_iters"] > wk["intervals"] > 0 and sum(wk["p_hist"]) == wk["intervals"]
        assert bool((s == s2).all()) and float((l - l2).abs().max()) <= 2 * parity.RTOL[prec]
        mv = engine.DeviceMoves.from_host(workloads.generate_moves(w, seqs, seed=6))
        cache = engine.RatioCache(m, seqs.n, max_ops=256)
        cache.build(d)
        a, b = cache.ratio(d, s, l, mv), cache.ratio(d, s, l, mv, stats=st)
        nz = a[0] != 0
        assert bool((a[0] == b[0]).all()) and float((a[1] - b[1])[nz].abs().max()) <= 2 * parity.RTOL[prec]
