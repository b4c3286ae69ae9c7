"""Cached states that are exactly zero, with operators at equal times beyond them (csrc/kt_eig.cuh).

At one time both spins' c and c^+ act on orbital a: the block path closes for every kept state, but
one whose blocks hold orbital a singly occupied becomes exactly zero there, and its later states are
cached as zero. The edited window then holds two more operators at equal times. Four and seven orbitals
have block counts that fill the model's tables to the last word (128 and 2,368 blocks). The cached
results are compared with the calls from scratch, which start from the kept states: two evaluations
of one ratio, each within RTOL of the exact value, and observables within the tolerances of
tests/test_measure_gpu.py.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0908_0681_gb300 import engine, kt, workloads  # noqa: E402
from tests import parity  # noqa: E402

BETA = 4.0
OBS_ATOL = {kt.KT_FP64: 1e-9, kt.KT_FP32_KRYLOV: 3e-5}
SPECS = {3: (0.0, 5.0), 4: (0.0, 8.0), 5: (1e-2, 13.0), 7: (3e-2, 24.0)}  # trunc_eps, mu: more than half filled


def _spec(n):
    eps, mu = SPECS[n]
    delta = tuple(np.linspace(-0.05, 0.07, n).tolist())
    return workloads.ModelSpec(n, 4.0, 0.75, mu=mu, delta=delta, beta=BETA, trunc_eps=eps)


def _csr(lists):
    offs = np.cumsum([0] + [len(x) for x in lists]).astype(np.int32)
    cat = [o for x in lists for o in x]
    return workloads.Sequences(offs, np.array([o[0] for o in cat], np.float64), np.array([o[1] for o in cat], np.uint8),
                               np.array([o[2] for o in cat], np.uint8))


def _batch(n, count, seed):
    """The zeroing group early or late, a pair beside it, two ties and the window of an insertion around them."""
    rng = np.random.default_rng(seed)
    lists, kind, flavor, td, ta, rem = [], [], [], [], [], []
    for i in range(count):
        a, b, c = rng.permutation(n)[:3] if n > 2 else (0, 1, 1)
        g = int(rng.integers(2))           # c c^+ or c^+ c
        group = [(0.5, 2 * a, g), (0.5, 2 * a, 1 - g), (0.5, 2 * a + 1, g), (0.5, 2 * a + 1, 1 - g)]
        h = int(rng.integers(2))
        side = [(0.9, 2 * b, h), (1.2, 2 * b, 1 - h)]
        h = int(rng.integers(2))
        ties = [(2.0, 2 * c, h), (2.0, 2 * b + 1, h), (2.6, 2 * c, 1 - h), (2.6 + 0.2 * (i % 2), 2 * b + 1, 1 - h)]
        ops = group + side + ties
        if i % 3 == 2:                     # the same, backwards in time
            ops = [(BETA - 0.25 - t, f, d) for t, f, d in reversed(ops)]
        lists.append(ops)
        if i % 4 == 3:                     # remove a tied operator and its partner
            r = next(j for j, o in enumerate(ops) if o[1] == 2 * c and o[0] not in (0.9, 1.2))
            kind.append(1), flavor.append(2 * c), td.append(0.0), ta.append(0.0), rem.append(r)
        else:
            mid = ops[6][0] if i % 3 != 2 else ops[3][0]
            lo, hi = mid - 0.1 - 0.3 * rng.random(), mid + 0.1 + 0.3 * rng.random()
            up = rng.integers(2)
            kind.append(0), flavor.append(2 * c + 1), td.append(lo if up else hi), ta.append(hi if up else lo), rem.append(0)
    mv = workloads.Moves(np.array(kind, np.uint8), np.array(flavor, np.uint8), np.array(td), np.array(ta),
                         np.array(rem, np.int32))
    return lists, mv


def _edited(ops, mv, i):
    f = int(mv.flavor[i])
    if mv.kind[i] == 0:
        ops = ops + [(float(mv.t_dag[i]), f, 1), (float(mv.t_ann[i]), f, 0)]
        return sorted(ops, key=lambda o: o[0])   # stable: equal times keep their order
    r = int(mv.rem_idx[i])
    mine = [j for j, o in enumerate(ops) if o[1] == f]
    s = mine[(mine.index(r) + 1) % len(mine)]
    return [o for j, o in enumerate(ops) if j not in (r, s)]


def _same(exact, full, part, prec):
    """Equal statuses, and equal signs and log|T| wherever the FP64 trace from scratch is not zero up to
    rounding (tests/parity.py: |T~| > zero_tol N_tr). Returns which these are."""
    f, p = ([t.cpu().numpy() for t in x] for x in (full, part))
    assert (f[2] == kt.KT_OK).all() and (p[2] == kt.KT_OK).all()
    m, call = exact
    q = kt.kt_model_query(m)
    sign, log = (t.cpu().numpy() for t in engine.trace_ratio(m, *call)[:2])
    nz = (sign != 0) & (log > np.log(parity.ZERO_TOL[kt.KT_FP64] * q["n_kept"]) - BETA * q["E0"])
    assert nz.any() and (f[0][nz] == p[0][nz]).all() and (f[0][nz] == sign[nz]).all()
    assert np.abs(f[1][nz] - p[1][nz]).max() <= parity.RATIO_RTOL[prec]
    return nz


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("n_orb,count", [(3, 240), (3, 2600), (4, 240), (5, 240), (7, 48)])
def test_ratios_and_commits(n_orb, count, prec):
    m, m64 = engine.model_from_spec(_spec(n_orb), precision=prec), engine.model_from_spec(_spec(n_orb))
    lists, mv = _batch(n_orb, count, 7 * n_orb)
    one, zero = torch.ones(count, dtype=torch.int8, device="cuda"), torch.zeros(count, dtype=torch.float64, device="cuda")
    cache = engine.RatioCache(m, count, max_ops=16)
    d = engine.DeviceSeqs.from_host(_csr(lists))
    cache.build(d)
    hits = 0
    for step in range(3):
        dm = engine.DeviceMoves.from_host(mv)
        full = engine.trace_ratio(m, d, one, zero, dm)
        if step == 0:
            _same((m64, (d, one, zero, dm)), full, cache.ratio(d, one, zero, dm), prec)
        part = cache.propose(d, one, zero, dm)
        hits += _same((m64, (d, one, zero, dm)), full, part, prec).sum()
        acc = torch.arange(count, device="cuda") % 2 == step % 2  # an update to a zero trace as well
        cache.commit(acc.to(torch.int8), part[2])
        keep = acc.cpu().numpy()
        lists = [_edited(ops, mv, i) if keep[i] else ops for i, ops in enumerate(lists)]
        d = engine.DeviceSeqs.from_host(_csr(lists))
        # next: another pair inside the window of the last one
        mv = workloads.Moves(np.zeros(count, np.uint8), mv.flavor ^ 1, np.full(count, 1.7 + 0.05 * step),
                             np.full(count, 2.3 + 0.05 * step), np.zeros(count, np.int32))
    assert hits > count // 4


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("n_orb,count", [(3, 600), (4, 300), (7, 60)])
def test_observables_of_cached_chains(n_orb, count, prec):
    """Each step's measurement starts from cached states; the accumulated increments against kt_measure."""
    spec = _spec(n_orb)
    m = engine.model_from_spec(spec, precision=prec)
    lists, _ = _batch(n_orb, count, 5 * n_orb)
    s = engine.trace(m, engine.DeviceSeqs.from_host(_csr(lists)))[0].cpu().numpy()
    lists = [ops for ops, x in zip(lists, s) if x != 0]
    assert len(lists) > count // 8
    sw = engine.Sweep(m, workloads.semicircular_hybridization(BETA, 2 * n_orb, n_quad=256), BETA, len(lists), k_cap=16,
                      n_bins=20, measure_obs=True, cache_ops=32)
    sw.set_configs(_csr(lists))
    g = torch.Generator(device="cuda").manual_seed(3)
    last = sw.accumulators()["obs_sum"].cpu().numpy()
    for _ in range(8):
        sw.run(torch.rand((1, len(lists), 6), dtype=torch.float64, device="cuda", generator=g), meas_every=1)
        now = sw.accumulators()["obs_sum"].cpu().numpy()
        sign = sw.state()["sign"].cpu().numpy().astype(np.float64)
        ref = engine.measure(m, engine.DeviceSeqs.from_host(_csr(sw.configs())))
        want = ref[2].cpu().numpy() * sign[:, None]
        # the sums before this step are at most 8 times the observables: their rounding is far below the bound
        assert np.abs((now - last) - want).max() <= 2 * OBS_ATOL[prec] * max(1.0, np.abs(want).max())
        last = now


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("n_orb,count", [(4, 240), (4, 2600), (7, 48)])
def test_a_stale_cache_stays_in_bounds(n_orb, count, prec):
    """Sequences of the cached lengths but not the cached ones: a half's block path breaks, which counts as a
    zero. The values mean nothing; after a build for the new sequences they are those from scratch again."""
    m, m64 = engine.model_from_spec(_spec(n_orb), precision=prec), engine.model_from_spec(_spec(n_orb))
    one, zero = torch.ones(count, dtype=torch.int8, device="cuda"), torch.zeros(count, dtype=torch.float64, device="cuda")
    old, _ = _batch(n_orb, count, 1)
    new, mv = _batch(n_orb, count, 2)
    cache = engine.RatioCache(m, count, max_ops=16)
    cache.build(engine.DeviceSeqs.from_host(_csr(old)))
    d, dm = engine.DeviceSeqs.from_host(_csr(new)), engine.DeviceMoves.from_host(mv)
    for call in (cache.ratio, cache.propose):
        sign, log, status = (t.cpu().numpy() for t in call(d, one, zero, dm))
        assert np.isin(sign, (-1, 0, 1)).all() and ((status == kt.KT_OK) | (status == kt.KT_ENUMERIC)).all()
    cache.build(d)
    call = (d, one, zero, dm)
    _same((m64, call), engine.trace_ratio(m, *call), cache.ratio(*call), prec)
