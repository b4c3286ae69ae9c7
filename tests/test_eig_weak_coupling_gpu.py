"""Traces that go through small matrix elements of the model (csrc/kt_refine.h, kt_eig_build.cu).

Two orbitals with crystal fields +-1.5: the doubly occupied ground state of one holds an admixture of about
J / 6 of the other, whatever the size of J. A c c^+ pair on the upper orbital reaches it only through that
admixture, twice. Zeros of the model stay exact zeros: without J the same sequences are structural zeros.
The reference is the long-double oracle; the tolerances are those of tests/parity.py.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0908_0681_gb300 import engine, kt, workloads  # noqa: E402
from tests import parity  # noqa: E402


def _case(J):
    spec = workloads.ModelSpec(2, 4.0, J, mu=3.0, delta=(1.5, -1.5), beta=10.0, trunc_eps=1e-6)
    rng = np.random.default_rng(5)
    lists = [[(2.0, 2, 0), (3.0, 2, 1)], [(1.0, 3, 0), (9.5, 3, 1)], [(0.0, 2, 0), (0.1, 3, 0), (0.2, 2, 1), (5.0, 3, 1)]]
    for _ in range(20):
        t = np.sort(rng.uniform(0, 10.0, 4))
        lists.append([(t[0], 2, 0), (t[1], 3, 0), (t[2], 2, 1), (t[3], 3, 1)])
    offs = np.cumsum([0] + [len(x) for x in lists]).astype(np.int32)
    cat = [o for x in lists for o in x]
    return spec, workloads.Sequences(offs, np.array([o[0] for o in cat]), np.array([o[1] for o in cat], np.uint8),
                                     np.array([o[2] for o in cat], np.uint8))


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("J", [1e-6, 1e-10, 1e-12, 1e-13, 1e-15, 0.0])
def test_admixtures_of_every_size(J, prec):
    spec, seqs = _case(J)
    o64, ox = parity.oracle_pair(spec)
    _, sx, lx = parity.oracle_traces(o64, ox, seqs)
    s, l, st = (t.cpu().numpy() for t in engine.trace(engine.model_from_spec(spec, precision=prec),
                                                      engine.DeviceSeqs.from_host(seqs)))
    assert (st == kt.KT_OK).all()
    assert (sx != 0).all() if J else (sx == 0).all()
    parity.compare(np.where(sx != 0, 2, 0), sx, lx, s, l, prec, ox.nkept, spec.beta * ox.E0, f"J = {J}")


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("name,n", [("three_orbital", 500), ("five_orbital", 96)])
def test_model_zeros_stay_zero(name, n, prec):
    """Parameters without a short binary form: energies that a symmetry makes equal differ in their last bits
    when they are summed in FP64, and elements that it forbids would not vanish."""
    w = workloads.WORKLOADS[name]()
    w.model.U, w.model.J = 5.9, 1.1
    w.model.mu = 0.5 * (5.9 + (w.model.n_orb - 1) * (2 * w.model.up - 1.1))  # half filling
    seqs = workloads.generate_sequences(w, n, seed=21)
    o64, ox = parity.oracle_pair(w.model)
    cls, sx, lx = parity.oracle_traces(o64, ox, seqs)
    assert (cls == 2).sum() > n // 5
    s, l, _ = (t.cpu().numpy() for t in engine.trace(engine.model_from_spec(w.model, precision=prec),
                                                     engine.DeviceSeqs.from_host(seqs)))
    parity.compare(cls, sx, lx, s, l, prec, ox.nkept, w.model.beta * ox.E0, name)
