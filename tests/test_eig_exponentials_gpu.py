"""The exponential of an interval in the block eigenbasis (csrc/kt_eig.cuh), over intervals of every size.

Two orbitals, c c^+ c c^+ of one flavor: between the two middle operators the vector has two components and
T is proportional to a + b exp(-x), x = dt gap. Bounds on log|T| against the long-double oracle: FP64 keeps
the exponential to a few ulp of the weight and x to an ulp, beside the ulp of the logarithms summed into
log|T|; a pair of floats keeps components above 1/16 to 2^-35, which four operators and the
exponential's 2^-36 leave below 2^-26.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_0908_0681_gb300 import engine, kt, workloads  # noqa: E402
from tests import parity  # noqa: E402


@pytest.mark.parametrize("prec", [kt.KT_FP64, kt.KT_FP32_KRYLOV])
@pytest.mark.parametrize("beta", [20.0, 450.0])  # x up to 35, to the last bit of log|T| = 100; up to 880
def test_intervals_of_every_size(beta, prec):
    spec = workloads.ModelSpec(2, 4.0, 1.0, mu=3.0, delta=(0.01, -0.01), beta=beta, trunc_eps=1e-10)
    dts = np.concatenate([np.geomspace(1e-9, beta - 3.0, 500), np.linspace(0.01, 17.0, 500)])
    n = len(dts)
    tau = np.stack([np.full(n, 1.0), np.full(n, 1.5), 1.5 + dts, 2.0 + dts], 1).ravel()
    seqs = workloads.Sequences(4 * np.arange(n + 1, dtype=np.int32), tau, np.full(4 * n, 1, np.uint8),
                               np.tile(np.array([0, 1, 0, 1], np.uint8), n))
    _, ox = parity.oracle_pair(spec)
    sx, lx, _ = ox.trace(parity.seqbatch(seqs))
    s, l, st = (t.cpu().numpy() for t in engine.trace(engine.model_from_spec(spec, precision=prec),
                                                      engine.DeviceSeqs.from_host(seqs)))
    assert (st == kt.KT_OK).all() and (sx != 0).all() and (s == sx).all()
    bound = 2.0 ** -52 * (16.0 + 2.0 * np.abs(lx)) if prec == kt.KT_FP64 else 2.0 ** -26 + 2.0 ** -52 * 2.0 * np.abs(lx)
    assert (np.abs(l - lx) <= bound).all()
