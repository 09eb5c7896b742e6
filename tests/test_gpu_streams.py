"""The kernels' tables of a context are rebuilt and uploaded on the context's stream when the constants they depend on
change: on a non-blocking stream, call after call with another screening constant, every result is bit for bit that of a
fresh context on the default stream."""
import numpy as np
import pytest

from paper_2109_09772_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import torch

    from paper_2109_09772_gb300 import build as B
    from paper_2109_09772_gb300 import rism

    B.build()
    torch.cuda.set_device(0)
    return rism


def _init(r, g):
    return r.init()


def _lra(r, g):
    T, sums = r.lra_integral(atom_sums=True)
    return {"T": T, "sums": sums}


def _backward(r, g):
    return r.backward(g, g, g)


@pytest.mark.parametrize("call, method, precision", [(_init, "DIRECT", "FP32"), (_init, "DIRECT", "FP64"),
                                                     (_init, "TREECODE", "FP32"), (_lra, "DIRECT", "FP32"),
                                                     (_backward, "DIRECT", "FP32"), (_backward, "TREECODE", "FP32")])
def test_tables_follow_the_solvent_on_a_non_blocking_stream(R, call, method, precision):
    import torch

    w = I.small_workload(n_atoms=90, n=(34, 20, 18), h=0.5, seed=81, ions=True, lj_rcut=5.0, net=1.0)
    opts = dict(method=getattr(R, "METHOD_" + method), precision=getattr(R, "PREC_" + precision))
    g = torch.randn((w.solvent.nsite, 18, 20, 34), dtype=torch.float64, device="cuda",
                    generator=torch.Generator("cuda").manual_seed(7))
    torch.cuda.synchronize()

    def solvent(r, scale):  # kappa grows with the square root of the ionic densities
        s = w.solvent
        r.set_solvent(s.q, s.sigma, s.eps, s.rho * np.where(s.is_ion != 0, scale, 1.0), s.is_ion)

    want = {}
    scales = (1.0, 9.0, 40.0)
    for scale in scales:
        r = R.from_workload(w, **opts)
        solvent(r, scale)
        want[scale] = call(r, g)
        torch.cuda.synchronize()
        r.close()
    r = R.from_workload(w, stream=torch.cuda.Stream(), **opts)
    for scale in scales * 3:
        solvent(r, scale)
        got = call(r, g)
        r.stream.synchronize()
        for k, v in want[scale].items():
            assert torch.equal(torch.as_tensor(got[k]), torch.as_tensor(v)), (scale, k)
    r.close()
