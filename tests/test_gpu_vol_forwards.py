"""The static formulas at forwards other than 1, against the FP64 oracle.  FP64:
1e-12 relative.  FP32: the 3e-5 that hold at a forward of 1, and 5e-6 for the
roundings that come with another: of f in ln(f/K) (nu / alpha <= 50, half a unit
in 2^-24: 1.5e-6) and of log2(K f), here up to 24 (24 x 2^-24 ln 2 in the exponent of
(K f)^((1 - beta)/2), which enters alpha / fk and z: below 3e-6)."""
import numpy as np
import pytest

import oracle as O
import paper_2407_20713_gb300 as sg

pytestmark = pytest.mark.gpu

TOL = {sg.FP64: 1e-12, sg.FP32: 3.5e-5}


@pytest.mark.parametrize("fwd", [0.03, 1.0, 87.5, 4000.0])
@pytest.mark.parametrize("prec", [sg.FP64, sg.FP32])
@pytest.mark.parametrize("model", [sg.HAGAN, sg.OBLOJ, sg.EXPANDED])
def test_static_formulas_at_any_forward(model, prec, fwd):
    rng = np.random.default_rng(7 + model)
    n = 256 + 19
    for trial in range(4):
        p = [rng.uniform(0.05, 0.8), rng.uniform(0, 1), rng.uniform(-0.95, 0.95), rng.uniform(0.05, 2.5)]
        p[0] *= fwd ** (1 - p[1])  # the same volatility at the money for every forward
        K = fwd * rng.uniform(0.5, 1.6, n)
        K[:5] = fwd * np.array([1.0, 1.0 + 1e-7, 1.0 - 1e-7, 1.0 + 1e-4, 0.999])
        T = rng.choice([0.05, 0.25, 1.0, 5.0], n)
        got = sg.implied_vol(model, p, fwd, T, K, prec=prec).cpu().numpy()
        ref = O.implied_vol(model, p, fwd, T, K)
        rel = np.abs(got - ref) / np.abs(ref)
        assert rel.max() <= TOL[prec], (p, rel.argmax(), rel.max())
