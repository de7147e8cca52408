"""The library's coexistence densities (closed-form bisection, then Newton steps
on the quadrature) against the oracle's Maxwell construction, from density
ratio 1600 to the neighbourhood of the critical point, where the closed form
alone would cancel.  The densities are as sharp as the root of the area: its
slope falls with the density gap, so the bar widens as 1e-9 / (1 - T)."""
import pytest

import oracle as O
from tests._cases import Case


@pytest.mark.parametrize("eos", [O.EOS_VDW, O.EOS_CS])
@pytest.mark.parametrize("T", [0.35, 0.5, 0.7, 0.9, 0.99, 0.999])
def test_densities_match_the_oracle(eos, T):
    from paper_1512_01977_gb300 import build, lbm

    build.build()
    gv, gl = lbm.lbm_eos_coexistence(lbm.make_eos(eos, T))
    rv, rl = Case(16, 16, eos=eos, T_over_Tc=T).coexistence()
    tol = 1e-9 / (1.0 - T)
    assert abs(gv / rv - 1) <= tol and abs(gl / rl - 1) <= tol
