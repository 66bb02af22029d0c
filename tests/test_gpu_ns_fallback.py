"""An NS solve whose FGMRES stagnates late goes on with the BiCGStab refinement, whose limit of 60
steps does not count the restart cycles before it.  FGMRES(16) with the inverted blocks on this
octree stagnates after more than 60 cycles or so (how many varies with the order of the
atomics), and the refinement then converges in a few steps."""
import numpy as np
import pytest

from paper_2301_05985_gb300 import workloads as W

from test_gpu_ns import NsPair, _vel

pytestmark = pytest.mark.gpu


def test_late_stagnation_is_refined():
    oc = W.random_balanced_octants(2, 2, 6, 0.3, 11)
    for _ in range(4):
        P = NsPair(oc, dict(eps=0.1, dt=1e-3, beta0=1.5, beta1=-2.0, beta2=0.5),
                   dict(ns_Sc=1.0, ns_kappa=0.5, ns_rtol=1e-11, ns_atol=0.0, ns_mg_levels=0, ns_max_it=20000,
                        ns_fgmres=16), lid=0.3)
        n = P.mesh.n_nodes
        rng = np.random.default_rng(5)
        U = W.random_state(P.mesh.ijk, oc.max_level, 2)
        P.set_history(_vel(n, 2, rng, 0.3), _vel(n, 2, rng, 0.3), U)
        st = P.ctx.ns_solve(raise_on_error=False)
        assert st.status == 0, (st.krylov_fallbacks, st.refinements, st.res_final / st.res0)
        assert st.floor_stop or st.res_final <= 1e-11 * st.res0
        P.ctx.close()
