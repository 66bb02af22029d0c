"""The NS V-cycle with different shares of its levels in one block: 2 levels (the coarsest by
launches or in the block), up to 5 (the smallest ones together in the block, with and without
hanging nodes), on quadrilaterals and hexahedra.  One cycle is a fixed linear map but for the
order of its FP32 sums (1e-7 of it), so FGMRES takes as many iterations, to the same residual,
as with the levels launched sweep by sweep; those values are recorded here.  Their residuals
are recorded to two digits: 10 % relative is the rounding of the smallest (4.55e-13) and its
distance from the FP64 rounding of the residual."""
import numpy as np
import pytest

from paper_2301_05985_gb300 import workloads as W

from test_gpu_ns import NsPair, _vel

pytestmark = pytest.mark.gpu

# mesh, {levels: (FGMRES iterations, ||F|| / ||F_0||)} of the cycle launched sweep by sweep
MESHES = {
    "3d_uniform": (lambda: W.uniform_octants(3, 4), {2: (12, 5.3e-12), 3: (12, 1.5e-12), 4: (12, 1.5e-12), 5: (12, 1.5e-12)}),
    "3d_octree": (lambda: W.random_balanced_octants(3, 2, 4, 0.3, 12),
                  {2: (10, 1.8e-12), 3: (10, 4.55e-13), 4: (10, 4.55e-13), 5: (10, 4.55e-13)}),
    "2d_uniform": (lambda: W.uniform_octants(2, 5), {2: (16, 2.8e-12), 3: (15, 2.8e-12), 4: (14, 9.2e-12), 5: (14, 9.2e-12)}),
    "2d_octree": (lambda: W.random_balanced_octants(2, 3, 6, 0.3, 11),
                  {2: (13, 4.4e-12), 3: (12, 2.2e-12), 4: (11, 2.7e-12), 5: (11, 3.8e-13)}),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_cycle_is_the_one_launched_sweep_by_sweep(name):
    make, recorded = MESHES[name]
    oc = make()
    kw = dict(eps=0.1, dt=1e-3, beta0=1.5, beta1=-2.0, beta2=0.5, mg_smooth=3, mg_omega=0.6, mg_coarse_its=32)
    for levels, (its, res) in recorded.items():
        P = NsPair(oc, kw, dict(ns_Sc=1.0, ns_kappa=0.5, ns_rtol=1e-11, ns_atol=0.0, ns_mg_levels=levels,
                                ns_max_it=2000), lid=0.3)
        n, dim = P.mesh.n_nodes, oc.dim
        rng = np.random.default_rng(5)
        U = W.random_state(P.mesh.ijk, oc.max_level, 2)
        P.set_history(_vel(n, dim, rng, 0.3), _vel(n, dim, rng, 0.3), U)
        st = P.ctx.ns_solve()
        assert st.status == 0 and st.inner_its == its, (levels, st.inner_its)
        assert abs(st.res_final / st.res0 / res - 1.0) <= 0.1, (levels, st.res_final / st.res0)
        P.ctx.close()
