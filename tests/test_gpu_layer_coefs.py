"""The damping layer's nodal coefficients as the kernels read them: Psi2 c^2 and Psi3 c^2 are formed in
FP64 and rounded once. Psi2_kk is a difference of the profile's components, which cancel where two
directions are damped, so formed from rounded components it would lose digits there.

Tolerance: one rounding to FP32, half a unit of the last place; and of the FP64 values before it, whose
differences may be contracted, a few units of FP64 of the terms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,k,grid", [(2, 3, (9, 8)), (3, 2, (6, 5, 7)), (3, 3, (4, 5, 3))])
def test_layer_coefficients_are_rounded_once(dim, k, grid):
    import paper_2108_10946_gb300 as pkg
    from synth import meshes, models
    pkg.build()
    V, C = meshes.structured_tri(*grid) if dim == 2 else meshes.kuhn_tets(*[np.linspace(0, 1, g + 1) for g in grid])
    m = pkg.Mesh(V, C, k, 10, cfl_factor=0.7, box=[(0.27, 0.71), (0.31, 0.78), (0.22, 0.83)][:dim],
                 layer_faces=0b1111 if dim == 2 else 0b111111, layer_width=0.3, sigma_max=7.0)
    c = (models.smooth2d if dim == 2 else models.smooth3d)(m.dof_coords())
    m.set_velocity(c)
    dofs, coefs = m.layer_coefs()
    s, cc = m.host_arrays()[3][dofs], (c * c)[dofs]
    assert len(np.unique(dofs)) == len(dofs) > 0
    psi2 = 2 * s - s.sum(1)[:, None]
    if dim == 2:
        want = psi2[:, :1]
    else:
        psi3 = np.stack([s[:, 1] * s[:, 2], s[:, 0] * s[:, 2], s[:, 0] * s[:, 1]], 1)
        want = np.hstack([psi2, psi3])
    want = want * cc[:, None]
    terms = (cc * s.max(1) * np.maximum(1, s.max(1)))[:, None]
    err = np.abs(coefs.astype(float) - want)
    assert np.all(err <= 2.0 ** -24 * np.abs(want) + 2.0 ** -48 * terms)
    # the case this is about: both directions damped, and a difference that is small beside its terms
    assert np.any((np.abs(psi2) < 0.2 * s.max(1)[:, None]) & (psi2 != 0))
    m.close()
