"""A host-only mesh (fwi_mesh_prepare_host) on a machine with a GPU: setting its velocity gives the
time step that an uploaded mesh gives, in every form of the tables; a batch on it, whose kernels
would read geometry that was never uploaded, is refused."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,layout,tc", [(2, 0, 0), (2, 1, 0), (2, 0, 1), (3, 0, 0), (3, 1, 0)])
def test_velocity_of_a_host_only_mesh(dim, layout, tc):
    import numpy as np

    import paper_2108_10946_gb300 as pkg
    from synth import meshes, models
    pkg.build()
    g = np.linspace(0, 1, 6)
    V, C = meshes.structured_tri(9, 8) if dim == 2 else meshes.kuhn_tets(g, g, g)
    dt = []
    for host_only in (True, False):
        m = pkg.Mesh(V, C, 2, 10, cfl_factor=0.8, box=[(0.2, 0.8)] * dim, layer_faces=0b1011, layer_width=0.2,
                     sigma_max=5.0, host_only=host_only, layout=layout, tensor_cores=tc)
        for f in (1.0, 1.1):  # the second call finds what the first one uploaded
            m.set_velocity(f * (models.smooth2d if dim == 2 else models.smooth3d)(m.dof_coords()))
            dt.append(m.dt)
        m.close()
    assert dt[:2] == dt[2:] and dt[0] > dt[1] > 0


def test_batch_on_a_host_only_mesh_is_refused():
    import numpy as np

    import paper_2108_10946_gb300 as pkg
    from paper_2108_10946_gb300.lib import FWI_EINVAL, FwiError
    from synth import meshes, models
    pkg.build()
    V, C = meshes.structured_tri(9, 8)
    m = pkg.Mesh(V, C, 2, 10, cfl_factor=0.8, host_only=True)
    m.set_velocity(models.smooth2d(m.dof_coords()))
    with pytest.raises(FwiError, match="host only") as ei:
        pkg.Batch(m, np.array([[0.5, 0.5]]), np.array([[0.4, 0.4]]))
    assert ei.value.code == FWI_EINVAL
    m.close()
