"""Where the chunk kernels put things in shared memory (host tables, no GPU).

A chunk's owned DoFs are one contiguous range of every array, copied in whole 16-byte groups from
the boundary at or below its start, while other threads copy the DoFs of the halo list one by one.
Nothing orders the two, so no group may reach a halo DoF's place. The test follows every array of
every width that a chunk kernel copies that way."""
import numpy as np
import pytest

SHARED = {(2, 2): 6, (2, 3): 9, (2, 4): 12, (2, 5): 15, (3, 2): 14, (3, 3): 28}

# k = 2 of 39,480 triangles and 20,160 tetrahedra: chunks of the most elements; the others: of 32
MESHES = [(2, 2, (140, 141)), (2, 2, (23, 19)), (2, 3, (31, 27)), (2, 4, (29, 30)), (2, 5, (33, 25)),
          (3, 2, (16, 15, 14)), (3, 2, (6, 5, 7)), (3, 3, (7, 6, 5))]


@pytest.mark.parametrize("dim,k,grid", MESHES)
def test_bulk_copies_of_owned_ranges_end_before_the_halo_places(dim, k, grid):
    import paper_2108_10946_gb300 as pkg
    from synth import meshes
    pkg.build()
    V, C = meshes.structured_tri(*grid) if dim == 2 else meshes.kuhn_tets(*[np.linspace(0, 1, g + 1) for g in grid])
    m = pkg.Mesh(V, C, k, 10, dt=1e-3, host_only=True, box=[(0.2, 0.8)] * (dim - 1) + [(-1.0, 0.8)],
                 layer_faces=0b1011 if dim == 2 else 0b101111, layer_width=0.2, sigma_max=10.0)
    nn, ns = m.element()[1].size, SHARED[dim, k]
    layer0, PE, desc, tab = m.chunk_tables()
    first_layer_dof = int(desc[layer0][2])
    assert 0 < layer0 < len(desc)
    halo_chunks = 0
    for c, (e0, ne, own, nsh, hp, hn, at, size) in enumerate(desc):
        ne &= 0xffff
        on = nsh + ne * (nn - ns)
        place = tab[2 * at:2 * at + ns * PE].reshape(ns, PE)[:, :ne].astype(int)
        halo = np.unique(place[place >= on])
        assert len(halo) == hn and np.all(place[place < on] < nsh)
        if hn == 0:
            continue
        halo_chunks += 1
        assert halo[-1] - halo[0] == hn - 1
        # (floats per DoF, array index of the first copied DoF, copied DoFs): c^2 and the gradient steps'
        # forward field like u; in the layer the nodal coefficients, omega and P (its shared DoFs)
        runs = [(1, own, on), (2, own, on), (4, own, on)]
        if c >= layer0:
            runs += [(w, own - first_layer_dof, on) for w in (1, 2, 4)]
            runs += [(dim * w, own - first_layer_dof, nsh) for w in (1, 2, 4)]
        for w, i0, n in runs:
            shift = i0 * w % 4
            end = (shift + n * w + 3) // 4 * 4 - shift  # past the first DoF's place, in floats
            assert end <= (halo[0] - on + n) * w, (c, w, i0, n)
    assert halo_chunks > len(desc) // 2
    m.close()
