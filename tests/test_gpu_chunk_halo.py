"""Chunk boundaries, every element and every group of shots: the chunked layout against the plain one
with a velocity that has nothing to do with itself from one DoF to the next, so that a chunk which
took a neighbour's value for one of its halo DoFs is off by as much as the value itself.

The sources are moved several times over the mesh, each near a receiver (a window this short fills
their surroundings only). Two grids per kind of launch: steps one by one, and inside one launch.

Both forms get the same residuals (records that differ in their last bits, each form's own, would
send the forms' adjoint solves out with different sources: a shot whose gradient is small next to
its residual then differs by more than either form's error).

Tolerance: each form alone lies within 7e-7 (norm) of 64 bits on windows of this length, so two of
them within twice that; twice again for margin: 3e-6. No single value may be off by more than 1e-4
of the largest (rounding is spread over all of them; a wrong halo value is not)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [(2, 2, (140, 141)), (2, 3, (100, 99)), (2, 4, (99, 100)), (2, 5, (72, 70)), (3, 2, (16, 15, 14)),
         (3, 3, (12, 12, 12)), (2, 2, (24, 23)), (2, 4, (13, 12)), (2, 5, (17, 16)), (3, 2, (5, 4, 4)), (3, 3, (4, 4, 3))]
NT, MOVES = 20, 4


def _mesh(dim, grid):
    from synth import meshes
    V, C = meshes.structured_tri(*grid, *[0.1 * g for g in grid]) if dim == 2 else meshes.kuhn_tets(
        *[0.1 * np.arange(g + 1) for g in grid])
    L = 0.1 * np.array(grid)
    inner = np.all((V > 1e-9) & (V < L - 1e-9), axis=1)
    V = V.copy()
    V[inner] += np.random.default_rng(sum(grid)).uniform(-0.01, 0.01, (inner.sum(), dim))
    return V, C, L


def _rough(x):
    return 2.2 + 0.8 * np.sin(991.0 * x[:, 0] + 577.0 * x[:, -1]) * np.cos(757.0 * x[:, 1] + 1.0)


@pytest.mark.parametrize("S", [1, 2, 4, 8])
@pytest.mark.parametrize("dim,k,grid", CASES)
def test_rough_velocity_matches_plain(dim, k, grid, S):
    import torch

    import paper_2108_10946_gb300 as pkg
    from synth import signals
    pkg.build()
    V, C, L = _mesh(dim, grid)
    box = [(0.1, l - 0.1) for l in L[:-1]] + [(-1.0, L[-1] - 0.1)]
    rng = np.random.default_rng(100 * k + S)
    recs = rng.uniform(0.02, 0.98, (48, dim)) * L
    at = [rng.choice(len(recs), S, replace=False) for _ in range(MOVES)]
    srcs = [np.clip(recs[i] + rng.uniform(-0.03, 0.03, (S, dim)), 1e-6, L - 1e-6) for i in at]
    obs = torch.from_numpy(rng.standard_normal((S, NT + 1, len(recs))).astype(np.float32)).cuda()
    dt, out, res = 0.0, {}, []
    for layout in (0, 1):
        m = pkg.Mesh(V, C, k, NT, dt=dt, cfl_factor=0.7, box=box, layer_faces=0b1011 if dim == 2 else 0b101111,
                     layer_width=0.1, sigma_max=signals.sigma_max(3.0, 0.1), absorbing=True, ckpt_stride=8,
                     water_speed=1.6, layout=layout)
        x = m.dof_coords()
        m.set_velocity(_rough(x))
        dt = dt or m.dt
        order = np.lexsort(np.round(x / L / 1e-7).T)
        wav = np.stack([signals.ricker_samples(2.0 / (NT * dt), dt, NT, t0=(0.3 + 0.02 * s) * NT * dt) for s in range(S)])
        wav = torch.from_numpy(wav.astype(np.float32)).cuda()
        b = pkg.Batch(m, srcs[0], recs)
        b.set_gradient_lanes(True)
        rec = torch.zeros((S, NT + 1, len(recs)), device="cuda")
        g = torch.zeros((S, m.N), dtype=torch.float64, device="cuda")
        out[layout] = []
        for i, s in enumerate(srcs):
            b.set_sources(s)
            b.forward(wav, rec)
            if layout == 0:
                res.append(rec - 0.1 * rec.abs().max() * obs)
            b.adjoint(res[i])
            b.gradient_lanes(g)
            out[layout].append((rec.double().cpu().numpy(), g.cpu().numpy()[:, order]))
        b.close()
        m.close()
    for move, (got, want) in enumerate(zip(out[0], out[1])):
        for name, a, w in zip(("records", "gradient"), got, want):
            norm, most = np.linalg.norm(a - w) / np.linalg.norm(w), np.abs(a - w).max() / np.abs(w).max()
            print(f"move {move}: {name} norm {norm:.2e}, largest {most:.2e}")
            assert np.any(w != 0) and norm < 3e-6 and most < 1e-4, name
