"""The chunked layout's kernels (derivatives in symmetry-adapted coordinates) against the plain
layout's (dense derivative matrices, global atomics) on the same inputs, at the sizes where chunks,
shot groups and launches change form: a few elements (one short chunk, steps run inside one
launch), just past the size from which chunks hold their most elements (a short last chunk), both
kinds of chunks in one launch, and every group of shots. Per-step launches (forced by the profile
switch) against steps inside one launch as well.

Tolerance: each form is held within 1e-5 (records) and 1e-4 (gradients) of the FP64 oracle elsewhere
in this suite, so two of them differ by at most twice that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# dim, k, grid, shots, whether the steps fit one launch
CASES = [(2, 2, (5, 3), 1, True), (2, 2, (140, 141), 4, False), (2, 3, (7, 5), 8, True),
         (2, 3, (100, 99), 2, False), (2, 4, (6, 5), 2, True), (2, 4, (99, 99), 4, False),
         (2, 5, (5, 5), 4, True), (2, 5, (72, 70), 1, False), (3, 2, (3, 3, 2), 2, True),
         (3, 2, (16, 15, 14), 1, False), (3, 3, (4, 3, 3), 4, True), (3, 3, (12, 12, 12), 2, False)]


def _mesh(dim, grid):
    from synth import meshes
    rng = np.random.default_rng(sum(grid))
    if dim == 2:
        V, C = meshes.structured_tri(*grid, *[0.1 * g for g in grid])
    else:
        V, C = meshes.kuhn_tets(*[0.1 * np.arange(g + 1) for g in grid])
    inner = np.all((V > 1e-9) & (V < 0.1 * np.array(grid) - 1e-9), axis=1)
    V = V.copy()
    V[inner] += rng.uniform(-0.01, 0.01, (inner.sum(), dim))
    return V, C


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dim,k,grid,S,one_launch", CASES)
def test_chunked_forms_match_plain(dim, k, grid, S, one_launch):
    import torch

    import paper_2108_10946_gb300 as pkg
    from synth import signals
    pkg.build()
    V, C = _mesh(dim, grid)
    L = 0.1 * np.array(grid)
    nt, ckpt = 24, 7
    box = [(0.1, l - 0.1) for l in L[:-1]] + [(-1.0, L[-1] - 0.1)]
    faces = 0b1011 if dim == 2 else 0b101111
    rng = np.random.default_rng(7)
    srcs = rng.uniform(0.3, 0.7, (S, dim)) * L
    recs = np.concatenate([srcs[:1] + 1e-3, rng.uniform(0.05, 0.95, (12, dim)) * L])
    dt = None
    out = {}
    for form in ("plain", "chunked", "steps"):
        m = pkg.Mesh(V, C, k, nt, dt=dt or 0.0, cfl_factor=0.7, box=box, layer_faces=faces, layer_width=0.1,
                     sigma_max=signals.sigma_max(3.0, 0.1), absorbing=True, ckpt_stride=ckpt, water_speed=1.55,
                     layout=1 if form == "plain" else 0)
        x = m.dof_coords()
        m.set_velocity(1.5 + 1.5 * x[:, -1] / L[-1])
        dt = dt or m.dt
        w = np.stack([signals.ricker_samples(2.0 / (nt * dt), dt, nt, t0=(0.3 + 0.02 * s) * nt * dt) for s in range(S)])
        obs = torch.from_numpy(np.random.default_rng(3).standard_normal((S, nt + 1, len(recs))).astype(np.float32)).cuda()
        b = pkg.Batch(m, srcs, recs)
        b.set_gradient_lanes(True)
        b.profile(form == "steps")
        rec = torch.zeros((S, nt + 1, len(recs)), device="cuda")
        pkg.launch_count()
        b.forward(torch.from_numpy(w).cuda(), rec)
        launches = pkg.launch_count()
        if form == "chunked":  # a launch per checkpoint, or one or two and the halo's per step; the last records
            assert launches == -(-nt // ckpt) + 1 if one_launch else launches >= 2 * nt + 1
        b.adjoint_misfit(obs)
        g = torch.zeros((S, m.N), dtype=torch.float64, device="cuda")
        J = b.gradient_lanes(g)
        order = np.lexsort(np.round(x / L / 1e-7).T)
        out[form] = (rec.cpu().numpy(), g.cpu().numpy()[:, order], J)
        b.close()
        m.close()
    for form in ("chunked", "steps"):
        assert _rel(out[form][0], out["plain"][0]) < 2e-5
        assert _rel(out[form][1], out["plain"][1]) < 2e-4
        assert np.allclose(out[form][2], out["plain"][2], rtol=2e-5)
    assert np.any(out["plain"][1] != 0)
