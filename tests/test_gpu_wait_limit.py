"""A bounded wait of the chunk kernels that gives up: the call returns FWI_ETIMEDOUT, and the same
batch, with the default limit again, gives what it gave before.

With 0 polls the waits for a chunk's copies give up at once. With 1 poll the copies usually arrive
(the hardware suspends a poll until they do, or for a while) and the meetings of a launch of several
steps give up, after chunks have added sums for halo DoFs that nothing takes any more: what the
next call must not find. Nothing here faults or hangs: every wait ends, at the latest by its limit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


# the steps in one launch (r, P; in 3D omega), and one by one (past the most such a launch takes)
@pytest.mark.parametrize("dim,k,grid,limits", [(2, 3, (40, 39), (0, 1)), (3, 2, (8, 7, 7), (0, 1)), (2, 5, (72, 70), (0,))])
def test_batch_is_sound_after_a_wait_that_gave_up(dim, k, grid, limits):
    import torch

    import paper_2108_10946_gb300 as pkg
    from paper_2108_10946_gb300.lib import FWI_ETIMEDOUT, FwiError
    from synth import meshes, models, signals
    pkg.build()
    L = 0.1 * np.array(grid)
    V, C = meshes.structured_tri(*grid, *L) if dim == 2 else meshes.kuhn_tets(*[0.1 * np.arange(g + 1) for g in grid])
    nt, S = 24, 4
    m = pkg.Mesh(V, C, k, nt, cfl_factor=0.7, box=[(0.2, l - 0.2) for l in L[:-1]] + [(-1.0, L[-1] - 0.2)],
                 layer_faces=0b1011 if dim == 2 else 0b101111, layer_width=0.2, sigma_max=signals.sigma_max(3.0, 0.2),
                 absorbing=True, ckpt_stride=8)
    x = m.dof_coords()
    m.set_velocity((models.smooth2d if dim == 2 else models.smooth3d)(x / L))
    rng = np.random.default_rng(5)
    srcs = rng.uniform(0.05, 0.95, (S, dim)) * L  # in the layer, too
    recs = np.concatenate([srcs + 0.01 * (0.5 * L - srcs), rng.uniform(0.05, 0.95, (20, dim)) * L])
    wav = torch.from_numpy(np.stack([signals.ricker_samples(2.0 / (nt * m.dt), m.dt, nt, t0=0.3 * nt * m.dt)] * S)).float().cuda()
    b = pkg.Batch(m, srcs, recs)
    rec = torch.zeros((S, nt + 1, len(recs)), device="cuda")
    g = torch.zeros(m.N, dtype=torch.float64, device="cuda")
    b.forward(wav, rec)
    res = (0.1 * rec).contiguous()

    def solve():
        b.forward(wav, rec)
        r = rec.cpu().numpy().astype(float)
        b.adjoint(res)
        b.gradient(g)
        return r, g.cpu().numpy().copy()

    want = solve()
    for polls in limits:
        for call in ("forward", "adjoint"):
            b.forward(wav, rec)
            b.set_wait_limit(polls)
            with pytest.raises(FwiError, match="gave up") as ei:
                b.forward(wav, rec) if call == "forward" else b.adjoint(res)
            assert ei.value.code == FWI_ETIMEDOUT
            b.set_wait_limit(-1)
            b.gradient(g)  # clears the gradient accumulators
            got = solve()
            # the same computation; only the order of the atomic sums differs
            assert _rel(got[0], want[0]) < 1e-5 and _rel(got[1], want[1]) < 1e-5, (polls, call)
    b.close()
    m.close()
