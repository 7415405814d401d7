"""Every tile and occupancy that the ensemble's autotuner may pick gives each mesh
the result of a run of its own. The choice is forced through the tuning cache, a
text file of "<key>\\t<candidate>" lines that a new context reads instead of timing
the candidates."""
import numpy as np
import pytest
import torch

import paper_1211_0582_gb300 as dg
import workloads as W

pytestmark = pytest.mark.gpu

# sizes of the meshes (n^3 x 6 tets): uneven, and together more elements than a round of the smallest candidate
# on half of the blocks, so that its blocks loop over full tiles and a spread remainder
SIZES = {1: (13, 9, 11), 2: (11, 8, 9), 3: (11, 8, 9), 4: (9, 7, 8), 5: (8, 5, 7), 6: (7, 4, 6), 7: (6, 4, 5),
         8: (5, 4, 6), 9: (4, 5, 3)}


@pytest.mark.parametrize("N", range(1, 10))
def test_every_candidate_matches_separate_runs(N, tmp_path, monkeypatch):
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("DGMX_TUNE_CACHE", str(cache))
    meshes, eps, dts, alone = [], [], [], []
    for i, n in enumerate(SIZES[N]):
        mesh = W.kuhn_cube(n, jitter=0.1, seed=10 + i)
        meshes.append(mesh)
        eps.append(W.element_eps(mesh[3].shape[0], seed=100 + i))
        dts.append(0.2 / n / max(N * N, 2.5))
        s = dg.Solver(N).upload(*mesh, eps=eps[-1])
        x, y, z = s.node_coords()
        u0 = s.to_device(W.gaussian_pulse(x, y, z, seed=7, index=i) + 0.1 * W.cavity_mode(x, y, z, 0.0))
        u, r = u0.clone(), s.zeros()
        s.step(u, r, dts[-1], 2)
        alone.append((u0, u))
    start = torch.cat([u0 for u0, _ in alone], dim=1).contiguous()

    def advance():
        ens = dg.Solver(N).upload_ensemble(meshes, eps, dts)
        u, res = start.clone(), torch.zeros_like(start)
        ens.ensemble_step(u, res, 2)
        ens.sync()
        return ens, u, ens.ensemble_tuning_grid()

    advance()  # tunes and writes the cache
    key = cache.read_text().splitlines()[-1].rpartition("\t")[0]
    for candidate in range(8):
        cache.write_text(f"{key}\t{candidate}\n")
        ens, u, (best, eb, _, ms) = advance()
        assert best == candidate and max(ms) == 0  # taken from the cache, not timed
        off = ens.ensemble_layout()
        for i, (_, ref) in enumerate(alone):
            err = float((u[:, off[i]:off[i + 1]] - ref).norm() / ref.norm())
            assert err < 1e-6, (candidate, eb[candidate], i, err)
        assert not u[:, :, ens.Np:].any()
