"""Tensor-core translations at the edges of their tiles, against the FP64 form of the same
plan (CUDA-core GEMMs over whole check potentials, no tiles of this kind)."""
import numpy as np
import pytest
import torch

import synth
from oracle.quadrature import quadrature_points
from paper_1605_01715_gb300 import Plan, Tree

pytestmark = pytest.mark.gpu

# Both forms truncate alike (same p and cut), so they differ by the mixed form's rounding:
# each of the two meets 1e-6 of the exact sum on these meshes where p allows it, so their
# difference stays below the sum of the two.
TOL = 2e-6


@pytest.mark.parametrize("kernel,p,freq,leaf", [
    ("sl", 4, 3, 8),      # K <= 128: one slab by 256 columns; 180 points, tiles of one to a few pairs
    ("sl", 4, 23, 16),    # the same, tiles past 128 columns (both column halves)
    ("sl", 6, 7, 12),     # K = 160: the second slab's last quarters are empty
    ("sl", 8, 16, 20),    # K = 208, tiles of 16 to 128 columns
    ("dl", 10, 5, 8),     # up rank past 256: a second row group of one partial slab
    ("dl", 10, 20, 24),   # the same with full tiles
    ("adl", 11, 12, 16),  # K = 256
])
def test_mixed_translations_match_fp64(kernel, p, freq, leaf):
    mesh = synth.geodesic_sphere(freq)
    xyz_h, w_h, nrm_h = quadrature_points(mesh.tri, mesh.sph)
    xyz, nrm = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (xyz_h, nrm_h))
    q = torch.from_numpy(synth.uniform_density(mesh.n, 11) * w_h).cuda()
    tree = Tree(xyz, max_leaf=leaf)
    out = {}
    for prec in ("mixed", "fp64"):
        plan = Plan(tree, kernel=kernel, p=p, precision=prec, pinv_cutoff=1e-8, src_nrm=nrm, trg_nrm=nrm)
        out[prec] = plan.matvec(q)
        plan.check()
    err = float((out["mixed"] - out["fp64"]).norm() / out["fp64"].norm())
    print("%s p=%d n=%d rel-L2 %.3e" % (kernel, p, mesh.n, err))
    assert err < TOL
