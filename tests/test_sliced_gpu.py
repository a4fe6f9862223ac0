"""FP64 translations from exact slices: every pipeline shape (one stage, a partial stage, one
accumulator chunk of 512 columns, two, three), extreme scales, and values that are not finite.

Tolerance: slices round each input once to 2^-56 of its vector's largest entry, and what
follows amplifies that by at most the pseudo-inverse's 1 / cut = 1e9: 1e9 * 2^-55 = 2.8e-8.
A lost slice would be 128 times that."""
import numpy as np
import pytest
import torch

import synth
from oracle.quadrature import quadrature_points
from paper_1605_01715_gb300 import Plan, Tree

pytestmark = pytest.mark.gpu
TOL = 3e-8


def _plan(kernel, precision, p):
    mesh = synth.geodesic_sphere(11)
    xyz, w, nrm = quadrature_points(mesh.tri, mesh.sph)
    xyz, nrm = (torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (xyz, nrm))
    plan = Plan(Tree(xyz, max_leaf=24), kernel=kernel, p=p, precision=precision, src_nrm=nrm, trg_nrm=nrm)
    return plan, mesh.n, torch.from_numpy(w).cuda()


@pytest.mark.parametrize("kernel,precision,p", [
    ("sl", "fp64", 2), ("sl", "fp64", 4), ("dl", "fp64", 10), ("sl", "fp64", 12), ("adl", "fp64", 16),
    ("sl", "cheb_fp64", 2), ("dl", "cheb_fp64", 5), ("sl", "cheb_fp64", 8),
])
def test_linear_and_scaled(kernel, precision, p):
    plan, n, w = _plan(kernel, precision, p)
    a = torch.from_numpy(synth.uniform_density(n, 1)).cuda() * w
    b = torch.from_numpy(synth.uniform_density(n, 2)).cuda() * w * 1e-3
    fa, fb, fab = plan.matvec(a), plan.matvec(b), plan.matvec(a + b)
    plan.check()
    assert float((fab - fa - fb).norm() / fab.norm()) < TOL
    for s in (2.0 ** -600, 2.0 ** 600):
        assert float((plan.matvec(a * s) / s - fa).norm() / fa.norm()) < TOL


@pytest.mark.parametrize("precision", ["fp64", "cheb_fp64"])
@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_not_finite_stays_not_finite(precision, bad):
    plan, n, w = _plan("sl", precision, 4)
    q = w.clone()
    q[n // 3] = bad
    out = plan.matvec(q)
    plan.check()
    fin = torch.isfinite(out)
    fin[n // 3] = False                        # the point's own pair is excluded: it may stay finite
    assert not bool(fin.any())
    assert bool(torch.isfinite(plan.matvec(w)).all())
