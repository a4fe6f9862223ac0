"""Passes of the warp near field: the width w (targets a lane, 8 w a pass) of the kernel's
widest, 4 and 2 that is cheapest by (4 + w) max(1, units / warps the chip holds); the widest for
two waves of units and more."""
import numpy as np
import pytest
import torch

import synth
from oracle.quadrature import quadrature_points
from paper_1605_01715_gb300 import Plan, Tree

pytestmark = pytest.mark.gpu
WIDEST = {"sl": 8, "dl": 6, "adl": 4, "field": 8}
UNIT_SOURCES = 2048


@pytest.mark.parametrize("kernel,p,freq,leaf", [
    ("sl", 6, 5, 40), ("dl", 10, 10, 64),           # every unit resident at w = 2
    ("dl", 10, 44, 192), ("dl", 10, 50, 160),       # leaves of several units
    ("dl", 10, 57, 96), ("adl", 11, 57, 96), ("sl", 6, 50, 64), ("field", 11, 44, 64),
    ("dl", 10, 85, 128), ("adl", 11, 85, 64),       # more than the chip holds at any width
])
def test_pass_width(kernel, p, freq, leaf):
    mesh = synth.geodesic_sphere(freq)
    xyz, w, nrm = (np.ascontiguousarray(a) for a in quadrature_points(mesh.tri, mesh.sph))
    xyz, nrm = torch.from_numpy(xyz).cuda(), torch.from_numpy(nrm).cuda()
    tree = Tree(xyz, max_leaf=leaf)
    plan = Plan(tree, kernel=kernel, p=p, precision="mixed", src_nrm=nrm, trg_nrm=nrm)
    t, q_points = tree.export(), 6 * (p - 1) ** 2 + 2
    n_src = t["range"][:, 1] - t["range"][:, 0]
    n_trg = t["range"][:, 3] - t["range"][:, 2]
    lists = {k: tree.list(k) for k in "UWX"}
    unit_targets = []                               # the target count of each unit's leaf
    for b in np.flatnonzero(t["leaf"] & (n_trg > 0)):
        src = sum(n_src[idx[off[b]:off[b + 1]]].sum() for k, (off, idx) in lists.items()
                  if k != "X" or n_trg[b] < q_points)
        unit_targets += [n_trg[b]] * max(1, -(-int(src) // UNIT_SOURCES))
    unit_targets = np.array(unit_targets)
    resident = 16 * torch.cuda.get_device_properties(0).multi_processor_count
    units = {w: int((-(-unit_targets // (8 * w))).sum()) for w in (WIDEST[kernel], 4, 2)}
    width = min(units, key=lambda w: (4 + w) * max(resident, units[w]))   # the first of equals
    if units[WIDEST[kernel]] >= 2 * resident:
        width = WIDEST[kernel]
    print(kernel, mesh.n, leaf, units, width)
    assert plan.stats()["near_units"] == units[width]
