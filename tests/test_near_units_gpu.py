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


@pytest.mark.parametrize("kernel,pairs,x_list,units,direct,captured", [
    # plans timed with and without (2,432 resident warps)
    ("dl", 3.6e6, 0, 628, True, True), ("sl", 11.1e6, 0, 2236, True, True), ("adl", 14.8e6, 1, 1348, True, True),
    ("sl", 30.7e6, 1, 2072, True, True), ("dl", 11.6e6, 0, 3248, True, True), ("sl", 23.5e6, 0, 5816, True, True),
    ("dl", 31.0e6, 0, 4864, True, False), ("sl", 32.6e6, 1, 4232, True, False), ("dl", 37.4e6, 0, 1784, True, False),
    ("dl", 17.2e6, 1, 4880, True, False), ("sl", 24.7e6, 1, 0, True, True), ("adl", 40.9e6, 1, 3546, True, False), ("sl", 77.2e6, 1, 2440, False, False),
    ("adl", 628.3e6, 1, 33792, False, False),
])
def test_early_launch_rule(kernel, pairs, x_list, units, direct, captured):
    import ctypes
    import device_probe
    from paper_1605_01715_gb300.capi import KERNELS
    f = device_probe.lib().probe_chain_early
    f.argtypes = [ctypes.c_int, ctypes.c_int, ctypes.c_longlong, ctypes.c_int, ctypes.c_longlong, ctypes.c_longlong]
    assert [bool(f(cap, KERNELS[kernel], int(pairs), x_list, units, 2432)) for cap in (0, 1)] == [direct, captured]
