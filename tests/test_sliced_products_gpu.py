"""The sliced FP64 products piece by piece, against extended precision on the host."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
LD = np.longdouble
U = LD(2) ** -53


def _surface(p):
    """The points of a p x p x p grid on the surface of the unit cube."""
    g = np.linspace(-1.0, 1.0, p)
    x = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    return np.ascontiguousarray(x[(np.abs(x) == 1.0).any(1)])


def _probe():
    import device_probe
    lib = device_probe.lib()
    par = (ctypes.c_int * 3)()
    lib.probe_slice_params(par)
    return lib, par[0], par[1], par[2]


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _p(t):
    return ctypes.c_void_p(0 if t is None else t.data_ptr())


@pytest.mark.parametrize("p", [2, 3, 6, 8, 10, 11, 12, 16])      # 8 to 1,352 points: every register form
@pytest.mark.parametrize("what", ["sl", "adl", "field"])
def test_evaluation_values(p, what):
    """1/r and n.(x - y)/r^3 of targets in boxes of several sizes, out of their digits.  With u =
    2^-53, r >= 1.95 and |x| <= 1: x - y is off by u (|x| + |x - y|), so r^2 by 6.8 u and 1/r,
    with rsqrt's one unit in the last place, by 5.4 u; the gradient by 25 u / r^2.  Fixed point
    rounds once more, to half a unit of 2^(e - bits)."""
    lib, slices, bits, _ = _probe()
    rng = np.random.default_rng(p)
    n, lvl = 37, np.array([0, 1, 3, 9], np.int32)
    root_h = 1.5
    ctr = rng.uniform(-1, 1, (4, 3))
    leaf = rng.integers(0, 4, n).astype(np.int32)
    half = root_h * 2.0 ** -lvl[leaf]
    x = rng.uniform(-1, 1, (n, 3))
    x[:8] = np.sign(x[:8])                          # corners of the box
    t = ctr[leaf] + x * half[:, None]
    nrm = rng.normal(size=(n, 3))
    nrm /= np.linalg.norm(nrm, axis=1, keepdims=True)
    y = 2.95 * _surface(p)
    Q, Kc = len(y), -(-len(y) // 32) * 32
    sl = torch.zeros(n * Kc * slices, dtype=torch.float16, device="cuda")
    exps = torch.zeros(n, dtype=torch.int32, device="cuda")
    osc = torch.zeros(n, dtype=torch.float64, device="cuda")
    keep = [_dev(a) for a in (leaf, t.T, nrm.T, lvl, ctr, y)]
    dl, dt, dn, dv, dc, dy = keep
    assert lib.probe_eval_rows(_p(dl), n, _p(dt), _p(dn if what == "adl" else None), 1 if what == "field" else 0, _p(dv), _p(dc),
                               ctypes.c_double(root_h), _p(dy), Q, int(what != "sl"), _p(sl), _p(exps), _p(osc)) == 0
    digits = sl.cpu().numpy().astype(LD).reshape(n, Kc // 32, slices, 32)
    assert np.abs(digits).max() <= 64
    got = sum(digits[:, :, s] * LD(128) ** (slices - 1 - s) for s in range(slices)).reshape(n, Kc)
    e = exps.cpu().numpy()
    got = got * LD(2) ** (e.astype(LD)[:, None] - bits)
    assert (got[:, Q:] == 0).all()
    d = ((t.astype(LD) - ctr[leaf].astype(LD)) / half[:, None].astype(LD))[:, None] - y.astype(LD)[None]
    inv = 1 / np.sqrt((d ** 2).sum(-1))
    unit = LD(2) ** (e.astype(LD)[:, None] - bits - 1)
    if what == "sl":
        want, tol = inv, 5.4 * U * inv + unit
    else:
        nv = nrm.astype(LD) if what == "adl" else np.broadcast_to(LD([0, 1, 0]), (n, 3))
        want, tol = (d * nv[:, None]).sum(-1) * inv ** 3, 25 * U * inv ** 2 + unit
    err = np.abs(got[:, :Q] - want)
    print("%s p=%d worst error / bound %.2f" % (what, p, float((err / tol).max())))
    assert (err <= tol).all()
    assert (osc.cpu().numpy() == (1.0 if what == "sl" else 1.0 / half)).all()
