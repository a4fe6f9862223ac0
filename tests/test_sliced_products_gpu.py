"""The sliced FP64 products piece by piece, against extended precision on the host."""
import ctypes
import functools
from fractions import Fraction

import numpy as np
import pytest
import torch

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


@pytest.mark.gpu
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


# ---------------------------------------------------------------- products
SLICES, BITS = 9, 62


def _low_digits(rng, shape, down):
    """Doubles below 2^62 whose base-128 digits are all 40 to 63 as far as their 53 bits go, to the
    eighth of nine; moved down by two digits, to the last."""
    n = np.zeros(shape, dtype=object)
    for _ in range(SLICES):
        n = n * 128 + rng.integers(40, 64, shape)
    return (n // 2 ** 14 if down else n // 2 ** 10 * 2 ** 10).astype(np.float64)


def _cancelling(rng, M, N, K, down):
    """Operator rows and vectors (one of them moved down, or neither) whose products cancel to 2^-40 of
    their terms, so that the sum's own rounding hides nothing: the second half of a row is a power
    of two, and the vectors' entries there take back the first half's products but for their low digits."""
    h = (K - 1) // 2
    a, b = np.zeros((M, K)), np.zeros((N, K))
    a[:, :h], b[:, :h] = _low_digits(rng, (1, h), down == "rows"), _low_digits(rng, (N, h), down == "vectors")
    a[:, h:2 * h] = 2.0 ** 61
    b[:, h:2 * h] = -np.rint(a[0, :h] * b[:, :h] / 2.0 ** 82) * 2.0 ** 21
    b[:, K - 1] = 2.0 ** 61                         # times 0: the vectors' scale
    return a * 2.0 ** rng.integers(-40, 40, (M, 1)), b * 2.0 ** rng.integers(-40, 40, (N, 1))


CANCELLING = [functools.partial(_cancelling, down=d) for d in ("rows", "vectors", "neither")]


def _dense(rng, M, N, K):
    return rng.normal(size=(M, K)) * 2.0 ** rng.integers(-12, 1, (M, K)), rng.normal(size=(N, K)) * 2.0 ** rng.integers(-12, 1, (N, K))


def _bound(a, b, exact, chunks):
    """For |a| < 2^ea, |b| < 2^eb by row: rounding both to 62 bits leaves 2^-62 of 2^(ea + eb) a column,
    the eight digit products with i + j = 9 and all below them 8 x 2^12 x 128^7 x 1.008 / 2^124 =
    1.008 x 2^-60: 1.26 x 2^-60 in all.  Each chunk of columns and each sum of chunks rounds once."""
    top = LD(2) ** (np.frexp(np.abs(a).max(1))[1][None, :] + np.frexp(np.abs(b).max(1))[1][:, None])
    return a.shape[1] * LD(1.26) * LD(2) ** -60 * top + 2 * U * sum(np.abs(c) for c in chunks) + 2 * U * np.abs(exact)


def _exact(a, b, step=10 ** 9):
    chunks = [b[:, k:k + step].astype(LD) @ a[:, k:k + step].astype(LD).T for k in range(0, a.shape[1], step)]
    return sum(chunks), chunks


def _digits(x):
    """A row's digits, as Python integers, and its exponent."""
    e = np.frexp(np.abs(x).max(1))[1]
    y = np.array([[round(Fraction(v) * Fraction(2) ** (BITS - int(ei))) for v in row] for row, ei in zip(x, e)], dtype=object)
    d = []
    for _ in range(SLICES - 1):
        r = (y + 64) % 128 - 64
        d.append(r)
        y = (y - r) // 128
    return [y] + d[::-1], e


def test_bound_tells_a_lost_product():
    """The digits multiplied on the host: within the bound when complete, beyond it for one of the
    inputs below without any one of the slice products that count (i + j <= 8)."""
    seen = set()
    for make in CANCELLING:
        a, b = make(np.random.default_rng(5), 3, 4, 33)
        exact, chunks = _exact(a, b)
        bound = _bound(a, b, exact, chunks)
        (da, ea), (db, eb) = _digits(a), _digits(b)
        prod = {(i, j): db[j].dot(da[i].T) * 128 ** (2 * (SLICES - 1) - i - j) for i in range(SLICES) for j in range(SLICES)}
        sh = LD(2) ** (ea[None, :] + eb[:, None] - 2 * BITS).astype(LD)
        missing = sum(v for (i, j), v in prod.items() if i + j >= SLICES)
        assert (np.abs(missing.astype(LD)) * sh <= bound).all()
        for ij in prod:
            if sum(ij) < SLICES and (np.abs((missing + prod[ij]).astype(LD)) * sh > bound).any():
                seen.add(ij)
    assert len(seen) == SLICES * (SLICES + 1) // 2, sorted(seen)


def _product(a_ops, b, M, tiles_of, oscale=None, ostride=None):
    """a_ops (ops, Mr, K) by vectors b (n, K) over pairs tiles_of = [(op, vectors, outputs)]."""
    lib, slices, bits, pairs = _probe()
    nops, Mr, K = a_ops.shape
    tiles, pin, pout = [], [], []
    for op, src, dst in tiles_of:
        for c in range(0, len(src), pairs):
            n = min(pairs, len(src) - c)
            tiles += [op, len(pin), n, 0]
            pin += list(src[c:c + n])
            pout += list(dst[c:c + n])
    nout, stride = max(pout) + 1, ostride or M
    out = torch.zeros((nout, stride), dtype=torch.float64 if oscale is None else torch.float32, device="cuda")
    if oscale is not None:
        out += 7.0                                   # stores overwrite, to the padding too
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    da, db = _dev(a_ops), _dev(b)
    di, do = _dev(np.array(pin, np.int32)), _dev(np.array(pout, np.int32))
    ds = None if oscale is None else _dev(oscale)
    ht = (ctypes.c_int * len(tiles))(*tiles)
    torch.cuda.synchronize()
    assert lib.probe_sliced_product(_p(da), nops, Mr, K, K, M, _p(db), len(b), K, ht, len(tiles) // 4, _p(di), _p(do), _p(out),
                                    stride, _p(ds), _p(err)) == 0
    assert int(err) == 0
    return out.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("make", CANCELLING + [_dense], ids=["rows", "vectors", "neither", "dense"])
@pytest.mark.parametrize("K,M,n", [(8, 5, 1), (32, 128, 47), (33, 129, 48), (448, 16, 49), (449, 130, 97), (512, 256, 48),
                                   (513, 1, 63), (1352, 253, 64)])
def test_product_is_exact_to_its_bound(make, K, M, n):
    rng = np.random.default_rng(K)
    a, b = make(rng, M, n, K)
    got = _product(a[None], b, M, [(0, np.arange(n), np.arange(n))])
    exact, chunks = _exact(a, b, 512)
    err, bound = np.abs(got - exact), _bound(a, b, exact, chunks)
    print("K=%d M=%d n=%d worst error / bound %.3f" % (K, M, n, float((err / bound).max())))
    assert (err <= bound).all()


@pytest.mark.gpu
def test_operators_outputs_and_stores():
    """Several operators with padded rows, several pairs into one output, and the stored form with its
    scale and padding."""
    rng = np.random.default_rng(3)
    M, Mr, K, n = 130, 144, 96, 53
    a = np.zeros((3, Mr, K))
    a[:, :M], b = rng.normal(size=(3, M, K)), rng.normal(size=(n, K))
    pairs = [(op, rng.integers(0, n, 70), rng.permutation(80)[:70]) for op in range(3)]
    got = _product(a, b, M, pairs)
    want, bound = np.zeros(got.shape, LD), np.zeros(got.shape, LD)
    for op, src, dst in pairs:
        e, c = _exact(a[op, :M], b[src])
        want[dst] += e
        bound[dst] += _bound(a[op, :M], b[src], e, c) + 3 * U * np.abs(e)      # the outputs' own sums
    assert (np.abs(got - want) <= bound).all()
    scale = 2.0 ** rng.integers(-3, 3, n) * 1.5
    got = _product(a, b, M, [(1, np.arange(n), np.arange(n))], oscale=scale, ostride=Mr)
    e, c = _exact(a[1, :M], b)
    assert (np.abs(got[:, :M] - e * scale[:, None]) <= _bound(a[1, :M], b, e, c) * scale[:, None]
            + LD(2) ** -24 * np.abs(e * scale[:, None]) * (1 + LD(2) ** -20)).all()
    assert (got[:, M:] == 0).all()


def _kernel_matrix(x, y):
    return 1.0 / np.sqrt(((x[:, None] - y[None]) ** 2).sum(-1))


def _pinv(A, cut):
    u, s, vt = np.linalg.svd(A)
    k = s > cut * s[0]
    return (vt[k].T / s[k]) @ u[:, k].T


def _in_order(a, b):
    """FP64 fused multiply-adds, one column after the other."""
    acc = np.zeros((len(b), len(a)))
    for k in range(a.shape[1]):
        acc = (b[:, k:k + 1].astype(LD) * a[:, k].astype(LD)[None] + acc.astype(LD)).astype(np.float64)
    return acc


@pytest.mark.gpu
@pytest.mark.parametrize("p", [4, 6, 8, 10])
@pytest.mark.parametrize("kernel", ["sl", "dl"])
def test_no_less_accurate_than_fp64(kernel, p):
    """The method's own operators (rows of very uneven entries) on check potentials of random sources:
    no larger an error than FP64 fused multiply-adds make.  (Eight slices made one 22 times as large
    for the neighbouring boxes of the double layer at p = 6.)"""
    rng = np.random.default_rng(p)
    s = _surface(p)
    y, q = rng.uniform(-1, 1, (24, 64, 3)), rng.uniform(-1, 1, (24, 64))
    d = 2.95 * s[None, :, None] - y[:, None]
    r = np.sqrt((d ** 2).sum(-1))
    nrm = rng.normal(size=(24, 1, 64, 3))
    up = ((1 / r if kernel == "sl" else (d * nrm).sum(-1) / r ** 3) * q[:, None]).sum(-1)
    pu = _pinv(_kernel_matrix(2.95 * s, 1.05 * s), 1e-9)
    pd = _pinv(_kernel_matrix(1.05 * s, 2.95 * s), 1e-9)
    child = np.array([0.5, -0.5, 0.5])
    far = _kernel_matrix(1.05 * s, 2.0 * np.array([2, 0, 0]) + 1.05 * s) @ pu
    dn = (up.astype(LD) @ far.astype(LD).T).astype(np.float64)
    for name, a, b in (("up to parent", 0.5 * _kernel_matrix(2.95 * s, child + 0.525 * s) @ pu, up),
                       ("neighbour", far, up), ("neighbour, mean removed", far - far.mean(0), up),
                       ("down to child", _kernel_matrix(child + 0.525 * s, 2.95 * s) @ pd, dn)):
        want, _ = _exact(a, b)
        got = _product(a[None], b, len(s), [(0, np.arange(24), np.arange(24))])
        norm = np.sqrt((want ** 2).sum(1, keepdims=True))
        mine, fp64 = (float(np.sqrt((((x - want) / norm) ** 2).sum(1).mean())) for x in (got, _in_order(a, b)))
        print("%s p=%d %s: sliced %.1e, FP64 in order %.1e" % (kernel, p, name, mine, fp64))
        assert mine <= fp64
