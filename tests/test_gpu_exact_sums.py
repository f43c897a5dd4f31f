"""One dot, one update and one block product of the fixed-point Gram-Schmidt against exact sums.

The vectors are graded (entries over 2^40 within a tile), their components stand in units 2^34
apart, and the components' lengths are no multiples of a tile.  The reference adds the exact
products (each split into a rounded product and its error) with math.fsum.

Bounds, per component where the result has components, with u = 2^-53:
* a dot rounds both factors to 2^-59 of their tile's largest entry and drops the products of the low
  halves (at most 2^-58 of the two largest, of either sign): 4 u |v| |w| summed over the components;
* an update of r rows also rounds each coefficient and drops low products, 4 r terms of at most
  d = 2^(h - 57) M, M the largest |coefficient| |entry| of a row and h the bits the coefficients give
  up (2 up to 32 rows, 3 above; block kernels: as many as r / 8 needs, at least 2).  They are independent
  and of either sign: six times their r.m.s. sqrt(4 r / 3) d, and u (|sum| + |w|) twice for rounding.
A product of a high and a low half that is wrong or missing errs by 2^-30 instead."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA not available", allow_module_level=True)

import paper_2411_15897_gb300 as bah  # noqa: E402
from paper_2411_15897_gb300 import _build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
U = 2.0 ** -53


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    bah.lib()
    out = str(tmp_path_factory.mktemp("gs") / "libgs_sums.so")
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", "-cudart", "shared", "-I", _build.CSRC, "-o", out,
                    os.path.join(HERE, "gs_sums.cu"), "-L", _build.LIBDIR, "-lbah", "-Xlinker", "-rpath=" + _build.LIBDIR],
                   check=True, timeout=300)
    return ctypes.CDLL(out)


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def graded(rng, count, nc, ncomp, unit=2.0 ** -34):
    g = lambda: rng.standard_normal((count, ncomp, nc)) * 2.0 ** (-40 * rng.uniform(size=(count, ncomp, nc)))
    v = g() + 1j * g()
    v[:, -1] *= unit
    return v


def split(a):
    t = 134217729.0 * a
    h = t - (t - a)
    return h, a - h


def two_prod(a, b):
    """a b as a rounded product and its exact error (Dekker)."""
    p = a * b
    ah, al = split(a)
    bh, bl = split(b)
    return p, ((ah * bh - p) + ah * bl + al * bh) + al * bl


def exact_dot(v, w):
    re = [x.ravel() for a, b in ((v.real, w.real), (v.imag, w.imag)) for x in two_prod(a, b)]
    im = [x.ravel() for a, b in ((v.real, w.imag), (-v.imag, w.real)) for x in two_prod(a, b)]
    return complex(math.fsum(np.concatenate(re)), math.fsum(np.concatenate(im)))


def exact_minus(w, V, c):
    """w - sum_i c_i V_i, every entry rounded once (V: rows x n)."""
    c = c[:, None]
    re = [x for a, b in ((-c.real, V.real), (c.imag, V.imag)) for x in two_prod(a + 0 * b, b)]
    im = [x for a, b in ((-c.real, V.imag), (-c.imag, V.real)) for x in two_prod(a + 0 * b, b)]
    re, im = np.concatenate([w.real[None]] + re), np.concatenate([w.imag[None]] + im)
    return np.array([complex(math.fsum(re[:, e]), math.fsum(im[:, e])) for e in range(w.size)])


def norms(v):
    return np.sqrt((np.abs(v) ** 2).sum(-1))          # per component


def update_bound(w, V, c, exact, rows, head):
    """Per component; w, exact: (ncomp, nc), V: (rows, ncomp, nc), c: (rows,)"""
    big = lambda z: np.maximum(np.abs(z.real), np.abs(z.imag)).max(-1)
    M = (np.maximum(np.abs(c.real), np.abs(c.imag))[:, None] * big(V)).max(0)
    return 6 * math.sqrt(4 * rows / 3) * 2.0 ** (head - 57) * M + 2 * U * (2 * big(w) + big(exact))


@pytest.mark.parametrize("nc,ncomp,k", [(400, 3, 1), (400, 3, 2), (400, 3, 7), (100, 3, 20), (700, 4, 33), (300, 1, 64),
                                        (28000, 3, 3), (60000, 3, 2)])
def test_dot_and_update(lib, nc, ncomp, k):
    rng = np.random.default_rng(1000 * k + nc)
    V, w = graded(rng, k, nc, ncomp), graded(rng, 1, nc, ncomp)[0]
    c = rng.standard_normal(k) + 1j * rng.standard_normal(k)
    n = ncomp * nc
    d_v, d_w, d_out = dev(V), dev(w), dev(np.zeros(k + 1, np.complex128))
    d_c, d_nm = dev(np.append(c, norms(w.ravel()) ** 2)), dev(np.zeros(1))
    assert lib.gs_pass(ptr(d_v), k, ptr(d_w), ctypes.c_longlong(n), ctypes.c_longlong(nc), ptr(d_out), ptr(d_c), ptr(d_nm)) == 0
    out, got = d_out.cpu().numpy(), d_w.cpu().numpy()
    for i in range(k):
        assert abs(out[i] - exact_dot(V[i], w)) <= 4 * U * (norms(V[i]) * norms(w)).sum(), i
    w2 = exact_dot(w, w).real
    assert abs(out[k] - w2) <= 4 * U * w2
    some = slice(None) if n <= 3000 else slice(0, None, 37)
    flat = lambda a: a.reshape(a.shape[:-2] + (-1,))[..., some]
    ref = exact_minus(flat(w), flat(V), c)
    b = np.repeat(update_bound(w, V, c, got, k, 2 if k <= 32 else 3), nc)[some]
    err = flat(got) - ref
    assert (np.maximum(np.abs(err.real), np.abs(err.imag)) <= b).all(), (np.abs(err) / b).max()
    assert abs(d_nm.item() - np.linalg.norm(got)) <= 1e-13 * np.linalg.norm(got)


@pytest.mark.parametrize("nc,ncomp,k,s", [(60, 3, 1, 2), (400, 3, 3, 5), (400, 3, 2, 8), (300, 3, 4, 9), (90, 3, 20, 16),
                                          (700, 3, 9, 8)])
def test_block_products(lib, nc, ncomp, k, s):
    rng = np.random.default_rng(100 * k + s)
    V, W = graded(rng, k * s, nc, ncomp), graded(rng, s, nc, ncomp)
    cplx = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    T, Y = np.triu(cplx(s, s)), cplx(k * s, s)
    n = ncomp * nc
    d = [dev(a) for a in (V, W, np.zeros((k * s, s), np.complex128), np.zeros((s, s), np.complex128), T, np.zeros_like(W), Y)]
    assert lib.block_products(ptr(d[0]), k, s, ptr(d[1]), ctypes.c_longlong(n), ctypes.c_longlong(nc),
                              *(ptr(t) for t in d[2:])) == 0
    got, C, G, W2 = (d[q].cpu().numpy() for q in (1, 2, 3, 5))
    rows = range(k * s) if k * s <= 40 else rng.choice(k * s, 40, replace=False)
    for r in rows:
        for b in range(s):
            assert abs(C[r, b] - exact_dot(V[r], W[b])) <= 4 * U * (norms(V[r]) * norms(W[b])).sum(), (r, b)
    for a in range(s):
        for b in range(s):
            assert abs(G[a, b] - exact_dot(W[a], W[b])) <= 4 * U * (norms(W[a]) * norms(W[b])).sum(), (a, b)
    head = 2
    while (8 << head) < k * s:
        head += 1
    some = slice(None) if n <= 600 else slice(0, None, 3)
    flat = lambda a: a.reshape(a.shape[:-2] + (-1,))[..., some]
    for b in range(s):
        ref = exact_minus(flat(W[b]), flat(V), Y[:, b])
        bound = np.repeat(update_bound(W[b], V, Y[:, b], got[b], k * s, head), nc)[some]
        err = flat(got[b]) - ref
        assert (np.maximum(np.abs(err.real), np.abs(err.imag)) <= bound).all(), (b, (np.abs(err) / bound).max())
        zero = np.zeros(n, np.complex128).reshape(ncomp, nc)
        ref = -exact_minus(flat(zero), flat(W), T[:, b])
        bound = np.repeat(update_bound(zero, W, T[:, b], W2[b], s, 2), nc)[some]
        err = flat(W2[b]) - ref
        assert (np.maximum(np.abs(err.real), np.abs(err.imag)) <= bound).all(), ("scale", b, (np.abs(err) / bound).max())


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_nonfinite_entries_are_seen(lib, bad):
    nc, ncomp, k = 400, 3, 5
    rng = np.random.default_rng(5)
    n = ncomp * nc
    for where in ("w", "V"):
        V, w = graded(rng, k, nc, ncomp), graded(rng, 1, nc, ncomp)[0]
        if where == "w":
            w[1, 300] = bad                           # the second tile of the second component
        else:
            V[2, 1, 300] = bad
        d_v, d_w, d_out = dev(V), dev(w), dev(np.zeros(k + 1, np.complex128))
        d_c, d_nm = dev(np.ones(k + 1, np.complex128)), dev(np.zeros(1))
        assert lib.gs_pass(ptr(d_v), k, ptr(d_w), ctypes.c_longlong(n), ctypes.c_longlong(nc), ptr(d_out), ptr(d_c),
                           ptr(d_nm)) == 0
        out, got = d_out.cpu().numpy(), d_w.cpu().numpy()
        seen = ~np.isfinite(out)
        assert seen.tolist() == ([True] * (k + 1) if where == "w" else [i == 2 for i in range(k + 1)])
        tile = ~np.isfinite(got)
        assert tile[1, 300] and not tile[0].any() and not tile[2].any() and not tile[1, :256].any()
        assert not np.isfinite(d_nm.item())
