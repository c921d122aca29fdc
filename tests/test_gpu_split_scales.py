"""Split-precision products scale by scale: a sum of one slice scale that is lost (or counted twice) in one exact chunk
of 256 stacked inner indices must show, for every layout with one accumulator per scale.

A system of three atoms in a row, two leaves of s orbitals around a separator of r: L = B A^{-1} (K = s), the Schur
update (K = s), T = G_RR L (K = r) and G_JJ = A^{-1} + L^T T (K = r) are the split products; every inverse stays on
the FP64 path (outer_block above the widths).  H has entries N(0, 1/n) and S = I, so that the spectrum is within
[-2, 2], cond(z S - H) <= 4 at Im z = 0.7, and the products' contributions are of the order of max|G|.

Limit.  The same elimination with the digits multiplied in FP64 on the host gives the error that cutting S digits and
leaving out the pairs t + u > S + 1 makes; the kernel differs from it by the rounding of the sums it reads out (2^-48 of
them), so eight times the model's error is allowed, and the FP64 parts have 20 sqrt(n) u cond (n <= 800: 2.5e-13).
The tail layouts lose the low bits of the scales that share an accumulator: 2^-38 (four) and 2^-43 (five) of a
product, 20 times that is added for them.  A scale of one chunk of one product left out is 100 times the model's
error or more; the model shows that it exceeds the limit for every scale of four, five and six slices.  Scale 6 of
seven slices lies below the FP64 parts' error and cannot show."""
import functools

import numpy as np
import pytest

from synth import csr_from_dense

Z = 0.3 + 0.7j
U = 2.0 ** -53


@functools.lru_cache(maxsize=None)
def matrices(s, r):
    rng = np.random.default_rng(1000 * s + r)
    n = 2 * s + r
    a = rng.normal(0, 1.0 / np.sqrt(n), (n, n))
    H = (a + a.T) / np.sqrt(2.0)
    H[:s, s + r:] = H[s + r:, :s] = 0.0
    return H, np.linalg.inv(Z * np.eye(n) - H)


def digits(x, S):
    """Balanced base-256 digits of the rows of x at a common exponent per row (real and imaginary parts)."""
    m = np.max(np.maximum(np.abs(x.real), np.abs(x.imag)), axis=1)
    E = np.frexp(m)[1]

    def cut(v):
        v = np.ldexp(v, (7 - E)[:, None])
        out = []
        for _ in range(S):
            d = np.rint(v)
            out.append(d)
            v = (v - d) * 256.0
        return out

    return E, [np.concatenate(p, axis=1) for p in zip(cut(x.real), cut(x.imag))]


def product(a, b, S, lost=None):
    """a @ b.T as the split product forms it; `lost`: scale whose first 256 stacked indices are left out."""
    ea, da = digits(a, S)
    eb, db = digits(b, S)
    k = a.shape[1]
    re = [np.concatenate([d[:, :k], -d[:, k:]], axis=1) for d in db]
    im = [np.concatenate([d[:, k:], d[:, :k]], axis=1) for d in db]
    out = np.zeros((a.shape[0], b.shape[0]), complex)
    for scale in range(S - 1, -1, -1):
        c = 0
        for t in range(scale + 1):
            x, u = da[t], scale - t
            if scale == lost:
                x = x.copy()
                x[:, :256] = 0.0
            c = c + (x @ re[u].T + 1j * (x @ im[u].T))
        out = out + c * 2.0 ** (-8 * scale - 14)
    return out * np.ldexp(1.0, ea)[:, None] * np.ldexp(1.0, eb)[None, :]


@functools.lru_cache(maxsize=None)
def model_error(s, r, S, lost=None, where=None):
    """Largest error of G on the pattern over max|G| with split products (a scale lost in L or T)."""
    H, X = matrices(s, r)
    A = Z * np.eye(2 * s + r) - H
    R = slice(s, s + r)
    leaves = [slice(0, s), slice(s + r, 2 * s + r)]
    P = [np.linalg.inv(A[J, J]) for J in leaves]
    L = [product(A[R, J], p, S, lost if where == "L" else None) for J, p in zip(leaves, P)]
    schur = A[R, R] - sum(product(l, A[R, J], S) for J, l in zip(leaves, L))
    G = np.linalg.inv(schur)
    err = np.max(np.abs(G - X[R, R]))
    for J, p, l in zip(leaves, P, L):
        T = product(G, l.T, S, lost if where == "T" else None)
        D = p + product(l.T, T.T, S)
        err = max(err, np.max(np.abs(-T - X[R, J])), np.max(np.abs(D - X[J, J])))
    return float(err / np.max(np.abs(X)))


def limit(s, r, S, bands=0):
    H, X = matrices(s, r)
    n = 2 * s + r
    fp64 = 20 * np.sqrt(n) * U * float(np.linalg.cond(X))
    tail = {0: 0.0, 4: 20 * 2.0 ** -38, 5: 20 * 2.0 ** -43}[bands if S > bands else 0]
    return 8 * model_error(s, r, S) + fp64 + tail


# separators at the edges of K blocks (32), chunks (128) and read-out periods (256, 512); leaves likewise
T_SHAPES = [(96, 128), (96, 129), (96, 256), (64, 257), (64, 384), (64, 513), (90, 600)]
L_SHAPES = [(256, 40), (257, 48), (385, 32)]


@pytest.mark.parametrize("S", [4, 5, 6])
@pytest.mark.parametrize("s,r,where", [(96, 129, "T"), (64, 257, "T"), (90, 600, "T"), (257, 48, "L")])
def test_a_lost_scale_exceeds_the_limit(S, s, r, where):
    for lost in range(S):
        assert model_error(s, r, S, lost, where) > 1.5 * limit(s, r, S), lost


def run(s, r, **opts):
    import torch
    import paper_1005_0088_gb300 as nd
    H, X = matrices(s, r)
    n = 2 * s + r
    centers = np.array([[0.0, 0, 0], [1.0, 0, 0], [2.0, 0, 0]])
    pattern = np.ones((n, n))
    pattern[:s, s + r:] = pattern[s + r:, :s] = 0.0
    sysm = csr_from_dense(np.where((H == 0) & (pattern > 0), 1e-300, H), np.eye(n), centers,
                          np.repeat(np.arange(3, dtype=np.int32), [s, r, s]))
    plan = nd.analyze_system(sysm, leaf_atoms=1, precision=nd.NDSI_PREC_SPLIT, outer_block=1024, **opts)
    f = nd.ndsi_factor_poles(plan, torch.as_tensor(sysm.H, device="cuda"), torch.as_tensor(sysm.S, device="cuda"), np.array([Z]))
    G = torch.zeros((1, sysm.nnz, 2), dtype=torch.float64, device="cuda")
    nd.ndsi_selinv(f, G)
    g = G.cpu().numpy()[0]
    return float(np.max(np.abs(g[:, 0] + 1j * g[:, 1] - X[sysm.rows(), sysm.col])) / np.max(np.abs(X)))


@pytest.mark.gpu
@pytest.mark.parametrize("S", [4, 5, 6, 7])
@pytest.mark.parametrize("s,r", T_SHAPES + L_SHAPES)
def test_every_scale_is_read_once(S, s, r):
    err = run(s, r, split_slices=S)
    assert err < limit(s, r, S), (err, limit(s, r, S), model_error(s, r, S))


@pytest.mark.gpu
@pytest.mark.parametrize("S", [4, 5, 6, 7])
@pytest.mark.parametrize("bands", [4, 5])
def test_tail_layouts(S, bands):
    err = run(64, 257, split_slices=S, split_bands=bands)
    assert err < limit(64, 257, S, bands), (err, limit(64, 257, S, bands))
