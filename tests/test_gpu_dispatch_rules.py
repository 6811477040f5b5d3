"""Calls that a rule on sizes or types sends to one of several kernels, at
the sizes where the rule turns, each against the float64 oracle or the
definition."""
import numpy as np
import pytest

import oracle as O
from paper_2408_02398_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

UNIT = {1: 2.0 ** -11, 2: 2.0 ** -8}  # unit roundoff of 16-bit spectra
C_TOL = 2e-5   # FP32 transforms of unit-variance data, as for every correlate test
W_TOL = 1e-5


@pytest.fixture(scope="module")
def T():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2408_02398_gb300 import build
    build.build()
    from paper_2408_02398_gb300 import ttm
    return ttm


@pytest.fixture(scope="module")
def ctx(T):
    return T.Context(0)


def dev(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


# register lengths of every axis in FP32, FP16 and BF16: at 1024 the strided
# passes and the 16-bit z pass keep 8 lines per CTA, the row passes 4; column
# and row counts leave remainders of both
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("shape", [(1024, 9, 14), (9, 1024, 14), (9, 10, 1024), (512, 9, 14), (9, 512, 14),
                                   (9, 10, 512), (200, 9, 14), (9, 200, 14), (9, 10, 200), (9, 10, 256),
                                   (9, 10, 128), (9, 10, 64)])
def test_register_lengths(T, ctx, shape, prec):
    V, N, r = int(np.prod(shape)), 9, 4.0
    tomo = synth.normals(3, 1, V).reshape(shape).astype(np.float32)
    tmpl = synth.gaussian_blob_template(N, seed=N)
    m, _ = O.mask(tmpl.shape, r)
    field = O.tensor_field(O.normalise_template(tmpl, m)[0], O.rotation_set(4), 2)
    plan = T.Plan(ctx, dev(field, torch.float64), T.params(order_n=2, mask_radius=r, n_rot_base=4), shape,
                  precision=prec)
    d_C = torch.empty((6,) + shape, device="cuda")
    T.ttm_correlate(plan, dev(tomo), d_C)
    vox = np.sort(np.random.default_rng(N).choice(V, size=400, replace=False))
    pr = O.Prepared(tomo.astype(np.float64), tmpl, r)
    w, _, _ = O.local_w(pr.g, pr.m, vox, periodic=True, floor=pr.floor)
    C = O.correlate(pr.g, field, vox, periodic=True, w=w)
    got = d_C.cpu().numpy().reshape(6, -1)[:, vox]
    if prec == 0:
        assert np.abs(got - C).max() <= C_TOL * max(1.0, np.abs(C).max())
    else:
        # three roundings of the storage format (stored spectrum, z- and y-pass stores)
        assert np.linalg.norm(got - C) <= 3 * UNIT[prec] * np.linalg.norm(C)
        assert np.abs(got - C).max() <= 3 * UNIT[prec] * np.abs(C).max()


# quaternion maximiser, n = 2 (closed form, its own register budget): less than
# one voxel block, and a volume of many
@pytest.mark.parametrize("shape", [(5, 6, 7), (96, 100, 126)])
def test_quaternion_order2_closed_form(T, ctx, shape):
    N, V = 5, int(np.prod(shape))
    field = torch.zeros((10, N, N, N), dtype=torch.float64, device="cuda")
    field[:, 2, 2, 2] = 1.0
    plan = T.Plan(ctx, field, T.params(order_n=2, mask_radius=2.0, dprime=4, n_rot_base=1), shape)
    C = torch.as_tensor(np.random.default_rng(V).standard_normal((10, V)), dtype=torch.float32, device="cuda")
    s = torch.full(shape, np.nan, device="cuda")
    q = torch.full((4,) + shape, np.nan, device="cuda")
    f = torch.full(shape, np.nan, device="cuda")
    T.ttm_peak_map(plan, C, s, q, f)
    at = np.unique(np.concatenate([np.arange(max(0, V - 2000), V), np.linspace(0, V - 1, 4000).astype(np.int64)]))
    c, A = C.cpu().numpy().astype(np.float64)[:, at], np.empty((len(at), 4, 4))
    for k, (i, j) in enumerate((i, j) for i in range(4) for j in range(i, 4)):
        A[:, i, j] = A[:, j, i] = c[k]
    F = np.sqrt((A * A).sum((1, 2)))
    got, u = s.cpu().numpy().ravel()[at], q.view(4, V).cpu().numpy().astype(np.float64)[:, at].T
    # sixteen FP32 products of |A| <= F: some 2^-22 F
    assert np.all(np.abs(got - np.linalg.eigvalsh(A)[:, -1]) <= 1e-5 * F)
    assert np.all(np.abs(np.einsum("vi,vij,vj->v", u, A, u) - got) <= 1e-5 * F)
    assert np.all(np.abs(f.cpu().numpy().ravel()[at] - F) <= 1e-6 * F)
    assert not torch.isnan(s).any() and not torch.isnan(q).any()


# plain maximiser, n = 2: less than one voxel block, a part of a wave of CTAs,
# one wave that takes several blocks each, and four blocks per CTA with a rest
@pytest.mark.parametrize("shape", [(5, 6, 7), (40, 42, 45), (75, 80, 81), (100, 126, 135)])
def test_plain_order2_closed_form(T, ctx, shape):
    N, V = 5, int(np.prod(shape))
    field = torch.zeros((6, N, N, N), dtype=torch.float64, device="cuda")
    field[:, 2, 2, 2] = 1.0
    plan = T.Plan(ctx, field, T.params(order_n=2, mask_radius=2.0, n_rot_base=1), shape)
    C = torch.as_tensor(np.random.default_rng(V).standard_normal((6, V)), dtype=torch.float32, device="cuda")
    s = torch.full(shape, np.nan, device="cuda")
    u = torch.full((3,) + shape, np.nan, device="cuda")
    f = torch.full(shape, np.nan, device="cuda")
    T.ttm_peak_map(plan, C, s, u, f)
    c, A = C.cpu().numpy().astype(np.float64), np.empty((V, 3, 3))
    for k, (i, j) in enumerate((i, j) for i in range(3) for j in range(i, 3)):
        A[:, i, j] = A[:, j, i] = c[k]
    F = np.sqrt((A * A).sum((1, 2)))
    got, d = s.cpu().numpy().ravel(), u.view(3, V).cpu().numpy().astype(np.float64).T
    # nine FP32 products of |A| <= F: some 2^-22 F
    assert np.all(np.abs(got - np.linalg.eigvalsh(A)[:, -1]) <= 1e-5 * F)
    assert np.all(np.abs(np.einsum("vi,vij,vj->v", d, A, d) - got) <= 1e-5 * F)
    assert np.all(np.abs(f.cpu().numpy().ravel() - F) <= 1e-6 * F)


def bf16(a):
    return torch.as_tensor(np.asarray(a, np.float32)).bfloat16().double().numpy()


def gelu(x):
    return 0.5 * x * (1 + np.tanh(np.sqrt(2 / np.pi) * (x + 0.044715 * x ** 3)))


def gelu_grad(x):
    c = np.sqrt(2 / np.pi)
    t = np.tanh(c * (x + 0.044715 * x ** 3))
    return 0.5 * (1 + t) + 0.5 * x * (1 - t * t) * c * (1 + 3 * 0.044715 * x * x)


def bf16_loss_grad(p, X, U):
    """Summed loss and gradient with the operands of every product rounded to BF16, all else in float64."""
    K, H = X.shape[1], 128
    at, w = 0, []
    for s in ((H, K), (H,), (H, H), (H,), (3, H), (3,)):
        w.append(p[at:at + int(np.prod(s))].reshape(s).astype(np.float64))
        at += int(np.prod(s))
    W1, b1, W2, b2, W3, b3 = w
    a1 = bf16(X) @ bf16(W1).T + b1
    a2 = bf16(gelu(a1)) @ bf16(W2).T + b2
    h2 = bf16(gelu(a2))
    y = h2 @ bf16(W3).T + b3
    ny = np.linalg.norm(y, axis=1, keepdims=True)
    u = y / ny
    dot = (u * U).sum(1, keepdims=True)
    g = -2 * dot * U
    dy = (g - (u * g).sum(1, keepdims=True) * u) / ny
    d2 = bf16(dy) @ bf16(W3) * gelu_grad(a2)
    d1 = bf16(d2) @ bf16(W2) * gelu_grad(a1)
    parts = [bf16(d1).T @ bf16(X), d1.sum(0), bf16(d2).T @ bf16(gelu(a1)), d2.sum(0), bf16(dy).T @ h2, dy.sum(0)]
    return float((1 - dot ** 2).sum()), np.concatenate([v.ravel() for v in parts])


# BF16 training products: one row, remainders of the 16-row steps and of the row
# splits, one and two column tiles of W1, two chunks of rows
@pytest.mark.parametrize("K,rows", [(6, 1), (15, 63), (28, 65), (28, 4097), (64, 80), (65, 200), (128, 1000),
                                    (15, 65537)])
def test_mlp_bf16_gradient_splits(T, ctx, K, rows):
    rng = np.random.default_rng(K + rows)
    X = rng.standard_normal((rows, K))
    U = rng.standard_normal((rows, 3))
    X = (X / np.linalg.norm(X, axis=1, keepdims=True)).astype(np.float32)
    U = (U / np.linalg.norm(U, axis=1, keepdims=True)).astype(np.float32)
    net = T.Mlp(ctx, K, seed=rows)
    net.set_precision(T.TTM_MLP_BF16)
    g = torch.full((net.num_params,), np.nan, device="cuda")
    L = net.loss_grad(dev(X), dev(U), g)
    Lo, go = bf16_loss_grad(net.get_params(), X, U.astype(np.float64))
    # FP32 sums, and here and there an operand that FP32 rounds to the
    # neighbouring BF16 value: 2^-8 of one term of some hundred
    assert abs(L - Lo) <= 2.0 ** -8 * max(Lo, 1.0)
    assert np.abs(g.cpu().numpy() - go).max() <= 2.0 ** -8 * np.abs(go).max()


# the list of maxima runs out before P peaks are found
@pytest.mark.parametrize("P,dist", [(1, 1e4), (3000, 0.0), (3000, 7.0), (3000, 1e4)])
def test_find_peaks_exhausts_its_maxima(T, ctx, P, dist):
    shape, N = (16, 25, 40), 5
    m = np.random.default_rng(P).integers(0, 50, shape).astype(np.float32)
    field = torch.zeros((6, N, N, N), dtype=torch.float64, device="cuda")
    field[:, 2, 2, 2] = 1.0
    plan = T.Plan(ctx, field, T.params(order_n=2, mask_radius=2.0, n_rot_base=1), shape)
    b = plan.valid_box()
    want_i, want_v = T.ttm_find_peaks_noalloc(ctx, dev(m), b, 16384, 0.0)  # all maxima, in order
    zyx = np.stack(np.unravel_index(want_i, shape), 1).astype(float)
    keep = []
    for k in range(len(want_i)):
        if len(keep) < P and all(((zyx[k] - zyx[a]) ** 2).sum() >= dist ** 2 for a in keep):
            keep.append(k)
    idx, val = T.ttm_find_peaks(plan, dev(m), P, dist)
    assert idx.tolist() == want_i[keep].tolist() and np.array_equal(val, want_v[keep])
    assert 0 < len(keep) < max(P, 2)
