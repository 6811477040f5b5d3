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
