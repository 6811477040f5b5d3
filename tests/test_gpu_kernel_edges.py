"""Edge sizes of the kernels' tiles and of the rules that choose between
kernels, each against the float64 oracle at sampled voxels."""
import json

import numpy as np
import pytest

import oracle as O
from paper_2408_02398_gb300 import synth

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

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


def check_correlate(T, ctx, shape, N, r, n, localsum, samples=400, seed=1):
    V = int(np.prod(shape))
    tomo = synth.normals(seed, 1, V).reshape(shape).astype(np.float32)
    tmpl = synth.gaussian_blob_template(N, seed=N)
    m, _ = O.mask(tmpl.shape, r)
    field = O.tensor_field(O.normalise_template(tmpl, m)[0], O.rotation_set(4), n)
    plan = T.Plan(ctx, dev(field, torch.float64), T.params(order_n=n, mask_radius=r, n_rot_base=4), shape)
    T.ttm_plan_set_localsum(plan, localsum)
    d_C = torch.empty((field.shape[0],) + tuple(shape), device="cuda")
    d_w = torch.empty(shape, device="cuda")
    T.ttm_correlate(plan, dev(tomo), d_C)
    T.ttm_plan_copy_w(plan, d_w)
    torch.cuda.synchronize()
    vox = np.sort(np.random.default_rng(N).choice(V, size=min(V, samples), replace=False))
    pr = O.Prepared(tomo.astype(np.float64), tmpl, r)
    w, _, _ = O.local_w(pr.g, pr.m, vox, periodic=True, floor=pr.floor)
    C = O.correlate(pr.g, field, vox, periodic=True, w=w)
    assert np.abs(d_w.cpu().numpy().ravel()[vox] - w).max() <= W_TOL * np.abs(w).max()
    got = d_C.cpu().numpy().reshape(field.shape[0], -1)[:, vox]
    assert np.abs(got - C).max() <= C_TOL * max(1.0, np.abs(C).max())


# shared-memory transforms: line counts that are no multiple of the tile
# width, every radix, and lengths at which the tile width drops to its least
@pytest.mark.parametrize("localsum", [0, 1])
@pytest.mark.parametrize("shape", [(14, 15, 45), (9, 10, 1260), (10, 1120, 9), (1050, 9, 14), (27, 49, 25),
                                   (16, 24, 40)])
def test_shared_memory_transform_tiles(T, ctx, shape, localsum):
    check_correlate(T, ctx, shape, 9, 4.0, 2, localsum)


def test_tile_width_of_a_loaded_record(T, tmp_path):
    """A tuning record may ask for any tile width: it is rounded down to a power of two."""
    c = T.Context(0)
    f = tmp_path / "tune.json"
    T.ttm_autotune_shape(c, (45, 45, 45))
    T.ttm_autotune_save(c, str(f))
    text = f.read_text()
    rec = json.loads(text)
    rows = rec["lengths"] if isinstance(rec, dict) and "lengths" in rec else rec
    for row in rows:
        if not row["reg"]:
            row["W"] = 12
    f.write_text("[\n" + ",\n".join(json.dumps(r) for r in rows) + "\n]\n")
    T.ttm_autotune_load(c, str(f))
    check_correlate(T, c, (45, 45, 45), 9, 4.0, 2, 0)


# weight gradients split over the rows: single rows, remainders of the k steps
# and of the splits, one and two column tiles of W1, and two chunks of rows
@pytest.mark.parametrize("K,rows", [(6, 1), (15, 63), (28, 65), (28, 4097), (64, 80), (65, 200), (128, 1000),
                                    (15, 65537)])
def test_mlp_gradient_splits(T, ctx, K, rows):
    rng = np.random.default_rng(K + rows)
    X = rng.standard_normal((rows, K))
    X /= np.linalg.norm(X, axis=1, keepdims=True)
    U = rng.standard_normal((rows, 3))
    U /= np.linalg.norm(U, axis=1, keepdims=True)
    X, U = X.astype(np.float32), U.astype(np.float32)
    net = T.Mlp(ctx, K, seed=rows)
    g = torch.zeros(net.num_params, device="cuda")
    L = net.loss_grad(dev(X), dev(U), g)
    _, Lo, go = O.mlp(net.get_params().astype(np.float64), X.astype(np.float64), U.astype(np.float64), want_grad=True)
    got = g.cpu().numpy()
    # the bounds of the gradient check in test_gpu_mlp.py
    assert abs(L - Lo) <= 1e-5 * max(Lo, 1e-3)
    assert np.abs(got - go).max() <= 1e-4 * np.abs(go).max()


def brute_peaks(m, box):
    """Strict 26-neighbour maxima inside the box (ties to the lower index, NaN neither a peak nor a rival)."""
    z0, z1, y0, y1, x0, x1 = box
    out = []
    for z in range(z0, z1):
        for y in range(y0, y1):
            for x in range(x0, x1):
                v = m[z, y, x]
                if v != v:
                    continue
                ok = True
                for c in range(max(z0, z - 1), min(z1, z + 2)):
                    for b in range(max(y0, y - 1), min(y1, y + 2)):
                        for a in range(max(x0, x - 1), min(x1, x + 2)):
                            o = m[c, b, a]
                            if o > v or (o == v and (c, b, a) < (z, y, x)):
                                ok = False
                if ok:
                    out.append((-v, (z * m.shape[1] + y) * m.shape[2] + x))
    return [i for _, i in sorted(out)]


# column tiles of 30, rows of 4, chunks of planes; ties, infinities and NaN
@pytest.mark.parametrize("shape,box", [((19, 9, 70), (0, 19, 0, 9, 0, 70)), ((18, 12, 62), (1, 18, 2, 11, 1, 61)),
                                       ((5, 7, 31), (0, 5, 0, 7, 0, 31)), ((4, 4, 64), (3, 4, 3, 4, 5, 6)),
                                       ((33, 5, 33), (0, 33, 0, 5, 2, 32)), ((3, 3, 3), (1, 1, 0, 3, 0, 3))])
def test_find_peaks_tiles_and_special_values(T, ctx, shape, box):
    rng = np.random.default_rng(sum(shape))
    for levels in (3, 1000):
        m = rng.integers(0, levels, shape).astype(np.float32)
        m[rng.random(shape) < 0.05] = np.nan
        m[rng.random(shape) < 0.02] = np.inf
        m[rng.random(shape) < 0.02] = -np.inf
        m[0, 0, 0] = -np.inf
        idx, val = T.ttm_find_peaks_noalloc(ctx, dev(m), box, 16384, 0.0)
        want = brute_peaks(m, box)
        assert idx.tolist() == want
        assert np.array_equal(val, m.ravel()[want])


# the reach list (odd and even templates, soft masks) and the path for
# quaternions that are not unit; peaks at the corners of the valid box
@pytest.mark.parametrize("scale", [1.0, 1.003])
@pytest.mark.parametrize("N,r,soft", [(9, 4.0, 0.0), (8, 3.5, 0.0), (12, 3.0, 2.5), (13, 5.0, 1.0)])
def test_refine_reach_against_direct_sum(T, ctx, N, r, soft, scale):
    shape = (20, 21, 25)
    rng = np.random.default_rng(N)
    tomo = synth.normals(N, 1, int(np.prod(shape))).reshape(shape).astype(np.float32)
    tmpl = synth.gaussian_blob_template(N, seed=N, std_lo=0.7, std_hi=1.5).astype(np.float32)
    pr = O.Prepared(tomo.astype(np.float64), tmpl.astype(np.float64), r, soft=soft)
    field = O.tensor_field(pr.tp, O.rotation_set(1), 2, 4)
    p = T.params(order_n=2, mask_radius=r, mask_soft_width=soft, dprime=4, n_rot_base=1)
    plan = T.Plan(ctx, dev(field, torch.float64), p, shape)
    T.ttm_correlate(plan, dev(tomo), torch.empty((10,) + shape, device="cuda"))
    d_w = torch.empty(shape, device="cuda")
    T.ttm_plan_copy_w(plan, d_w)
    w = d_w.cpu().numpy().astype(np.float64)
    q = rng.standard_normal((4,) + shape)
    q = (scale * q / np.linalg.norm(q, axis=0)).astype(np.float32)
    b = plan.valid_box()
    at = [(b[0], b[2], b[4]), (b[1] - 1, b[3] - 1, b[5] - 1), (b[0], b[3] - 1, b[4])]
    peaks = np.array([(z * shape[1] + y) * shape[2] + x for z, y, x in at])
    idx, quat, lncc = T.ttm_refine_peaks(plan, dev(tmpl), dev(q), peaks, r_s=0.0)
    assert np.array_equal(idx, peaks)
    h = N // 2
    for (z, y, x), ql, c in zip(at, quat, lncc):
        assert np.array_equal(ql, q[:, z, y, x])
        tv = synth.resample_rotated(pr.tp, synth.quat_matrix(ql.astype(np.float64)))
        win = pr.g.reshape(shape)[z - h:z - h + N, y - h:y - h + N, x - h:x - h + N]
        # FP32 coordinates, samples and partial sums of |t'| = 1 against windows of norm 1 / w
        assert abs(c - w[z, y, x] * (tv * win).sum()) <= 2e-5


@pytest.mark.parametrize("prec", [0, 1])
def test_side_stream_local_sums_on_user_streams(T, ctx, prec):
    """FP64 local sums run beside the FP32 passes: the same bits on any stream, back to back, and replayed from a graph."""
    shape, N, r = (24, 21, 20), 7, 3.0
    tmpl = synth.gaussian_blob_template(N, seed=N)
    m, _ = O.mask(tmpl.shape, r)
    field = dev(O.tensor_field(O.normalise_template(tmpl, m)[0], O.rotation_set(4), 2), torch.float64)
    tomos = [dev(synth.normals(k, 1, int(np.prod(shape))).reshape(shape)) for k in (1, 2, 3)]
    plan = T.Plan(ctx, field, T.params(order_n=2, mask_radius=r, n_rot_base=4), shape, precision=prec)
    T.ttm_plan_enable_timing(plan, True)  # timed stages run in sequence
    want = []
    for t in tomos:
        d_C = torch.empty((6,) + shape, device="cuda")
        T.ttm_correlate(plan, t, d_C)
        want.append(d_C)
    torch.cuda.synchronize()
    T.ttm_plan_enable_timing(plan, False)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    got = [torch.empty((6,) + shape, device="cuda") for _ in tomos]
    with torch.cuda.stream(s):
        for t, c in zip(tomos, got):
            T.ttm_correlate(plan, t, c)
    s.synchronize()
    for a, b in zip(want, got):
        assert torch.equal(a, b)
    d_C, d_t = torch.zeros((6,) + shape, device="cuda"), tomos[0].clone()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        T.ttm_correlate(plan, d_t, d_C)
    for t, w in zip(tomos, want):
        d_t.copy_(t)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(d_C, w)
