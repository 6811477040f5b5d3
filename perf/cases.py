"""The work that a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values; its "kind" names the call:

  match      ttm_correlate and ttm_peak_map of one tomogram (Matcher.run)
  correlate  ttm_correlate alone: tomogram -> K normalised tensor components
  peak_map   ttm_peak_map alone: components -> score, orientation, Frobenius norm
  find_peaks ttm_find_peaks on a score map
  refine     ttm_refine_peaks (TTM-ref) of a list of peaks
  batch      Batch.run: sub-tomograms of uneven sizes x templates, one graph
  blocked    Blocked.run: a tomogram in pinned host memory, in z-slabs
  mlp_train  Mlp.train: the warm-start network on one set of pairs

Inputs are made on the GPU by torch from the seed alone (noise with planted
rotated copies, the tensor field by Alg. 1 over a small rotation set), so
that they do not depend on the code that is measured; `exact` evaluates the
same definitions in float64.
"""
import functools
import math

import numpy as np
import torch

from paper_2408_02398_gb300 import ttm

DEV = "cuda"
FILTER_A = 0.2
N_ROT = 192                 # rotations of the tensor fields made here
SMOOTH = [48, 50, 54, 60, 63, 64, 70, 72, 75, 80, 81, 84, 90, 96, 98, 100, 105, 108, 112, 120, 125, 126, 128, 135,
          140, 144, 147, 150, 160, 162, 168, 175, 180, 189, 192, 196, 200, 210, 216, 224, 225, 240, 243, 245, 250,
          252, 256, 270, 280, 288, 294, 300, 315, 320, 324, 336, 343, 350, 360, 375, 378, 384, 392, 400, 405, 420,
          432, 441, 448, 450, 480, 486, 490, 500, 504, 512]


# ------------------------------------------------------------------ cases --

def listed():
    return [
        # the 64^3 test volume: one small sub-tomogram matched with the defaults, where launches count
        {"name": "match_n2_64", "kind": "match", "Z": 64, "Y": 64, "X": 64, "t": 16, "n": 2, "d": 3, "sums": "fp64",
         "prec": "fp32"},
        # the benchmark's tomogram and template: the correlate stage of a whole cryo-ET volume
        {"name": "correlate_n4_512", "kind": "correlate", "Z": 200, "Y": 512, "X": 512, "t": 40, "n": 4, "d": 3,
         "sums": "df64", "prec": "fp32"},
        # a cropped volume of odd 7-smooth extents with every default (FP64 local sums)
        {"name": "correlate_n4_ragged", "kind": "correlate", "Z": 126, "Y": 270, "X": 315, "t": 32, "n": 4, "d": 3,
         "sums": "fp64", "prec": "fp32"},
        # order 6 with 16-bit spectra, as the mixed-precision benchmark runs it
        {"name": "correlate_n6_fp16", "kind": "correlate", "Z": 256, "Y": 512, "X": 512, "t": 48, "n": 6, "d": 3,
         "sums": "df64", "prec": "fp16"},
        # the score and orientation maps of the benchmark's tomogram: the largest share of its step
        {"name": "peak_map_n4_512", "kind": "peak_map", "Z": 200, "Y": 512, "X": 512, "t": 40, "n": 4, "d": 3},
        # the same for order 6 on a sub-volume
        {"name": "peak_map_n6", "kind": "peak_map", "Z": 64, "Y": 256, "X": 256, "t": 48, "n": 6, "d": 3},
        # full rotations: the quaternion form's maps
        {"name": "peak_map_d4_n4", "kind": "peak_map", "Z": 100, "Y": 256, "X": 256, "t": 40, "n": 4, "d": 4},
        # the peak list of the whole volume, exclusion 2 r
        {"name": "find_peaks_512", "kind": "find_peaks", "Z": 200, "Y": 512, "X": 512, "t": 40, "P": 300},
        # TTM-ref of a volume's peaks over the radius-3 ball
        {"name": "refine_300", "kind": "refine", "Z": 128, "Y": 256, "X": 256, "t": 40, "P": 300, "rs": 3.0},
        # picked sub-tomograms of uneven sizes against several templates
        {"name": "batch_6x2", "kind": "batch", "tomos": 6, "templates": 2, "lo": 96, "hi": 176, "t": 32, "n": 4,
         "sums": "df64"},
        # a tomogram that stays in host memory, processed in slabs, down to its peak list
        {"name": "blocked_host", "kind": "blocked", "Z": 128, "Y": 224, "X": 288, "t": 40, "n": 4, "slab": 48,
         "P": 48},
        # one epoch of the warm-start network on correlation pairs, default arithmetic
        {"name": "mlp_train_n6", "kind": "mlp_train", "n": 6, "pairs": 65536, "batch": 4096, "epochs": 1,
         "prec": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _peak_count(rng, t, dims, hi):
    """Up to hi peaks, as many as surely find room at distance 2 r in the valid box."""
    room = 1.0
    for s in dims:
        room *= s - t + 1
    return _log_int(rng, 1, max(1, min(hi, int(0.3 * room / (2 * _radius(t)) ** 3))))


def _grid(rng, t, most):
    """Three 7-smooth extents >= the template with at most `most` voxels, their product spread over its logarithm."""
    target = math.exp(rng.uniform(math.log(max(t, 48) ** 3), math.log(most)))
    while True:
        z, y = rng.choice(SMOOTH), rng.choice(SMOOTH)
        x = min(SMOOTH, key=lambda s: abs(s - target / (z * y)))
        if min(z, y, x) >= t and 0.5 * target <= z * y * x <= min(most, 2 * target):
            return {"Z": z, "Y": y, "X": x}


def draw(rng):
    kind = rng.choice(["match", "correlate", "correlate", "correlate", "peak_map", "peak_map", "peak_map",
                       "find_peaks", "refine", "batch", "blocked", "mlp_train"])
    t = rng.choice([12, 16, 21, 24, 31, 32, 40, 48])
    n = rng.choice([2, 4, 4, 6])
    if kind == "match":
        return {"kind": kind, **_grid(rng, t, 2 ** 20), "t": t, "n": 2, "d": 3, "sums": rng.choice(["fp64", "df64"]),
                "prec": "fp32"}
    if kind == "correlate":
        d = rng.choice([3, 3, 3, 4])
        return {"kind": kind, **_grid(rng, t, 2 ** 25 // (4 if d == 4 else 2 if n == 6 else 1)), "t": t, "n": n, "d": d,
                "sums": rng.choice(["fp64", "df64"]), "prec": rng.choice(["fp32", "fp32", "fp16", "bf16"])}
    if kind == "peak_map":
        d = rng.choice([3, 3, 3, 4])
        return {"kind": kind, **_grid(rng, t, 2 ** 24 // (1 if d == 3 else 4 if n < 6 else 16)), "t": t, "n": n, "d": d}
    if kind == "find_peaks":
        g = _grid(rng, t, 2 ** 25)
        return {"kind": kind, **g, "t": t, "P": _peak_count(rng, t, g.values(), 1000)}
    if kind == "refine":
        return {"kind": kind, **_grid(rng, max(t, 60), 2 ** 23), "t": t, "P": _log_int(rng, 10, 300),
                "rs": rng.choice([2.0, 3.0])}
    if kind == "batch":
        lo = rng.randint(max(t, 48), 110)
        return {"kind": kind, "tomos": rng.randint(2, 6), "templates": rng.randint(1, 3), "lo": lo,
                "hi": lo + rng.randint(8, 64), "t": t, "n": rng.choice([2, 4]), "sums": rng.choice(["fp64", "df64"])}
    if kind == "blocked":
        dims = [rng.randint(t + 30, 150), rng.randint(t + 20, 256), rng.randint(t + 20, 320)]
        return {"kind": kind, "Z": dims[0], "Y": dims[1], "X": dims[2], "t": t, "n": rng.choice([2, 4]),
                "slab": rng.randint(16, 80), "P": _peak_count(rng, t, dims, 100)}
    return {"kind": kind, "n": n, "pairs": _log_int(rng, 8192, 65536), "batch": _log_int(rng, 512, 4096),
            "epochs": 1, "prec": "fp32"}


# ----------------------------------------------------------------- inputs --

def _generator(seed, stream):
    return torch.Generator(device=DEV).manual_seed((seed * 1000003 + stream * 7919 + 12345) % (1 << 62))


def _radius(t):
    return {16: 7.0, 21: 9.0}.get(t, float(int(0.4 * t)))  # 12 for 32, 16 for 40, 19 for 48


def _exponents(n, d):
    """Exponents of the degree-n monomials in d variables, graded-lex descending."""
    if d == 1:
        return [(n,)]
    return [(a,) + r for a in range(n, -1, -1) for r in _exponents(n - a, d - 1)]


def _multinomial(e):
    m = math.factorial(sum(e))
    for a in e:
        m //= math.factorial(a)
    return m


def _monomials(u, n):
    """[K, ...] monomials of the components u[0..d-1] (tensors)."""
    rows = []
    for e in _exponents(n, u.shape[0]):
        v = torch.ones_like(u[0])
        for c, a in zip(u, e):
            if a:
                v = v * c ** a
        rows.append(v)
    return torch.stack(rows)


def _unit_quats(count, gen):
    q = torch.randn(count, 4, generator=gen, device=DEV, dtype=torch.float64)
    return q / q.norm(dim=1, keepdim=True)


def _rotations(q):
    w, x, y, z = q.unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], dim=1).view(-1, 3, 3)


def _offsets(t):
    """[t^3, 3] offsets (x, y, z) from the centre, C order over (z, y, x)."""
    a = torch.arange(t, device=DEV, dtype=torch.float64) - t // 2
    z, y, x = torch.meshgrid(a, a, a, indexing="ij")
    return torch.stack([x, y, z], dim=-1).view(-1, 3)


def _template(t, gen):
    """Six anisotropic Gaussian blobs, maximum 1 (float32 [t][t][t])."""
    p = _offsets(t)
    out = torch.zeros(t ** 3, device=DEV, dtype=torch.float64)
    scale = t / 40.0
    for R in _rotations(_unit_quats(6, gen)):
        c = torch.randn(3, generator=gen, device=DEV, dtype=torch.float64)
        c = 5.0 * scale * c / c.norm() * torch.rand(1, generator=gen, device=DEV, dtype=torch.float64) ** (1 / 3)
        s = scale * (1.0 + 2.0 * torch.rand(3, generator=gen, device=DEV, dtype=torch.float64)) + 0.3
        out += torch.exp(-0.5 * (((p - c) @ R / s) ** 2).sum(1))
    return (out / out.max()).view(t, t, t).float()


def _sample(vol, R):
    """vol sampled at R^T p for every rotation of R [B, 3, 3]: [B, t^3] float64."""
    t = vol.shape[0]
    src = torch.einsum("bij,ni->bnj", R, _offsets(t)) + t // 2  # (R^T p) + centre, order (x, y, z)
    grid = (2.0 * src / (t - 1) - 1.0)[None, :, :, None, :]
    return torch.nn.functional.grid_sample(vol[None, None], grid, mode="bilinear", padding_mode="zeros",
                                           align_corners=True)[0, 0, :, :, 0]


def _mask(t):
    return ((_offsets(t) ** 2).sum(1).sqrt() <= _radius(t)).double().view(t, t, t)


def _filter(v, a=FILTER_A):
    """The separable taps (a, 1 - 2a, a) on each axis, zero padded."""
    for ax in range(3):
        n = v.shape[ax]
        o = v * (1 - 2 * a)
        o.narrow(ax, 1, n - 1).add_(v.narrow(ax, 0, n - 1), alpha=a)
        o.narrow(ax, 0, n - 1).add_(v.narrow(ax, 1, n - 1), alpha=a)
        v = o
    return v


def _normalised_template(tmpl):
    """Eq. 4: filtered, masked, zero mean and unit norm under the mask."""
    m = _mask(tmpl.shape[0])
    s = m * _filter(tmpl.double())
    M = m.sum()
    return m * (s - (s * m).sum() / M) / ((s * s).sum() - s.sum() ** 2 / M).sqrt()


def _field(tmpl, n, d):
    """Alg. 1 over N_ROT rotations: float64 [K][t][t][t]."""
    t = tmpl.shape[0]
    q = _unit_quats(N_ROT, _generator(99, 1))
    R = _rotations(q)
    u = R[:, :, 2].T.contiguous() if d == 3 else q.T.contiguous()
    tp = _normalised_template(tmpl)
    out = None
    for s in range(0, N_ROT, 32):
        part = _monomials(u[:, s:s + 32], n) @ _sample(tp, R[s:s + 32])
        out = part if out is None else out + part
    return (out / N_ROT).view(-1, t, t, t).contiguous()


def _tomogram(shape, tmpl, gen, lowpass=True):
    """Unit-variance noise (low-passed, sigma 1) with rotated copies planted at SNR 0.1, float32."""
    v = torch.randn(shape, generator=gen, device=DEV)
    if lowpass:
        f = torch.fft.rfftn(v)
        for ax, n in enumerate(shape):
            k = (torch.fft.rfftfreq(n, device=DEV) if ax == 2 else torch.fft.fftfreq(n, device=DEV))
            view = [1, 1, 1]
            view[ax] = -1
            f *= torch.exp(-2.0 * (math.pi * k) ** 2).view(view)
        v = torch.fft.irfftn(f, s=shape)
        v = v / v.std()
    t = tmpl.shape[0]
    amp = float((0.1 / tmpl[_mask(t) > 0].var()).sqrt())
    copies = min(300, max(1, int(np.prod(shape) / (8 * t ** 3))))
    rot = _sample(tmpl.double(), _rotations(_unit_quats(min(copies, 16), gen))).view(-1, t, t, t).float() * amp
    at = torch.rand(copies, 3, generator=gen, device=DEV).cpu().numpy()
    for i, a in enumerate(at):
        z, y, x = (int(a[k] * (shape[k] - t + 1)) for k in range(3))
        v[z:z + t, y:y + t, x:x + t] += rot[i % rot.shape[0]]
    return v.contiguous()


def _place(t_vol, shape):
    """[..., t, t, t] placed with its centre at the origin of a periodic grid."""
    t = t_vol.shape[-1]
    out = t_vol.new_zeros(t_vol.shape[:-3] + tuple(shape))
    out[..., :t, :t, :t] = t_vol
    return torch.roll(out, (-(t // 2),) * 3, dims=(-3, -2, -1))


def _normaliser(g, t):
    """w of Eq. 2 on the periodic grid of g (float64)."""
    m = _mask(t)
    M = float(m.sum())
    fm = torch.fft.rfftn(_place(m, g.shape)).conj()
    s1 = torch.fft.irfftn(torch.fft.rfftn(g) * fm, s=g.shape)
    s2 = torch.fft.irfftn(torch.fft.rfftn(g * g) * fm, s=g.shape)
    var = s2 - s1 * s1 / M
    keep = (var > 1e-8 * M * (g * g).mean()) & (var > 1e-10 * s2)
    return torch.where(keep, var.clamp_min(1e-300).rsqrt(), torch.zeros_like(var))


def _components(tomo, field, dtype):
    """C = w (g * T) on the periodic grid: [K, Z, Y, X] in dtype (the sums always in float64)."""
    shape = tuple(tomo.shape)
    g = _filter(tomo.double())
    w = _normaliser(g, field.shape[-1]).to(dtype)
    G = torch.fft.rfftn(g.to(dtype))
    out = torch.empty((field.shape[0],) + shape, dtype=dtype, device=DEV)
    for k in range(field.shape[0]):
        T = torch.fft.rfftn(_place(field[k].to(dtype), shape))
        out[k] = w * torch.fft.irfftn(G * T.conj(), s=shape)
    return out


def _probes(count, d):
    """Spread unit vectors (d = 3: spherical Fibonacci; d = 4: seeded), [d, count] float64."""
    if d == 4:
        return _unit_quats(count, _generator(7, 7)).T.contiguous()
    i = torch.arange(count, device=DEV, dtype=torch.float64)
    z = (i + 0.5) / count
    ph = math.pi * (3.0 - math.sqrt(5.0)) * i
    r = (1 - z * z).sqrt()
    return torch.stack([r * ph.cos(), r * ph.sin(), z])


def _weighted(u, n):
    mult = torch.tensor([_multinomial(e) for e in _exponents(n, u.shape[0])], dtype=u.dtype, device=DEV)
    return mult[:, None] * _monomials(u, n)


def _score_map(tomo, tmpl):
    """A score map of order 4 as the maximiser gives it, to the spacing of 64 directions (float32)."""
    C = _components(tomo, _field(tmpl, 4, 3), torch.float32)
    W = _weighted(_probes(64, 3), 4).float().T.contiguous()
    flat = C.view(C.shape[0], -1)
    return torch.cat([(W @ c).amax(0) for c in flat.split(1 << 22, dim=1)]).view(tomo.shape)


def _batch_shapes(case):
    r = np.random.RandomState(case["tomos"] * 1000 + case["lo"])
    return [tuple(int(v) for v in r.randint(case["lo"], case["hi"] + 1, 3)) for _ in range(case["tomos"])]


def _pairs(case, seed):
    """Unit-norm tensor components near planted axes and those axes: the network's training pairs."""
    n, N = case["n"], case["pairs"]
    gen = _generator(seed, 5)
    u = torch.randn(3, N, generator=gen, device=DEV)
    u = u / u.norm(dim=0)
    C = _monomials(u, n)
    C = C + 0.3 * C.std() * torch.randn(C.shape, generator=gen, device=DEV)
    mult = torch.tensor([_multinomial(e) for e in _exponents(n, 3)], dtype=C.dtype, device=DEV)
    C = C / (mult[:, None] * C * C).sum(0).sqrt()
    return C.T.contiguous(), u.T.contiguous()


@functools.lru_cache(maxsize=None)
def _context():
    return ttm.Context(0)  # a program keeps one


def _params(case):
    return ttm.params(order_n=case.get("n", 4), mask_radius=_radius(case["t"]), dprime=case.get("d", 3),
                      filter_a=FILTER_A, n_rot_base=8)


PREC = {"fp32": ttm.TTM_PREC_FP32, "fp16": ttm.TTM_PREC_FP16_SPECTRA, "bf16": ttm.TTM_PREC_BF16_SPECTRA}
SUMS = {"fp64": ttm.TTM_LOCALSUM_FP64, "df64": ttm.TTM_LOCALSUM_DF64}


def _plan(case, field, shape):
    plan = ttm.Plan(_context(), field, _params(case), shape, precision=PREC[case.get("prec", "fp32")])
    ttm.ttm_plan_set_localsum(plan, SUMS[case.get("sums", "fp64")])
    return plan


def _maps(shape, d):
    return {"score": torch.zeros(shape, device=DEV), "orient": torch.zeros((d,) + tuple(shape), device=DEV),
            "frob": torch.zeros(shape, device=DEV)}


def _volume(case, seed):
    """Template and tomogram of the single-tomogram kinds."""
    tmpl = _template(case["t"], _generator(seed, 1))
    return tmpl, _tomogram((case["Z"], case["Y"], case["X"]), tmpl, _generator(seed, 2), lowpass=case.get("n", 4) == 4)


def _refine_inputs(case, seed):
    """Peaks spread over the valid box and a quaternion map."""
    gen = _generator(seed, 3)
    t = case["t"]
    dims = [case["Z"], case["Y"], case["X"]]
    r = torch.rand(case["P"], 3, generator=gen, device=DEV, dtype=torch.float64).cpu().numpy()
    p = [t // 2 + (r[:, k] * (dims[k] - t + 1)).astype(np.int64) for k in range(3)]
    q = torch.randn(4, *dims, generator=gen, device=DEV)
    q = q / q.norm(dim=0)
    return (p[0] * dims[1] + p[1]) * dims[2] + p[2], (q * torch.where(q[0] < 0, -1.0, 1.0)).contiguous()


def _mlp_init(case):
    """Initial parameters N(0, 1 / fan_in), biases zero (one flat float32 array)."""
    K = len(_exponents(case["n"], 3))
    r = np.random.RandomState(17)
    parts = [r.standard_normal((128, K)) / math.sqrt(K), np.zeros(128), r.standard_normal((128, 128)) / math.sqrt(128),
             np.zeros(128), r.standard_normal((3, 128)) / math.sqrt(128), np.zeros(3)]
    return np.concatenate([p.ravel() for p in parts]).astype(np.float32)


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "mlp_train":
        st["X"], st["U"] = _pairs(case, seed)
        st["mlp"] = ttm.Mlp(_context(), st["X"].shape[1], seed=1)
        st["mlp"].set_precision(ttm.TTM_MLP_BF16 if case["prec"] == "bf16" else ttm.TTM_MLP_FP32)
        st["init"] = _mlp_init(case)
        return st
    if kind == "batch":
        st["tmpls"] = [_template(case["t"], _generator(seed, 10 + j)) for j in range(case["templates"])]
        fields = [_field(t, case["n"], 3) for t in st["tmpls"]]
        tomos = [_tomogram(s, st["tmpls"][i % len(fields)], _generator(seed, 50 + i), lowpass=False)
                 for i, s in enumerate(_batch_shapes(case))]
        pairs = [(i, j) for i in range(len(tomos)) for j in range(len(fields))]
        st["maps"] = [_maps(tomos[i].shape, 3) for i, _ in pairs]
        st["batch"] = ttm.Batch(_context(), _params(case), fields, tomos,
                                [(i, j, m["score"], m["orient"], m["frob"]) for (i, j), m in zip(pairs, st["maps"])],
                                n_branches=4, flags=ttm.TTM_BATCH_LOCALSUM_DF64 if case["sums"] == "df64" else 0)
        return st
    tmpl, tomo = _volume(case, seed)
    shape = tuple(tomo.shape)
    if kind == "find_peaks":
        st["map"] = _score_map(tomo, tmpl)
        st["plan"] = _plan({**case, "n": 2}, _field(tmpl, 2, 3), shape)
        return st
    n, d = case.get("n", 4), 4 if kind == "refine" else case.get("d", 3)
    field = _field(tmpl, n, d)
    K = field.shape[0]
    if kind == "blocked":
        st["tomo"] = torch.empty(shape, pin_memory=True).copy_(tomo)
        st["blocked"] = ttm.Blocked(_context(), field, _params(case), shape, case["slab"])
        return st
    if kind == "refine":
        # the plan after a correlate: refinement reads its filtered tomogram and normaliser
        st["plan"] = _plan({**case, "n": 2, "d": 4}, _field(tmpl, 2, 4), shape)
        st["tmpl"] = tmpl
        st["peaks"], st["orient"] = _refine_inputs(case, seed)
        ttm.ttm_correlate(st["plan"], tomo, torch.empty((10,) + shape, device=DEV))
        return st
    st["plan"] = _plan(case, field, shape)
    if kind == "peak_map":
        st["C"] = _components(tomo, field, torch.float32)
    else:
        st["tomo"] = tomo
        st["C"] = torch.empty((K,) + shape, device=DEV)
    if kind != "correlate":
        st["maps"] = _maps(shape, d)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "correlate":
        ttm.ttm_correlate(st["plan"], st["tomo"], st["C"])
        return {"C": st["C"]}
    if kind == "peak_map":
        m = st["maps"]
        ttm.ttm_peak_map(st["plan"], st["C"], m["score"], m["orient"], m["frob"])
        return m
    if kind == "match":
        m = st["maps"]
        ttm.ttm_correlate(st["plan"], st["tomo"], st["C"])
        ttm.ttm_peak_map(st["plan"], st["C"], m["score"], m["orient"], m["frob"])
        return {"C": st["C"], **m}
    if kind == "find_peaks":
        idx, val = ttm.ttm_find_peaks(st["plan"], st["map"], case["P"], 2.0 * _radius(case["t"]))
        return {"idx": idx, "val": val}
    if kind == "refine":
        idx, quat, lncc = ttm.ttm_refine_peaks(st["plan"], st["tmpl"], st["orient"], st["peaks"], case["rs"])
        return {"idx": idx, "quat": quat, "lncc": lncc}
    if kind == "batch":
        st["batch"].run()
        return st["maps"]
    if kind == "blocked":
        idx, val = st["blocked"].run(st["tomo"], case["P"], 2.0 * _radius(case["t"]))
        return {"idx": idx, "val": val}
    st["mlp"].set_params(st["init"])
    loss = st["mlp"].train(st["X"], st["U"], epochs=case["epochs"], batch=case["batch"], lr=1e-3, seed=3)
    return {"params": st["mlp"].get_params(), "loss": loss}


# ------------------------------------------------------------------- work --

def _shape_work(V, K, d, correlate, peak_map, n=4):
    b = f = 0.0
    if correlate:  # tomogram in, K components out; image, K inverse and 4 local-sum real transforms
        b += 4.0 * V * (1 + (0 if peak_map else K))
        f += (K + 5) * 2.5 * V * math.log2(V) + 4.0 * K * V
    if peak_map:   # components in, maps out; three evaluations of the value, gradient and Hessian
        b += 4.0 * V * (2 + d + (0 if correlate else K))
        f += 3.0 * V * 2 * len(_exponents(n - 2, d)) * (d * (d + 1) // 2)
    return b, f


def work(case):
    kind = case["kind"]
    n, d = case.get("n", 4), case.get("d", 3)
    K = len(_exponents(n, d))
    if kind == "mlp_train":
        rows = case["epochs"] * (case["pairs"] // case["batch"]) * case["batch"]
        return {"bytes": 4.0 * rows * (K + 3), "flops": 6.0 * rows * (128 * K + 128 * 128 + 128 * 3)}
    if kind == "batch":
        b = f = 0.0
        for s in _batch_shapes(case):
            x = _shape_work(float(np.prod(s)), K, 3, True, True, n)
            b, f = b + case["templates"] * x[0], f + case["templates"] * x[1]
        return {"bytes": b, "flops": f}
    V = float(case["Z"] * case["Y"] * case["X"])
    if kind == "find_peaks":
        return {"bytes": 4.0 * V, "flops": 26.0 * V}
    if kind == "refine":
        t, r = case["t"], int(case["rs"])
        cand = sum(1 for a in range(-r, r + 1) for b in range(-r, r + 1) for c in range(-r, r + 1)
                   if a * a + b * b + c * c <= case["rs"] ** 2)
        inside = 4.19 * _radius(t) ** 3
        return {"bytes": 4.0 * case["P"] * (t + 2 * r) ** 3 + 20.0 * case["P"] * cand,
                "flops": 40.0 * case["P"] * cand * inside}
    b, f = _shape_work(V, K, d, kind != "peak_map", kind != "correlate", n)
    if kind == "match":
        b += 4.0 * K * V  # the components are an output too
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ exact --

def _contract(C, u, n):
    """A_ij = sum_beta (n-2)!/beta! C_{e_i + e_j + beta} u^beta: dict of [V] for i <= j."""
    d = u.shape[0]
    where = {e: k for k, e in enumerate(_exponents(n, d))}
    beta = _exponents(n - 2, d)
    W = _monomials(u, n - 2) if n > 2 else torch.ones_like(u[:1])
    A = {}
    for i in range(d):
        for j in range(i, d):
            a = torch.zeros_like(u[0])
            for b, e in enumerate(beta):
                k = list(e)
                k[i] += 1
                k[j] += 1
                a.addcmul_(W[b], C[where[tuple(k)]], value=float(_multinomial(e)))
            A[i, j] = A[j, i] = a
    return A


def _apply(A, v):
    return torch.stack([sum(A[i, j] * v[j] for j in range(v.shape[0])) for i in range(v.shape[0])])


def _solve(H, g):
    """H x = g for symmetric H [V, d, d], g [V, d]."""
    if H.shape[1] != 3:
        return torch.linalg.solve_ex(H, g[:, :, None])[0][:, :, 0]
    h = H.unbind(1)
    c = [torch.linalg.cross(h[(i + 1) % 3], h[(i + 2) % 3]) for i in range(3)]
    return sum(c[i] * g[:, i:i + 1] for i in range(3)) / (h[0] * c[0]).sum(1, keepdim=True)


def _max_score(C, n, d):
    """max over unit u of C . u^n in float64, C [K, V]: starts from a dense probe set, then Riemannian Newton steps
    that are kept where the value does not fall, and shifted power steps elsewhere."""
    P = _probes(256 if d == 3 else 1024, d)
    W = _weighted(P, n).T.contiguous()
    near = (P.T @ P).abs() >= math.cos(math.radians(18.0))
    eye = torch.eye(d, dtype=C.dtype, device=DEV)
    out = torch.empty(C.shape[1], dtype=C.dtype, device=DEV)
    for s in range(0, C.shape[1], 1 << 18):
        c = C[:, s:s + (1 << 18)].contiguous()
        mult = torch.tensor([_multinomial(e) for e in _exponents(n, d)], dtype=C.dtype, device=DEV)
        F = (mult[:, None] * c * c).sum(0).sqrt()
        val = W @ c
        best = torch.full_like(F, -math.inf)
        for _ in range(4):
            top = val.argmax(0)
            val.masked_fill_(near[top].T, -math.inf)
            u = P[:, top].clone()
            A = _contract(c, u, n)
            Au = _apply(A, u)
            p = (u * Au).sum(0)
            for _ in range(10):
                # tangent gradient n (Au - p u); minus the Riemannian Hessian n p I - n (n-1) P A P, plus F u u^T
                M = torch.stack([torch.stack([A[i, j] for j in range(d)], -1) for i in range(d)], -2)
                Pu = eye - u.T[:, :, None] * u.T[:, None, :]
                H = n * p[:, None, None] * eye - n * (n - 1) * Pu @ M @ Pu
                H = H + (F[:, None, None] + 1e-300) * (u.T[:, :, None] * u.T[:, None, :])
                g = n * (Au - p * u)
                H = H + 1e-13 * F.clamp_min(1e-300)[:, None, None] * eye
                x = torch.nan_to_num(_solve(H, g.T).T)
                x = x * (0.3 / x.norm(dim=0).clamp_min(0.3))
                power = (Au + (n - 1) * F * u)
                for step in (u + x, power):
                    v = step / step.norm(dim=0).clamp_min(1e-300)
                    Av = _contract(c, v, n)
                    Avv = _apply(Av, v)
                    q = (v * Avv).sum(0)
                    ok = q >= p if step is not power else q > p
                    u, p, Au = torch.where(ok, v, u), torch.where(ok, q, p), torch.where(ok, Avv, Au)
                    A = {k: torch.where(ok, Av[k], A[k]) for k in A}
            best = torch.maximum(best, p)
        out[s:s + (1 << 18)] = torch.where(F > 0, best, torch.zeros_like(best))
    return out


def _frob(C, n, d):
    mult = torch.tensor([_multinomial(e) for e in _exponents(n, d)], dtype=torch.float64, device=DEV)
    out = torch.zeros(C.shape[1:], dtype=torch.float64, device=DEV)
    for k in range(C.shape[0]):
        out += mult[k] * C[k].double() ** 2
    return out.sqrt()


def _exact_maps(C, n, d, most):
    """Score (where it takes seconds, not minutes) and Frobenius norm; the maximising direction has no value of its own
    where two maxima tie."""
    V = C[0].numel()
    score = _max_score(C.double().view(C.shape[0], V), n, d).view(C.shape[1:]) if V <= most else None
    return {"score": score, "orient": None, "frob": _frob(C, n, d)}


def _greedy_peaks(score, P, min_dist):
    """Values of the P highest strict 26-neighbour maxima that keep min_dist."""
    top = torch.nn.functional.max_pool3d(score[None, None], 3, stride=1, padding=1)[0, 0]
    at = (score >= top).nonzero()
    order = score[at[:, 0], at[:, 1], at[:, 2]].argsort(descending=True)[: 100 * P]
    at = at[order].cpu().numpy()
    kept = np.zeros((0, 3))
    for p in at:
        if len(kept) == P:
            break
        if not len(kept) or ((kept - p) ** 2).sum(1).min() >= min_dist ** 2:
            kept = np.vstack([kept, p])
    k = torch.as_tensor(kept, dtype=torch.int64, device=DEV)
    return score[k[:, 0], k[:, 1], k[:, 2]]


def _box(shape, t):
    return tuple(slice(t // 2, s - (t - t // 2) + 1) for s in shape)


def _exact_refine(case, seed):
    tmpl, tomo = _volume(case, seed)
    peaks, orient = _refine_inputs(case, seed)
    t, rs = case["t"], case["rs"]
    g = _filter(tomo.double())
    w = _normaliser(g, t)
    tp = _normalised_template(tmpl)
    r = int(rs)
    offs = [(0, 0, 0)] + [(a, b, c) for a in range(-r, r + 1) for b in range(-r, r + 1) for c in range(-r, r + 1)
                          if (a, b, c) != (0, 0, 0) and a * a + b * b + c * c <= rs * rs]
    offs = torch.tensor(offs, device=DEV)
    box = _box(tomo.shape, t)
    dims = torch.tensor(tomo.shape, device=DEV)
    quat, lncc = [], []
    win = torch.arange(t, device=DEV) - t // 2
    for pk in peaks:
        z, y, x = pk // (dims[1] * dims[2]), (pk // dims[2]) % dims[1], pk % dims[2]
        at = torch.stack([z, y, x]) + offs
        ok = torch.ones(len(at), dtype=torch.bool, device=DEV)
        for k in range(3):
            ok &= (at[:, k] >= box[k].start) & (at[:, k] < box[k].stop)
        at = at[ok]
        q = orient[:, at[:, 0], at[:, 1], at[:, 2]].T.double()
        s = _sample(tp, _rotations(q))
        iz, iy, ix = (at[:, k, None] + win for k in range(3))
        gw = g[iz[:, :, None, None], iy[:, None, :, None], ix[:, None, None, :]].view(len(at), -1)
        c = w[at[:, 0], at[:, 1], at[:, 2]] * (s * gw).sum(1)
        b = int(c.argmax())
        quat.append(q[b])
        lncc.append(c[b])
    return {"idx": None, "quat": torch.stack(quat), "lncc": torch.stack(lncc)}


def _splitmix(z):
    z = (z + np.uint64(0x9E3779B97F4A7C15))
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def _exact_train(case, seed):
    """Mlp.train in float64: the documented SplitMix64 permutation, Adam, mean loss."""
    X, U = (v.double() for v in _pairs(case, seed))
    N, K = X.shape
    B = min(case["batch"], N)
    p = torch.as_tensor(_mlp_init(case), device=DEV).double()
    sizes = [(128, K), (128,), (128, 128), (128,), (3, 128), (3,)]
    m, v, step, last = torch.zeros_like(p), torch.zeros_like(p), 0, 0.0
    for ep in range(case["epochs"]):
        with np.errstate(over="ignore"):
            i = np.arange(N, dtype=np.uint64)
            u = (_splitmix(np.uint64(3 + 17 + ep) ^ (i * np.uint64(0xD1B54A32D192ED03))) >> np.uint64(11)) * 2.0 ** -53
        pick = np.minimum((u * (np.arange(N) + 1.0)).astype(np.int64), np.arange(N)).tolist()
        perm = list(range(N))
        for k in range(N - 1, 0, -1):
            perm[k], perm[pick[k]] = perm[pick[k]], perm[k]
        perm = torch.tensor(perm, device=DEV)
        for s in range(0, N - B + 1, B):
            x, us = X[perm[s:s + B]], U[perm[s:s + B]]
            q = p.clone().requires_grad_()
            w1, b1, w2, b2, w3, b3 = (t.view(z) for t, z in zip(q.split([int(np.prod(z)) for z in sizes]), sizes))
            h = torch.nn.functional.gelu(x @ w1.T + b1, approximate="tanh")
            h = torch.nn.functional.gelu(h @ w2.T + b2, approximate="tanh")
            y = h @ w3.T + b3
            loss = (1 - ((y / y.norm(dim=1, keepdim=True)) * us).sum(1) ** 2).mean()
            g, = torch.autograd.grad(loss, q)
            step += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 1e-3 * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
            last = loss.detach()
    return {"params": p, "loss": last}


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp_train":
        return _exact_train(case, seed)
    if kind == "find_peaks":
        return None  # indices and copies of the map's own values
    if kind == "refine":
        return _exact_refine(case, seed)
    n, d = case["n"], case.get("d", 3)
    if kind == "batch":
        tmpls = [_template(case["t"], _generator(seed, 10 + j)) for j in range(case["templates"])]
        out = []
        for i, s in enumerate(_batch_shapes(case)):
            tomo = _tomogram(s, tmpls[i % len(tmpls)], _generator(seed, 50 + i), lowpass=False)
            for t in tmpls:
                box = _box(s, case["t"])
                C = _components(tomo, _field(t, n, 3), torch.float64)[(slice(None),) + box]
                whole = {"orient": None}
                for k, v in _exact_maps(C.contiguous(), n, 3, 1 << 22).items():
                    if v is not None:
                        whole[k] = torch.zeros(s, dtype=torch.float64, device=DEV)
                        whole[k][box] = v
                    else:
                        whole[k] = None
                out.append(whole)
        return out
    tmpl, tomo = _volume(case, seed)
    field = _field(tmpl, n, d)
    if kind == "peak_map":
        return _exact_maps(_components(tomo, field, torch.float32), n, d, 1 << 22 if d == 3 else 1 << 20)
    C = _components(tomo, field, torch.float64)
    if kind == "correlate":
        return {"C": C}
    if kind == "match":
        return {"C": C, **_exact_maps(C, n, d, 1 << 22)}
    box = _box(tomo.shape, case["t"])
    C = C[(slice(None),) + box].contiguous()
    if C[0].numel() > 1 << 22:
        return None  # the 64-bit maxima of every voxel would take too long
    score = _max_score(C.view(C.shape[0], -1), n, d).view(C.shape[1:])
    return {"idx": None, "val": _greedy_peaks(score, case["P"], 2.0 * _radius(case["t"]))}
