"""The work a user of this library has it do, as cases that can be timed.

A case is one call of the public binding (`paper_2110_10156_gb300.cs_ngf`) on a
volume pair:

  align    best (score, rotation, shift) over R rotations of a prepared pair
  score    best score and shift of every rotation
  host     the same from host arrays, copies inside the call
  map      a new fixed volume, then the score map of one rotation over all shifts
  search   the paper's pyramid search of a pair, nothing prepared

`prepare` makes the pair and, except for `search`, the handle with the fixed
volume's spectra that a program keeps while it scores floating volumes.
"""
import math

import numpy as np
import torch

from paper_2110_10156_gb300 import cs_ngf

GAMMA, EPS = 0.5, 1e-5


def _case(name, op, dims, rotations, masks="threshold", precision="fp32", measure="squared", pad_mode="bound"):
    nz, ny, nx = dims
    c = dict(op=op, nz=nz, ny=ny, nx=nx, rotations=rotations, masks=masks, precision=precision,
             measure=measure, pad_mode=pad_mode)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # the smallest pair of the configurations: a few candidate rotations of a
        # 32^3 patch without masks, where launches and waits are the cost
        _case("align_32", "align", (32, 32, 32), 8, masks="full"),
        # one evaluation of a small ragged patch pair, both volumes new
        _case("map_31x37x29", "map", (31, 37, 29), 1),
        # one all-shift evaluation of a pair at the largest side of the paper's
        # run-time table, both volumes new
        _case("map_128", "map", (128, 128, 128), 1),
        # the small job of the serving mix
        _case("align_64", "align", (64, 64, 64), 200),
        # an anisotropic scan of the serving mix, from host memory
        _case("host_96x128x128", "host", (96, 128, 128), 64),
        # the headline workload: 150^3 brain-sized block, 1000 rotations
        _case("align_150", "align", (150, 150, 150), 1000),
        # the same block in the BF16 form (tensor-core z pass)
        _case("align_150_bf16", "align", (150, 150, 150), 300, precision="bf16"),
        # odd sides in the FP16 form
        _case("align_151x137x122_fp16", "align", (151, 137, 122), 120, precision="fp16"),
        # the unsquared measure on a pair without masks: every shift down to
        # half overlap is admitted on every axis
        _case("score_unsquared_110x96x101", "score", (110, 96, 101), 40, masks="full", measure="unsquared"),
        # full linear-correlation padding for every rotation, every rotation's result
        _case("score_padfull_120x144x132", "score", (120, 144, 132), 48, pad_mode="full"),
        # the largest supported volume
        _case("align_256", "align", (256, 256, 256), 256),
        # the whole alignment with the paper's schedule (8325 rotations on four levels)
        _case("search_150", "search", (150, 150, 150), 8325),
    ]


def draw(rng):
    """Sides log-uniform in [24, 224] with a spread of up to 1.4 between axes,
    odd ones among them; rotations log-uniform in [1, 600], bounded so that no
    case costs more than the largest listed one."""
    op = rng.choice(["align", "align", "align", "score", "host", "map"])
    base = math.exp(rng.uniform(math.log(24), math.log(224)))
    dims = tuple(max(16, min(256, int(round(base * math.exp(rng.uniform(-0.17, 0.17)))))) for _ in range(3))
    vox = dims[0] * dims[1] * dims[2]
    precision = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp16"]) if op in ("align", "map") else "fp32"
    most = max(1, min(600, int(2.0e9 / vox)))
    if op in ("score", "host"):
        most = min(most, 64)
    rotations = 1 if op == "map" else int(round(math.exp(rng.uniform(0.0, math.log(most)))))
    return _case("", op, dims, max(1, rotations), masks=rng.choice(["threshold", "threshold", "full"]),
                 precision=precision, measure=rng.choice(["squared", "squared", "squared", "unsquared"]),
                 pad_mode=rng.choice(["bound", "bound", "bound", "full"]))


# ----------------------------------------------------------------- inputs
def _matrix(q):
    w, x, y, z = (float(v) / math.sqrt(sum(float(u) ** 2 for u in q)) for v in q)
    return np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                     [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                     [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])


def _quaternions(rng, k):
    """Uniform random unit quaternions (w, x, y, z), w >= 0."""
    q = rng.normal(size=(k, 4))
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    q[q[:, 0] < 0] *= -1.0
    return q


def _axes(dims, device):
    return [torch.arange(n, dtype=torch.float32, device=device) for n in dims]


def _blur(v, sigma):
    r = int(4 * sigma + 0.5)
    k = torch.exp(-0.5 * (torch.arange(-r, r + 1, dtype=torch.float32, device=v.device) / sigma) ** 2)
    k = k / k.sum()
    for axis in range(3):
        n = v.shape[axis]
        idx = torch.arange(n, device=v.device)
        out = torch.zeros_like(v)
        for j in range(2 * r + 1):
            out += k[j] * v.index_select(axis, (idx + (j - r)).clamp(0, n - 1))
        v = out
    return v


def _moved(v, R, t):
    """out(y) = v(R^T (y - c) + c - t), trilinear, zero outside; t in (x, y, z)."""
    nz, ny, nx = v.shape
    z, y, x = _axes(v.shape, v.device)
    c = [(nx - 1) / 2, (ny - 1) / 2, (nz - 1) / 2]
    d = [(x - c[0])[None, None, :], (y - c[1])[None, :, None], (z - c[2])[:, None, None]]
    p = [R[0][i] * d[0] + R[1][i] * d[1] + R[2][i] * d[2] + (c[i] - float(t[i])) for i in range(3)]
    g = torch.stack([2 * p[i] / (n - 1) - 1 for i, n in enumerate((nx, ny, nz))], dim=-1)
    return torch.nn.functional.grid_sample(v[None, None], g[None], mode="bilinear", padding_mode="zeros",
                                           align_corners=True)[0, 0]


def _pair(case, seed):
    """A brain-like pair: A a blurred sum of ellipsoids around the middle, B the
    same moved by a known rotation and shift, through a non-monotone intensity
    map, with noise; masks are the foreground, or everything; rotations are
    uniform with the true one among them."""
    dims = (case["nz"], case["ny"], case["nx"])
    dev = torch.device("cuda")
    rng = np.random.default_rng([7, int(seed)])
    side = max(dims)
    z, y, x = _axes(dims, dev)
    A = torch.zeros(dims, device=dev)
    for q in _quaternions(rng, 32):
        R = _matrix(q)
        centre = rng.uniform(0.25, 0.75, size=3) * np.array(dims[::-1])
        radii = rng.uniform(side / 30, side / 5, size=3)
        level = float(rng.uniform())
        d = [(x - centre[0])[None, None, :], (y - centre[1])[None, :, None], (z - centre[2])[:, None, None]]
        s = sum(((R[0][i] * d[0] + R[1][i] * d[1] + R[2][i] * d[2]) / radii[i]) ** 2 for i in range(3))
        A += level * (s <= 1.0)
    A = _blur(A, max(1.0, side / 75))
    axis = rng.normal(size=3)
    axis /= np.linalg.norm(axis)
    half = 0.5 * math.radians(rng.uniform(9.0, 30.0))
    q_true = np.array([math.cos(half), *(math.sin(half) * axis)])
    most = max(1, min(20, side // 7))
    t = rng.integers(-most, most + 1, size=3)
    R = _matrix(q_true)
    Bg = _moved(A, R, t)
    lo, hi = float(Bg.min()), float(Bg.max())
    knots = torch.tensor(np.concatenate([rng.uniform(size=8), [0.0]]), dtype=torch.float32, device=dev)
    u = ((Bg - lo) / max(hi - lo, 1e-6) * 7).clamp(0, 7)
    i = u.floor().long().clamp(max=6)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 2 + 1)
    B = torch.lerp(knots[i], knots[i + 1], u - i) + 0.01 * torch.randn(dims, generator=gen, device=dev)
    if case["masks"] == "full":
        MA = torch.ones(dims, dtype=torch.uint8, device=dev)
        MB = MA.clone()
    else:
        MA = (A > 0.05 * A.max()).to(torch.uint8)
        MB = (_moved(MA.float(), R, t) > 0.5).to(torch.uint8)
    quats = _quaternions(rng, case["rotations"])
    quats[int(rng.integers(0, len(quats)))] = q_true
    return A.contiguous(), MA, B.contiguous(), MB, quats


# ----------------------------------------------------------------- the calls
def prepare(case, seed):
    A, MA, B, MB, quats = _pair(case, seed)
    s = dict(op=case["op"], A=A, MA=MA, B=B, MB=MB, quats=quats, measure=case["measure"], seed=int(seed))
    if case["op"] != "search":
        s["fixed"] = cs_ngf.prepare_fixed(A, MA, eps=EPS, gamma=GAMMA, measure=case["measure"],
                                          precision=case["precision"], pad_mode=case["pad_mode"])
    if case["op"] == "host":
        s["B"], s["MB"] = B.cpu().numpy(), MB.cpu().numpy()
    return s


def run(s):
    op = s["op"]
    if op == "search":
        return cs_ngf.global_align(s["A"], s["MA"], s["B"], s["MB"], seed=s["seed"], eps=EPS, gamma=GAMMA,
                                   measure=s["measure"])
    f = s["fixed"]
    if op == "align":
        return f.align(s["B"], s["MB"], s["quats"])
    if op == "score":
        return f.score_rotations(s["B"], s["MB"], s["quats"])
    if op == "host":
        return f.score_rotations_host(s["B"], s["MB"], s["quats"])
    f.update_fixed(s["A"], s["MA"])
    return f.score_map(s["B"], s["MB"], s["quats"][0])


def work(case):
    """Bytes: every input and result once.  Flops: per rotation the real
    transforms of the channels (six, or three unsquared) and the mask, and the
    two inverse ones (numerator and overlap), at no more than the volume's own
    size; a map also transforms the fixed volume."""
    vox = case["nz"] * case["ny"] * case["nx"]
    R = case["rotations"]
    one = 2.5 * vox * math.log2(vox)
    fwd = (3 if case["measure"] == "unsquared" else 6) + 1
    out = 16 * R
    if case["op"] == "map":
        out = 4 * (2 * case["nz"] - 1) * (2 * case["ny"] - 1) * (2 * case["nx"] - 1)
    if case["op"] == "search":      # 5001 rotations at 1/64 of the voxels, 3323 at 1/8, one or more in full
        return dict(bytes=10.0 * vox, flops=(5001 / 64 + 3323 / 8 + 3) * (fwd + 2) * one)
    vols = 2 if case["op"] == "map" else 1
    return dict(bytes=5.0 * vols * vox + 32.0 * R + out, flops=(R * (fwd + 2) + (fwd if vols == 2 else 0)) * one)


# ----------------------------------------------------------------- 64 bits
def _rotated(B, MB, q):
    """B at R (x - c) + c by trilinear interpolation in 64 bits, and the rotated
    mask [trilinear mask >= 1/2].  The sample point and the mask decision are
    defined in round-to-nearest 32-bit steps, so they are taken in those."""
    R = _matrix(q)
    for v in (-1.0, 0.0, 1.0):
        R[np.abs(R - v) <= 1e-9] = v
    R = R.astype(np.float32)
    nz, ny, nx = B.shape
    f32 = lambda v: torch.tensor(float(v), dtype=torch.float32, device=B.device)
    z, y, x = _axes(B.shape, B.device)
    c = [f32((nx - 1) / 2), f32((ny - 1) / 2), f32((nz - 1) / 2)]
    d = [(x - c[0])[None, None, :], (y - c[1])[None, :, None], (z - c[2])[:, None, None]]
    i0, t, inside = [], [], None
    for i, n in enumerate((nx, ny, nz)):
        a = f32(R[i, 0]) * d[0]
        a = a + f32(R[i, 1]) * d[1]
        a = a + f32(R[i, 2]) * d[2]
        p = a + c[i]
        slack = f32(1e-4)
        ok = (p >= -slack) & (p <= f32(n - 1) + slack)
        inside = ok if inside is None else inside & ok
        p = p.clamp(0.0, float(n - 1))
        k = p.floor().long().clamp(max=n - 2)
        i0.append(k)
        t.append(p - k.float())
    base = (i0[2] * ny + i0[1]) * nx + i0[0]
    corner = lambda v, dz, dy, dx: v.reshape(-1)[base + (dz * ny + dy) * nx + dx]
    lerp = lambda a, b, w: a + w * (b - a)
    V, M, td = B.double(), MB.float(), [w.double() for w in t]
    val, m = [], []
    for dz in (0, 1):
        val.append(lerp(lerp(corner(V, dz, 0, 0), corner(V, dz, 0, 1), td[0]),
                        lerp(corner(V, dz, 1, 0), corner(V, dz, 1, 1), td[0]), td[1]))
        m.append(lerp(lerp(corner(M, dz, 0, 0), corner(M, dz, 0, 1), t[0]),
                      lerp(corner(M, dz, 1, 0), corner(M, dz, 1, 1), t[0]), t[1]))
    Bh = torch.where(inside, lerp(val[0], val[1], td[2]), torch.zeros((), dtype=torch.float64, device=B.device))
    return Bh, (inside & (lerp(m[0], m[1], t[2]) >= 0.5)).double()


def _channels(V, M, measure):
    g = []
    for axis in (2, 1, 0):
        n = V.shape[axis]
        i = torch.arange(n, device=V.device)
        g.append((V.index_select(axis, (i + 1).clamp(max=n - 1)) - V.index_select(axis, (i - 1).clamp(min=0))) / 2)
    eps = float(np.float32(EPS)) ** 2
    inv = M / torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2 + eps)
    g = [v * inv for v in g]
    if measure == "unsquared":
        return [(1.0, v) for v in g]
    return [(1.0 if i == j else 2.0, g[i] * g[j]) for i in range(3) for j in range(i, 3)]


def _exact_map(fixed, fft, Bh, Mh, sum_a, dims, measure):
    acc = None
    for (w, a), (_, b) in zip(fixed[:-1], _channels(Bh, Mh, measure)):
        term = w * a.conj() * torch.fft.rfftn(b, s=fft)
        acc = term if acc is None else acc + term
    X = torch.fft.irfftn(acc, s=fft)
    N = torch.fft.irfftn(fixed[-1][1].conj() * torch.fft.rfftn(Mh, s=fft), s=fft)
    for axis, (n, p) in enumerate(zip(dims, fft)):
        k = torch.arange(-(n - 1), n, device=X.device) % p
        X, N = X.index_select(axis, k), N.index_select(axis, k).round()
    need = max(1, math.ceil(GAMMA * min(sum_a, int(Mh.sum()))))
    return torch.where(N >= need, X / N.clamp(min=1.0), torch.full((), -math.inf, dtype=torch.float64, device=X.device))


def _best(m, dims):
    k = int(m.argmax())
    score = float(m.reshape(-1)[k])
    if not math.isfinite(score):
        return score, (0, 0, 0)
    at = np.unravel_index(k, tuple(m.shape))
    return score, tuple(int(i) - (n - 1) for i, n in zip(at, dims))


def exact(case, seed):
    dims = (case["nz"], case["ny"], case["nx"])
    fft = tuple(2 * n for n in dims)
    if case["op"] == "search" or case["rotations"] * fft[0] * fft[1] * fft[2] > 9.0e8:
        return None
    A, MA, B, MB, quats = _pair(case, seed)
    measure = case["measure"]
    ma = (MA != 0).double()
    fixed = [(w, torch.fft.rfftn(c, s=fft)) for w, c in _channels(A.double(), ma, measure)]
    fixed.append((1.0, torch.fft.rfftn(ma, s=fft)))
    if case["op"] == "map":
        return _exact_map(fixed, fft, *_rotated(B, MB, quats[0]), int(ma.sum()), dims, measure)
    best = [_best(_exact_map(fixed, fft, *_rotated(B, MB, q), int(ma.sum()), dims, measure), dims) for q in quats]
    if case["op"] == "align":
        r = int(np.argmax([b[0] for b in best]))
        return best[r][0], r, best[r][1]
    return (np.array([b[0] for b in best]), np.array([b[1] for b in best], dtype=np.int64))
