"""Performance cases of the alignment library: what a user's program has it do.

A case is one call (or one pass of calls) through the public entry points of
``paper_2011_05755_gb300`` on synthetic particle stacks: blob references,
particles that are rotated, shifted, mirrored and noisy copies of them.

``op`` says what one pass does:

* ``align``: poses of a stack against the references that the handle holds
  (what the serving loop does for each batch);
* ``classify``: one pass of the classification loop: new references in,
  align, class averages, reference refresh;
* ``graph``: the same pass without the refresh as one ``mra_run_graph`` call;
* ``host``: the same pass from pinned host buffers (``mra_run_host``);
* ``average``: class averages of a stack from given poses.
"""
import math

import torch

import paper_2011_05755_gb300 as mra

PRECISION = {"fp32": mra.MRA_FP32, "bf16": mra.MRA_BF16_RESCORE, "fp16": mra.MRA_FP16_RESCORE}


def _case(op, precision, n, L, K, last, shift, step=1.0, first=1, ring_step=1, mirror=1, snr=0.1):
    return {"op": op, "precision": precision, "n": n, "L": L, "K": K, "first_ring": first, "last_ring": last,
            "ring_step": ring_step, "shift_range": float(shift), "shift_step": float(step), "mirror": mirror,
            "snr": float(snr)}


def listed():
    named = [
        # one new particle against a resident reference set (an interactive call): launches and latency
        ("align_1_L64_K50_bf16", _case("align", "bf16", 1, 64, 50, 28, 3)),
        # the smallest request of the serving stream
        ("align_200_L76_K100_bf16", _case("align", "bf16", 200, 76, 100, 34, 3)),
        # an ordinary request of the serving stream, M = 512, in FP16
        ("align_1500_L96_K200_fp16", _case("align", "fp16", 1500, 96, 200, 44, 3)),
        # a small binned box on a half-pixel grid, K not a tile multiple, M = 128
        ("align_5003_L32_K11_half_bf16", _case("align", "bf16", 5003, 32, 11, 12, 1.5, 0.5)),
        # part of the benchmark stack: the whole pass as one graph launch
        ("graph_12000_L76_K100_bf16", _case("graph", "bf16", 12000, 76, 100, 35, 4)),
        # the large-box workload
        ("graph_600_L128_K200_bf16", _case("graph", "bf16", 600, 128, 200, 60, 6, snr=0.05)),
        # a pass of the classification loop with many classes
        ("classify_6000_L76_K500_bf16", _case("classify", "bf16", 6000, 76, 500, 35, 3)),
        # end to end from host memory
        ("host_2000_L76_K100_bf16", _case("host", "bf16", 2000, 76, 100, 35, 4)),
        # the small workload, and part of the benchmark stack, on the FP32 path
        ("align_500_L76_K10_fp32", _case("align", "fp32", 500, 76, 10, 35, 2)),
        ("classify_1200_L76_K100_fp32", _case("classify", "fp32", 1200, 76, 100, 35, 4)),
        # reference-free alignment: one common reference, 90-pixel particles
        ("align_3000_L90_K1_fp32", _case("align", "fp32", 3000, 90, 1, 36, 3)),
        # class averages of a stack whose poses are known
        ("average_30000_L76_K100", _case("average", "fp32", 30000, 76, 100, 35, 4)),
    ]
    return [dict(c, name=name) for name, c in named]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["m256", "m256", "m256", "m512", "small", "fp32", "one_ref", "average"])
    op = rng.choice(["align", "align", "classify", "graph", "host"])
    precision = rng.choice(["bf16", "bf16", "fp16"])
    first, ring_step, step = rng.choice([1, 1, 1, 2, 3]), 1, 1.0
    mirror = rng.choice([1, 1, 1, 0])
    K = _log_int(rng, 5, 500)
    shift = rng.randint(1, 5)
    if kind == "m256":  # rings up to 21..40
        L = 2 * rng.randint(29, 46)
        last = min(40, L // 2 - rng.randint(4, 6))
    elif kind == "m512":  # rings up to 41..60
        L = 2 * rng.randint(46, 64)
        last = max(41, L // 2 - 4)
        K = _log_int(rng, 5, 200)
    elif kind == "small":
        L = 2 * rng.randint(12, 24)
        last = L // 2 - 3
        if rng.random() < 0.5:
            shift, step = rng.choice([1.0, 1.5, 2.0]), 0.5
    else:
        L = 2 * rng.randint(16, 50)
        last = L // 2 - rng.randint(4, 6)
        precision = "fp32"
        ring_step = rng.choice([1, 1, 2])
        if kind == "one_ref":
            K, op = 1, "align"
        elif kind == "average":
            op = "average"
    c = _case(op, precision, 1, L, K, last, shift, step, first, ring_step, mirror)
    if op == "average":
        c["n"] = _log_int(rng, 200, 30000)
        return c
    # the number of images: log-uniform up to what costs no more than the largest listed case
    largest = max(work(x)["flops"] for x in listed())
    per_image = work(dict(c, n=1001))["flops"] - work(dict(c, n=1))["flops"]
    most = largest / 3 / (per_image / 1000) / (3 if precision == "fp32" else 2 if last > 40 else 1)
    c["n"] = _log_int(rng, 1, max(2, min(20000, int(most))))
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _blobs(cx, cy, sigma, amp, L):
    """Sums of isotropic Gaussians on the pixel grid, [B, L, L]."""
    grid = torch.arange(L, dtype=torch.float32, device=cx.device) - L / 2
    inv = (0.5 / (sigma * sigma))[..., None]
    ex = torch.exp(-(grid - cx[..., None]) ** 2 * inv)
    ey = torch.exp(-(grid - cy[..., None]) ** 2 * inv) * amp[..., None]
    return torch.bmm(ey.transpose(1, 2), ex)


def _standard(x):
    m = x.mean(dim=(1, 2), keepdim=True)
    return (x - m) / (x - m).square().mean(dim=(1, 2), keepdim=True).sqrt()


def _inputs(case, seed):
    """References [K, L, L], particles [n, L, L] and their true classes, on the GPU."""
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(seed)
    n, L, K, G = case["n"], case["L"], case["K"], 20

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=g, device=dev)

    sigma, amp = uniform(0.04 * L, 0.105 * L, K, G), uniform(0.5, 1.5, K, G)
    rho, psi = 0.37 * L * uniform(0, 1, K, G).sqrt(), uniform(0, 2 * math.pi, K, G)
    cx, cy = rho * psi.cos(), rho * psi.sin()
    refs = _standard(_blobs(cx, cy, sigma, amp, L)).contiguous()
    k = torch.randint(0, K, (n,), generator=g, device=dev)
    alpha = uniform(0, 2 * math.pi, n, 1)
    T = int(case["shift_range"])
    t = torch.randint(-T, T + 1, (n, 2), generator=g, device=dev).float()
    sign = 1.0 - 2.0 * torch.randint(0, 2, (n, 1), generator=g, device=dev) * case["mirror"]
    imgs = torch.empty((n, L, L), dtype=torch.float32, device=dev)
    for b in range(0, n, 4096):
        s = slice(b, min(n, b + 4096))
        kk = k[s]
        x = sign[s] * (alpha[s].cos() * cx[kk] - alpha[s].sin() * cy[kk] + t[s, :1])
        y = alpha[s].sin() * cx[kk] + alpha[s].cos() * cy[kk] + t[s, 1:]
        img = _standard(_blobs(x, y, sigma[kk], amp[kk], L))
        noise = torch.randn(img.shape, generator=g, device=dev)
        imgs[s] = _standard(img + noise * case["snr"] ** -0.5)
    return refs, imgs, k


def _given_poses(case, k, seed):
    """Pose rows (mra_pose_t) with the true classes and random shifts, angles and mirrors."""
    n, nx = case["n"], _axis(case)
    g = torch.Generator(device=k.device).manual_seed(seed + 1)
    p = torch.zeros((n, 8), dtype=torch.int32, device=k.device)
    p[:, 0] = k
    p[:, 1] = torch.randint(0, _angles(case), (n,), generator=g, device=k.device)
    p[:, 2] = torch.randint(0, 2, (n,), generator=g, device=k.device) * case["mirror"]
    p[:, 3] = torch.randint(0, nx * nx, (n,), generator=g, device=k.device)
    f = p.view(torch.float32)
    f[:, 4] = p[:, 1] * (360.0 / _angles(case))
    f[:, 5] = (p[:, 3] % nx) * case["shift_step"] - case["shift_range"]
    f[:, 6] = (p[:, 3] // nx) * case["shift_step"] - case["shift_range"]
    return p


def prepare(case, seed):
    refs, imgs, k = _inputs(case, seed)
    n, L, K = case["n"], case["L"], case["K"]
    al = mra.Aligner(L, case["first_ring"], case["last_ring"], case["ring_step"], case["shift_range"],
                     case["shift_step"], case["mirror"], PRECISION[case["precision"]])
    s = {"op": case["op"], "al": al, "refs": refs, "imgs": imgs,
         "poses": torch.zeros((n, 8), dtype=torch.int32, device=imgs.device),
         "avg": torch.zeros((K, L, L), dtype=torch.float32, device=imgs.device),
         "counts": torch.zeros((K,), dtype=torch.int32, device=imgs.device)}
    if case["op"] in ("align", "average"):
        al.set_refs(refs)
    if case["op"] == "average":
        s["poses"] = _given_poses(case, k, seed)
    if case["op"] == "host":
        for name in ("refs", "imgs", "poses", "avg", "counts"):
            s[name] = s[name].cpu().pin_memory()
    return s


def run(s):
    al, imgs, poses, avg, counts = s["al"], s["imgs"], s["poses"], s["avg"], s["counts"]
    if s["op"] == "align":
        al.align(imgs, poses)
        return _poses_out(poses)
    if s["op"] == "average":
        al.average(imgs, poses, avg, counts)
        return {"avg": avg, "counts": counts}
    if s["op"] == "graph":
        mra.mra_run_graph(al.h, s["refs"], imgs, poses, avg, counts)
    elif s["op"] == "host":
        mra.mra_run_host(al.h, s["refs"], imgs, poses, avg, counts)
    else:
        al.set_refs(s["refs"])
        al.align(imgs, poses)
        avg.copy_(s["refs"])  # a class that stays empty keeps its reference
        al.average(imgs, poses, avg, counts)
        mra.mra_refresh_refs(al.h, avg, counts)
    return dict(_poses_out(poses), avg=avg, counts=counts)


def _poses_out(poses):
    """mra_pose_t rows as their whole-number and floating fields (views)."""
    return {"pose": poses[:, :4], "geometry": poses.view(torch.float32)[:, 4:]}


# --------------------------------------------------------------------------
# sizes and work
# --------------------------------------------------------------------------
def _rings(case):
    out = []
    for r in range(case["first_ring"], case["last_ring"] + 1, case["ring_step"]):
        N = 1
        while N < 2 * math.pi * r:
            N *= 2
        out.append((r, N))
    return out


def _angles(case):
    return max(N for _, N in _rings(case))


def _axis(case):
    return int(round(2 * case["shift_range"] / case["shift_step"])) + 1


def work(case):
    n, L, K, S = case["n"], case["L"], case["K"], _axis(case) ** 2
    rings, M = _rings(case), _angles(case)
    image, poses = 4 * L * L, 32 * n
    if case["op"] == "average":
        return {"bytes": n * image + poses + K * image + 4 * K, "flops": n * L * L * 20}
    bins = sum(N // 2 + 1 for _, N in rings)
    pair = 8 * bins + 5 * M * math.log2(M)  # contraction and inverse DFT of one (image, shift, reference)
    row = sum(2.5 * N * math.log2(N) + 9 * N for _, N in rings)  # resampling and ring FFTs of one (image, shift)
    w = {"bytes": n * image + K * image + poses, "flops": n * S * (K * pair + row)}
    if case["op"] != "align":
        w["bytes"] += K * image + 4 * K
        w["flops"] += n * L * L * 20
    return w


# --------------------------------------------------------------------------
# the same in 64 bits
# --------------------------------------------------------------------------
def _sample(imgs, x, y):
    """Bilinear samples of imgs [B, L, L] at x, y ([P] or [B, P]), zero outside: [B, P]."""
    B, L = imgs.shape[0], imgs.shape[-1]
    padded = torch.nn.functional.pad(imgs, (1, 1, 1, 1)).reshape(B, -1)
    x0, y0 = x.floor(), y.floor()
    fx, fy = x - x0, y - y0
    out = 0
    for dx, dy, w in ((0, 0, (1 - fx) * (1 - fy)), (1, 0, fx * (1 - fy)), (0, 1, (1 - fx) * fy), (1, 1, fx * fy)):
        xi, yi = (x0 + dx).long().clamp(-1, L) + 1, (y0 + dy).long().clamp(-1, L) + 1
        i = (yi * (L + 2) + xi).expand(B, -1)
        out = out + w * padded.gather(1, i)
    return out


def _spectra(imgs, case, sx, sy, M):
    """Ring spectra of imgs at one shift: complex [B, rings, M / 2 + 1], zero above each ring's N / 2."""
    c0, rings = imgs.shape[-1] / 2, _rings(case)
    out = torch.zeros((imgs.shape[0], len(rings), M // 2 + 1), dtype=torch.complex128, device=imgs.device)
    for i, (r, N) in enumerate(rings):
        th = torch.arange(N, dtype=torch.float64, device=imgs.device) * (2 * math.pi / N)
        out[:, i, : N // 2 + 1] = torch.fft.rfft(_sample(imgs, c0 + sx + r * th.cos(), c0 + sy + r * th.sin()))
    return out


def _exact_poses(case, refs, imgs):
    n, K, M, nx = case["n"], case["K"], _angles(case), _axis(case)
    S, H = nx * nx, M // 2
    rings, dev = _rings(case), imgs.device
    w = torch.zeros((len(rings), H + 1), dtype=torch.float64, device=dev)
    for i, (r, N) in enumerate(rings):
        w[i, : N // 2 + 1] = 2 * math.pi * r * case["ring_step"] / (N * N)
        if N < M:
            w[i, N // 2] *= 0.5
    Y = _spectra(refs, case, 0.0, 0.0, M) * w
    first = [next(i for i, (_, N) in enumerate(rings) if N // 2 >= f) for f in range(H + 1)]
    grid = [i * case["shift_step"] - case["shift_range"] for i in range(nx)]
    half_turn = 1.0 - 2.0 * (torch.arange(H + 1, device=dev) % 2)
    step = max(1, int(2e9 / (K * M * 8 * 4)))
    cc = torch.full((n,), -math.inf, dtype=torch.float64, device=dev)
    flat = torch.zeros((n,), dtype=torch.int64, device=dev)
    for b in range(0, n, step):
        s = slice(b, min(n, b + step))
        im = imgs[s].double()
        for si in range(S):
            X = _spectra(im, case, grid[si % nx], grid[si // nx], M)
            U = torch.empty((im.shape[0], K, H + 1), dtype=torch.complex128, device=dev)
            V = torch.empty_like(U)
            for f in range(H + 1):
                a, y = X[:, first[f]:, f], Y[:, first[f]:, f]
                p1, p2, p3, p4 = a.real @ y.real.T, a.imag @ y.imag.T, a.real @ y.imag.T, a.imag @ y.real.T
                U[:, :, f] = torch.complex(p1 + p2, p3 - p4)  # conj(X) Y
                V[:, :, f] = torch.complex(p1 - p2, p3 + p4)  # X Y
            for m, Z in enumerate((U, V * half_turn)[: 1 + case["mirror"]]):
                best, at = (torch.fft.irfft(Z, n=M) * M).flatten(1).max(dim=1)
                # among equal values the smallest (reference, shift, mirror, angle)
                index = ((at // M * S + si) * 2 + m) * M + at % M
                new = (best > cc[s]) | ((best == cc[s]) & (index < flat[s]))
                cc[s] = torch.where(new, best, cc[s])
                flat[s] = torch.where(new, index, flat[s])
    j, m, si, k = flat % M, flat // M % 2, flat // (2 * M) % S, flat // (2 * M * S)
    sx, sy = (si % nx) * case["shift_step"] - case["shift_range"], (si // nx) * case["shift_step"] - case["shift_range"]
    return (torch.stack([k, j, m, si], 1).int(),
            torch.stack([360.0 * j / M, sx.double(), sy.double(), cc], 1))


def _exact_average(case, imgs, pose, geometry, start):
    n, L, K = case["n"], case["L"], case["K"]
    c = torch.arange(L, dtype=torch.float64, device=imgs.device) - L / 2
    wy, wx = (v.reshape(1, -1) for v in torch.meshgrid(c, c, indexing="ij"))
    total = torch.zeros((K, L * L), dtype=torch.float64, device=imgs.device)
    for b in range(0, n, 1024):
        s = slice(b, min(n, b + 1024))
        th = pose[s, 1:2].double() * (2 * math.pi / _angles(case))
        sign = 1.0 - 2.0 * pose[s, 2:3]
        x = L / 2 + geometry[s, 1:2] + sign * (th.cos() * wx + th.sin() * wy)
        y = L / 2 + geometry[s, 2:3] + (th.cos() * wy - th.sin() * wx)
        total.index_add_(0, pose[s, 0].long(), _sample(imgs[s].double(), x, y))
    counts = torch.bincount(pose[:, 0].long(), minlength=K)
    avg = torch.where(counts[:, None] > 0, total / counts[:, None].clamp(min=1), start.reshape(K, -1).double())
    return avg.reshape(K, L, L), counts.int()


def exact(case, seed):
    refs, imgs, k = _inputs(case, seed)
    if case["op"] == "average":
        p = _given_poses(case, k, seed)
        avg, counts = _exact_average(case, imgs, p[:, :4], p.view(torch.float32)[:, 4:].double(), torch.zeros_like(refs))
        return {"avg": avg, "counts": counts}
    if work(case)["flops"] > 4e12 * (0.5 if case["last_ring"] > 40 else 1.0):
        return None  # too long in 64 bits
    pose, geometry = _exact_poses(case, refs.double(), imgs)
    if case["op"] == "align":
        return {"pose": pose, "geometry": geometry}
    classify = case["op"] == "classify"
    avg, counts = _exact_average(case, imgs, pose, geometry, refs if classify else torch.zeros_like(refs))
    if classify:
        d = avg - avg.mean(dim=(1, 2), keepdim=True)
        sd = d.square().mean(dim=(1, 2), keepdim=True).sqrt()
        fresh = torch.where(sd > 0, d / sd.clamp(min=1e-300), torch.zeros_like(d))
        avg = torch.where((counts > 0)[:, None, None], fresh, avg)
    if case["op"] == "host":
        return {"pose": pose.cpu(), "geometry": geometry.cpu(), "avg": avg.cpu(), "counts": counts.cpu()}
    return {"pose": pose, "geometry": geometry, "avg": avg, "counts": counts}
