"""The solver's measured workloads: what a program that uses this framework has it do.

Every case is one complete call sequence through the package's public entry points
(`Solver`, `Batch`, `autograd.UnrolledDDTV`): the data of an image (or of several) goes
in, some outer iterations of Algorithm 1 run, and the image, the energy, the gap or the
gradients come out.  `listed()` gives the fixed cases, `draw()` further ones of the same
ranges; `prepare()` makes what a program holds before the call (data on the GPU, the
solver handle), `run()` is one pass, `work()` its indispensable traffic and arithmetic,
and `exact()` the same outputs from a float64 evaluation of the method in plain torch.

Images are seeded piecewise-constant scenes of rectangles and disks with Gaussian noise
(denoising, segmentation) or salt-and-pepper noise (TV-L1), optionally with a random
inpainting domain, the recipe of the repository's workloads.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1901_00682_gb300 import _lib as L
from paper_1901_00682_gb300.autograd import UnrolledDDTV

ALPHA = {"l2": 10.0, "l1": 1.5, "seg": 20.0}
C1, C2 = 0.2, 0.8          # segmentation constants
# arithmetic of one pixel and inner iteration: divergence 3, u-step 5, two dual dofs 10 each
FLOPS_PX_ITER = 28


def listed():
    solve = dict(kind="solve", fidelity="l2", mask=False, inner=10, path="fused", tol=0.0)
    return [
        # the small denoising problem, 2 x 2 subdomains of 64 x 64: one short solve, where
        # launches and latency count
        dict(solve, name="rof_128", height=128, width=128, rows=2, cols=2, outer=200),
        # the throughput workload: a large image in subdomains of 128 x 128
        dict(solve, name="rof_4096", height=4096, width=4096, rows=32, cols=32, outer=60),
        # TV-L1 inpainting with impulse noise, every option of the fidelity in use
        dict(solve, name="tvl1_inpaint_2048", height=2048, width=2048, rows=16, cols=16, outer=100, fidelity="l1",
             mask=True),
        # a photograph whose sides do not divide into 128 x 128: subdomains of 120 x 128
        dict(solve, name="rof_1080x1920", height=1080, width=1920, rows=9, cols=15, outer=40),
        # a small photograph with odd sides, two-phase segmentation, subdomains of 107 x 120/121
        dict(solve, name="seg_321x481", height=321, width=481, rows=3, cols=4, outer=100, fidelity="seg"),
        # subdomains of 64 x 64, the other side the autotuner tries, L2 inpainting
        dict(solve, name="inpaint_tiles64_1024x768", height=1024, width=768, rows=16, cols=12, outer=50, mask=True),
        # 16 x 16 subdomains of 32 x 32 on a 512 x 512 image: the finest grid one splits it into
        dict(solve, name="tvl1_tiles32_512", height=512, width=512, rows=16, cols=16, outer=50, fidelity="l1"),
        # the adaptive inner stop of the paper, at most 20 inner iterations
        dict(solve, name="rof_adaptive_1024", height=1024, width=1024, rows=8, cols=8, outer=50, inner=20, tol=1e-4),
        # the undecomposed primal-dual iteration (N = 1), odd sides
        dict(solve, name="fulldim_1001x1503", height=1001, width=1503, rows=1, cols=1, outer=30, path="fulldim"),
        # training through the unrolled iterations: forward and backward, two images
        dict(kind="adjoint", name="unrolled_2x1024", images=2, height=1024, width=1024, rows=8, cols=8, outer=20,
             inner=10, every=5, fidelity="l2"),
        # the same for one odd image in uneven subdomains
        dict(kind="adjoint", name="unrolled_250x261", images=1, height=250, width=261, rows=2, cols=3, outer=30,
             inner=10, every=10, fidelity="l2"),
        # a batch of images of mixed shapes and fidelities, denoising and segmentation
        dict(kind="batch", name="batch_12", images=12, smallest=256, largest=1024, tile=128, inner=10, outer=20,
             shapes=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


MAX_WORK = 4096 * 4096 * 60 * 10   # pixels x inner iterations of the largest listed case


def draw(rng):
    """A further case: solves of every fidelity, subdomain size and path, unrolled
    differentiation and mixed batches, with sides from about a hundred pixels to four
    thousand (log-uniform, mostly not multiples of the subdomain side)."""
    kind = rng.choice(["solve"] * 6 + ["adaptive", "fulldim", "adjoint", "batch"])
    if kind == "batch":
        case = dict(kind="batch", images=rng.randint(2, 16), smallest=256, largest=rng.choice([512, 1024]),
                    tile=rng.choice([64, 128, 128]), inner=rng.choice([5, 10, 20]), shapes=rng.randint(1, 10 ** 6))
        px = sum(h * w for h, w, _ in _shapes(case))
        return dict(case, outer=_outer(rng, 8, 40, 4 * px * case["inner"]))
    fidelity = rng.choice(["l2", "l1", "seg"])
    if kind == "adjoint":
        h, w = _log_int(rng, 96, 1024), _log_int(rng, 96, 1024)
        rows, cols = _grid(rng, h, w)
        images, inner = rng.randint(1, 3), rng.choice([5, 10])
        return dict(kind="adjoint", images=images, height=h, width=w, rows=rows, cols=cols,
                    outer=_outer(rng, 10, 30, 16 * images * h * w * inner), inner=inner, every=rng.choice([5, 10]),
                    fidelity=rng.choice(["l2", "seg"]))
    inner = rng.choice([5, 10, 10, 20])
    if kind == "fulldim":
        h, w, rows, cols = _log_int(rng, 96, 2048), _log_int(rng, 96, 2048), 1, 1
    elif rng.random() < 0.35:   # sides that divide into equal subdomains
        t = rng.choice([32, 64, 128, 128])
        rows, cols = _log_int(rng, 2, 4096 // t), _log_int(rng, 2, 4096 // t)
        h, w = t * rows, t * cols
    else:
        h, w = _log_int(rng, 96, 4096), _log_int(rng, 96, 4096)
        rows, cols = _grid(rng, h, w)
    # a pass of the undecomposed path, and of the fused one on small or uneven subdomains,
    # takes several times that of the largest listed case's kernel
    return dict(kind="solve", height=h, width=w, rows=rows, cols=cols, fidelity=fidelity,
                mask=fidelity != "seg" and rng.random() < 0.4, inner=inner,
                outer=_outer(rng, 20, 200, (10 if kind == "fulldim" else 5) * h * w * inner),
                path="fulldim" if kind == "fulldim" else "fused",
                tol=rng.choice([1e-3, 1e-4]) if kind == "adaptive" else 0.0)


def _outer(rng, lo, hi, work):
    """Outer iterations of a drawn case, of `work` weighted pixel iterations each."""
    return max(2, min(rng.randint(lo, hi), MAX_WORK // work))


def _grid(rng, h, w):
    side = _log_int(rng, 24, 128)   # largest subdomain side
    return -(-h // side), -(-w // side)


# ---- inputs

def _scene(h, w, rng):
    img = np.full((h, w), rng.random(), dtype=np.float32)
    m = min(h, w)
    for _ in range(max(4, 400 * h * w // (4096 * 4096))):
        val = np.float32(rng.random())
        if rng.random() < 0.5:
            rh, rw = int(rng.uniform(h / 16, h / 4)), int(rng.uniform(w / 16, w / 4))
            r0, c0 = int(rng.integers(0, h)), int(rng.integers(0, w))
            img[r0:r0 + max(rh, 1), c0:c0 + max(rw, 1)] = val
        else:
            rad, cy, cx = rng.uniform(m / 32, m / 8), rng.uniform(0, h), rng.uniform(0, w)
            y0, y1 = max(int(cy - rad) - 1, 0), min(int(cy + rad) + 2, h)
            x0, x1 = max(int(cx - rad) - 1, 0), min(int(cx + rad) + 2, w)
            yy = np.arange(y0, y1, dtype=np.float32)[:, None] + np.float32(0.5 - cy)
            xx = np.arange(x0, x1, dtype=np.float32)[None, :] + np.float32(0.5 - cx)
            img[y0:y1, x0:x1][yy * yy + xx * xx <= rad * rad] = val
    return img


def _image(h, w, fidelity, masked, rng):
    """(noisy image, mask or None, clean image)."""
    clean = _scene(h, w, rng)
    if fidelity == "l1":
        f = clean.copy()
        hit = rng.random((h, w), dtype=np.float32)
        f[hit < 0.05] = 0.0
        f[hit > 0.95] = 1.0
    else:
        sigma = 0.1 if h * w >= 2048 * 2048 else 0.05
        f = clean + np.float32(sigma) * rng.standard_normal((h, w), dtype=np.float32)
    mask = None
    if masked:
        mask = (rng.random((h, w), dtype=np.float32) < 0.2).astype(np.uint8)
        f[mask == 1] = 0.0
    return f, mask, clean


def _shapes(case):
    """Sides and fidelity of a batch's images: short side smallest, 2 smallest, ... or
    largest, aspect 1:1, 1:2 or 2:1, denoising and segmentation in turn."""
    rng = np.random.default_rng(case["shapes"])
    sides = [case["smallest"] * 2 ** k for k in range(int(math.log2(case["largest"] // case["smallest"])) + 1)]
    out = []
    for i in range(case["images"]):
        s, aspect = int(rng.choice(sides)), int(rng.integers(0, 3))
        h, w = ((s, s), (s, 2 * s), (2 * s, s))[aspect]
        out.append((h, w, "l2" if i % 2 == 0 else "seg"))
    return out


def _inputs(case, seed):
    """The host arrays of a case: a list of (f, mask, clean)."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "batch":
        return [_image(h, w, fid, False, rng) for h, w, fid in _shapes(case)]
    if case["kind"] == "adjoint":
        return [_image(case["height"], case["width"], case["fidelity"], False, rng) for _ in range(case["images"])]
    return [_image(case["height"], case["width"], case["fidelity"], case["mask"], rng)]


def _region_constants(fidelity):
    return dict(c1=C1, c2=C2) if fidelity == "seg" else {}


def prepare(case, seed):
    data = _inputs(case, seed)
    if case["kind"] == "batch":
        images = [dict(height=h, width=w, fidelity=fid, alpha=ALPHA[fid], **_region_constants(fid))
                  for h, w, fid in _shapes(case)]
        fs = [torch.from_numpy(f).cuda() for f, _, _ in data]
        return dict(case=case, batch=L.Batch(images, inner_iters=case["inner"], tile=case["tile"]), fs=fs,
                    us=[torch.empty_like(f) for f in fs])
    if case["kind"] == "adjoint":
        fid = case["fidelity"]
        f = torch.from_numpy(np.stack([d[0] for d in data])).cuda().requires_grad_(True)
        target = torch.from_numpy(np.stack([d[2] for d in data])).cuda()
        alpha = torch.tensor(ALPHA[fid], dtype=torch.float64, device="cuda", requires_grad=True)
        model = UnrolledDDTV(case["height"], case["width"], case["rows"], case["cols"], case["outer"],
                             checkpoint_every=case["every"], fidelity=fid, inner_iters=case["inner"],
                             **_region_constants(fid))
        return dict(case=case, model=model, f=f, alpha=alpha, target=target)
    f, mask, _ = data[0]
    p = L.make_params(case["height"], case["width"], case["rows"], case["cols"], fidelity=case["fidelity"],
                      alpha=ALPHA[case["fidelity"]], inner_iters=case["inner"], outer_iters=case["outer"],
                      path=case["path"], inner_tol=case["tol"], **_region_constants(case["fidelity"]))
    fd = torch.from_numpy(f).cuda()
    return dict(case=case, solver=L.Solver(p), f=fd, u=torch.empty_like(fd),
                mask=None if mask is None else torch.from_numpy(mask).cuda())


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        # a batch solved together, then every image read out with its energy
        b = state["batch"]
        b.load(state["fs"])
        b.iterate(case["outer"])
        return dict(u=[b.get_u(i, u) for i, u in enumerate(state["us"])],
                    energy=[b.energy(i) for i in range(len(state["us"]))])
    if case["kind"] == "adjoint":
        # one training step's forward and backward: loss 1/2 ||u_N - g||^2
        f, alpha = state["f"], state["alpha"]
        f.grad = alpha.grad = None
        u = state["model"](f, alpha)
        (0.5 * ((u - state["target"]) ** 2).sum()).backward()
        return dict(u=u.detach(), grad_f=f.grad, grad_alpha=alpha.grad)
    # a solve: load, iterate, read the image and the certificate of where it stands
    s = state["solver"]
    s.load(state["f"], state["mask"])
    s.iterate(case["outer"])
    u = s.get_u(state["u"])
    if case["path"] == "fulldim" or case["fidelity"] == "l1" or case["mask"]:
        return dict(u=u, energy=s.current_energy())   # no finite dual value is defined there
    primal, dual = s.gap()
    return dict(u=u, energy=primal, dual=dual)


def work(case):
    if case["kind"] == "batch":
        px = sum(h * w for h, w, _ in _shapes(case))
        return dict(bytes=8 * px, flops=FLOPS_PX_ITER * px * case["inner"] * case["outer"])
    px = case["height"] * case["width"]
    if case["kind"] == "adjoint":
        px *= case["images"]
        # f and the target in, u and df out; the reverse of an iteration costs about two
        return dict(bytes=16 * px, flops=3 * FLOPS_PX_ITER * px * case["inner"] * case["outer"])
    # the adaptive stop runs about four inner iterations where its cap allows 20
    inner = 4 if case["tol"] > 0 else case["inner"]
    return dict(bytes=(9 if case["mask"] else 8) * px, flops=FLOPS_PX_ITER * px * inner * case["outer"])


# ---- the method in float64 (plain torch, torn layout)

def _partition(n, parts):
    return [a * n // parts for a in range(parts + 1)]


class _Torn:
    """Index tables of one axis (n pixels in `parts` subdomains): torn edge positions
    run over n + parts values, every subdomain holding both its end edges."""

    def __init__(self, n, parts, dev):
        start = _partition(n, parts)
        before, after, first, lim, s_edge = [], [], [], [], []
        for a in range(parts):
            for k in range(start[a], start[a + 1] + 1):
                before.append(k - 1 if k > start[a] else n)   # n: the zero pad
                after.append(k if k < start[a + 1] else n)
                lim.append(0.0 if k in (0, n) and (a == 0 and k == 0 or a == parts - 1 and k == n) else 1.0)
            first += [k + a for k in range(start[a], start[a + 1])]
            s_edge.append(start[a + 1] + a)
        t = lambda v, d=torch.int64: torch.tensor(v, dtype=d, device=dev)
        self.before, self.after, self.first = t(before), t(after), t(first)
        self.lim = t(lim, torch.float64)
        self.s = t(s_edge[:-1])       # last edge of every subdomain that has one after it
        self.size = n + parts


class _Method:
    def __init__(self, h, w, rows, cols, fidelity, alpha, inner, dev, fulldim=False):
        self.fid, self.alpha, self.inner, self.full = fidelity, alpha, inner, fulldim
        self.r, self.c = _Torn(h, rows, dev), _Torn(w, cols, dev)
        self.tau = 1.0 if fidelity == "seg" else 50.0
        self.sigma, self.gamma = 0.5 / self.tau, 1.0 / (8.0 * self.tau)
        self.dev, self.h, self.w = dev, h, w

    def start(self, f, mask):
        z = lambda *s: torch.zeros(*s, dtype=torch.float64, device=self.dev)
        u = torch.full_like(f, 0.5) if self.fid == "seg" else (f if mask is None else torch.where(mask, 0.0 * f, f))
        p1, p2 = z(self.r.size, self.w), z(self.h, self.c.size)
        lam1, lam2 = z(len(self.r.s), self.w), z(self.h, len(self.c.s))
        return u, p1, p2, lam1, lam2, p1, p2

    def div(self, p1, p2):
        r, c = self.r.first, self.c.first
        return p1[r + 1] - p1[r] + p2[:, c + 1] - p2[:, c]

    def grad(self, u):
        a = torch.cat([u, torch.zeros_like(u[:1])])
        b = torch.cat([u, torch.zeros_like(u[:, :1])], 1)
        return a[self.r.after] - a[self.r.before], b[:, self.c.after] - b[:, self.c.before]

    def prox(self, ub, f, mask, s):
        if self.fid == "seg":
            return (ub - s * ((f - C1) ** 2 - (f - C2) ** 2)).clamp(0.0, 1.0)
        if self.fid == "l2":
            v = (ub + s * f) / (1.0 + s)
        else:
            v = ub - torch.minimum(torch.maximum(ub - f, -s + 0.0 * f), s + 0.0 * f)
        return v if mask is None else torch.where(mask, ub, v)

    def outer(self, f, mask, alpha, u, p1, p2, lam1, lam2, o1, o2):
        l1, l2 = self.r.lim[:, None], self.c.lim[None, :]
        proj = lambda t, lim: torch.minimum(torch.maximum(t, -lim), lim)
        tk, sk = 10.0, 1.0 / 80.0
        if self.full:
            # o1, o2 carry the extrapolated field
            for _ in range(self.inner):
                u = self.prox(u + sk * self.div(o1, o2), f, mask, sk * alpha)
                g1, g2 = self.grad(u)
                n1, n2 = proj(p1 + tk * g1, l1), proj(p2 + tk * g2, l2)
                o1, o2, p1, p2 = 2.0 * n1 - p1, 2.0 * n2 - p2, n1, n2
            return u, p1, p2, lam1, lam2, o1, o2
        rs, cs = self.r.s, self.c.s
        x1, x2 = 2.0 * p1 - o1, 2.0 * p2 - o2
        lam1 = lam1 + self.sigma * (x1[rs] - x1[rs + 1])
        lam2 = lam2 + self.sigma * (x2[:, cs] - x2[:, cs + 1])
        h1 = p1.index_add(0, rs, -self.tau * lam1).index_add(0, rs + 1, self.tau * lam1)
        h2 = p2.index_add(1, cs, -self.tau * lam2).index_add(1, cs + 1, self.tau * lam2)
        o1, o2, q1, q2 = p1, p2, p1, p2
        for _ in range(self.inner):
            u = self.prox(u + sk * self.div(q1, q2), f, mask, sk * alpha)
            g1, g2 = self.grad(u)
            n1 = proj((self.tau * (p1 + tk * g1) + tk * h1) / (self.tau + tk), l1)
            n2 = proj((self.tau * (p2 + tk * g2) + tk * h2) / (self.tau + tk), l2)
            th = 1.0 / math.sqrt(1.0 + 2.0 * self.gamma * tk)
            q1, q2, p1, p2 = n1 + th * (n1 - p1), n2 + th * (n2 - p2), n1, n2
            tk, sk = th * tk, sk / th
        return u, p1, p2, lam1, lam2, o1, o2

    def iterate(self, f, mask, n, checkpoint=False):
        st = self.start(f, mask)
        for _ in range(n):
            if checkpoint:
                st = torch.utils.checkpoint.checkpoint(self.outer, f, mask, self.alpha, *st, use_reentrant=False)
            else:
                st = self.outer(f, mask, self.alpha, *st)
        return st

    def energy(self, u, f, mask):
        if self.fid == "seg":
            fit = (u * ((f - C1) ** 2 - (f - C2) ** 2)).sum()
        else:
            e = 0.5 * (u - f) ** 2 if self.fid == "l2" else (u - f).abs()
            fit = (e if mask is None else torch.where(mask, 0.0 * e, e)).sum()
        return float(self.alpha * fit + (u[1:] - u[:-1]).abs().sum() + (u[:, 1:] - u[:, :-1]).abs().sum())

    def dual(self, f, p1, p2):
        # the two copies of an interface edge averaged
        p1, p2, rs, cs = p1.clone(), p2.clone(), self.r.s, self.c.s
        p1[rs] = p1[rs + 1] = 0.5 * (p1[rs] + p1[rs + 1])
        p2[:, cs] = p2[:, cs + 1] = 0.5 * (p2[:, cs] + p2[:, cs + 1])
        d = self.div(p1, p2)
        if self.fid == "seg":
            return float((self.alpha * ((f - C1) ** 2 - (f - C2) ** 2) - d).clamp(max=0.0).sum())
        return float((-(d + self.alpha * f) ** 2 / (2.0 * self.alpha) + 0.5 * self.alpha * f * f).sum())


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    host = lambda t: t.detach().cpu()
    data = [(torch.from_numpy(f).to(dev).double(), None if m is None else torch.from_numpy(m).to(dev).bool(),
             torch.from_numpy(g).to(dev).double()) for f, m, g in _inputs(case, seed)]
    if case["kind"] == "batch":
        us, js = [], []
        for (f, _, _), (h, w, fid) in zip(data, _shapes(case)):
            m = _Method(h, w, h // case["tile"], w // case["tile"], fid, ALPHA[fid], case["inner"], dev)
            u = m.iterate(f, None, case["outer"])[0]
            us.append(host(u))
            js.append(m.energy(u, f, None))
        return dict(u=us, energy=js)
    fid = case["fidelity"]
    if case["kind"] == "adjoint":
        us, gfs, ga = [], [], 0.0
        for f, _, g in data:
            f = f.requires_grad_(True)
            alpha = torch.tensor(ALPHA[fid], dtype=torch.float64, device=dev, requires_grad=True)
            m = _Method(case["height"], case["width"], case["rows"], case["cols"], fid, alpha, case["inner"], dev)
            u = m.iterate(f, None, case["outer"], checkpoint=True)[0]
            (0.5 * ((u - g) ** 2).sum()).backward()
            us.append(host(u))
            gfs.append(host(f.grad))
            ga = ga + host(alpha.grad)
        return dict(u=torch.stack(us), grad_f=torch.stack(gfs), grad_alpha=ga)
    if case["tol"] > 0:
        return None   # the stop is decided on float32 sums: a near tie gives another count in 64 bits
    f, mask, _ = data[0]
    m = _Method(case["height"], case["width"], case["rows"], case["cols"], fid, ALPHA[fid], case["inner"], dev,
                fulldim=case["path"] == "fulldim")
    u, p1, p2 = m.iterate(f, mask, case["outer"])[:3]
    out = dict(u=host(u), energy=m.energy(u, f, mask))
    if not (case["path"] == "fulldim" or fid == "l1" or case["mask"]):
        out["dual"] = m.dual(f, p1, p2)
    return out
