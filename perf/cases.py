"""Performance cases of the segmentation library: the work its users have it do, through its public calls.

A case is a dict of plain values.  Its "kind" says which call it stands for:

  step     a context with an image set, as an interactive or resumed program holds it: the phase field is set, the
           time steps are taken and the new field and the energy are read back (ac.Segmenter, device buffers);
  segment  the whole call of a program that labels pictures: image from host memory, start field, time steps, pixel
           labels and the composite back in host memory;
  batch    one time step of many uneven images (ac.Batch);
  train    one gradient evaluation of a loss on the final field (adjoint.SegmentationSteps and its backward).

Images are piecewise-smooth Voronoi regions with colour ramps and noise.  A "random" start is a Dirichlet draw at
every node (the first steps of a segmentation, every node undecided); a "formed" start has phases separated by
interfaces a few pixels wide (the later steps, and a resumed run).

Tolerances: one digit below the library's default (1e-10), so that the results of two solvers agree to nine digits
(the error of a step is up to a few tens of its residual).  Sizes that are not multiples of 16 are solved to 1e-12, as
the parity tests solve ragged sizes: a solve with few grid levels stops on a smooth error that is larger still.
"""
import math
import random

import numpy as np
import torch

from paper_0710_0736_gb300 import ac, adjoint


def listed():
    step = dict(kind="step", precision="mixed", eps=2.0, lam=1.0, steps=1, start="random", refine=0, projection="simplex",
                stream="own", tol=1e-11)
    return [
        # the smallest call: the plain 64 x 64 workload in binary64 (latency and launches)
        dict(step, name="step_fp64_64_n4", W=64, H=64, N=4, precision="fp64"),
        # a small picture of the batch workload on its own
        dict(step, name="step_mixed_128_n6", W=128, H=128, N=6),
        # an ordinary picture, as the README's example calls it (torch's default stream, two steps)
        dict(step, name="step_mixed_512_n4_default_stream", W=512, H=512, N=4, steps=2, stream="default"),
        # the two-phase wide picture of the batch workload, solved on the grid refined once, projection by node
        dict(step, name="step_mixed_768x512_n2_refined", W=768, H=512, N=2, refine=1, projection="node"),
        # a picture whose sides are odd
        dict(step, name="step_mixed_1001x751_n5", W=1001, H=751, N=5, tol=1e-12),
        # the 1024 x 1024 workload in its two precisions
        dict(step, name="step_fp64_1024_n4", W=1024, H=1024, N=4, precision="fp64", start="formed"),
        dict(step, name="step_mixed_1024_n4", W=1024, H=1024, N=4),
        # the large picture, in its first steps and once the phases have formed
        dict(step, name="step_mixed_4096_n8_first", W=4096, H=4096, N=8, eps=3.0, lam=2.0),
        dict(step, name="step_mixed_4096_n8_formed", W=4096, H=4096, N=8, eps=3.0, lam=2.0, start="formed"),
        # a full-HD frame from host memory to labels and composite
        dict(kind="segment", name="segment_1920x1080_n4", W=1920, H=1080, N=4, precision="mixed", eps=2.0, lam=1.0,
             steps=3, start="random", refine=0, projection="simplex", stream="own", tol=1e-12),
        # the batch workload's mix of sizes and phase counts
        dict(kind="batch", name="batch_24_uneven", count=24, specs=5, precision="mixed", eps=2.0, lam=1.0, steps=1,
             start="random", streams=16, tol=1e-11),
        # gradients through a few steps (the 512 x 512 workload), as a torch program calls them
        dict(kind="train", name="train_512_n4", W=512, H=512, N=4, precision="fp64", eps=2.0, lam=1.0, steps=4, every=2,
             start="random", refine=0, projection="simplex", stream="default", tol=1e-12),
    ]


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["segment", "batch", "train"])
    eps, lam = rng.choice([1.5, 2.0, 2.5, 3.0]), rng.choice([0.5, 1.0, 2.0])
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(3, 24), specs=rng.randint(0, 10 ** 6), precision="mixed",
                    eps=rng.choice([1.5, 2.0]), lam=lam, steps=1, start=rng.choice(["random", "formed"]),
                    streams=rng.choice([4, 8, 16]), tol=1e-11)
    even = rng.random() < 0.5
    precision = "fp64" if kind == "train" or (kind == "step" and rng.random() < 0.3) else "mixed"
    if kind == "train":
        eps = 2.0
    N = rng.randint(2, 8)
    refine = 1 if kind == "step" and rng.random() < 0.2 else 0
    # unknowns of the solve grid: the odd sizes have few grid levels, and binary64 runs at a fraction of the float
    # rate, so that the same time buys fewer of them
    top = {("mixed", True): 2 ** 25, ("mixed", False): 2 ** 22, ("fp64", True): 2 ** 21,
           ("fp64", False): 2 ** 18}[(precision, even)]
    if kind == "train":
        top = min(top, 2 ** 20)
    if kind == "segment":
        top = min(top, 2 ** 23)
    px = math.exp(rng.uniform(math.log(48.0 ** 2), math.log(top / N))) / 4 ** refine
    side = math.sqrt(px)
    aspect = math.exp(rng.uniform(-0.6, 0.6))
    W, H = max(16, int(side * aspect)), max(16, int(side / aspect))
    if even:
        W, H = max(16, W // 16 * 16), max(16, H // 16 * 16)
    case = dict(kind=kind, W=W, H=H, N=N, precision=precision, eps=eps, lam=lam, steps=1,
                start=rng.choice(["random", "formed"]), refine=refine,
                projection=rng.choice(["simplex"] * 4 + ["node"]) if kind == "step" else "simplex",
                stream=rng.choice(["own", "default"]), tol=1e-11 if even else 1e-12)
    if kind == "segment":
        case.update(steps=rng.randint(1, 2), tol=1e-12)
    if kind == "train":
        case.update(steps=rng.randint(1, 3), every=1, stream="default", tol=1e-12)
    return case


# ---- inputs ---------------------------------------------------------------------------------------------------------

BATCH_SIZES = [(128, 128), (256, 256), (512, 512), (1024, 1024), (768, 512)]


def batch_images(case):
    """(W, H, N, noise) of a batch's images: the mix of the batch workload."""
    rng = random.Random(case["specs"])
    return [rng.choice(BATCH_SIZES) + (rng.choice([2, 4, 6]), rng.uniform(0.02, 0.15)) for _ in range(case["count"])]


def simplex_rows(y):
    """Projection of every column of y (phases first) onto the simplex: Newton's iteration for the threshold."""
    theta = (y.sum(0) - 1) / y.shape[0]
    for _ in range(y.shape[0] - 1):
        kept = y > theta
        theta = (torch.where(kept, y, 0.0).sum(0) - 1) / kept.sum(0)
    return (y - theta).clamp_(min=0)


class Inputs:
    """Image (H x W x 3 float32) and start field (nodes x N float64) of one picture, on the GPU."""

    def __init__(self, W, H, N, seed, noise, eps, start, refine=0):
        g = torch.Generator(device="cuda").manual_seed(seed)

        def rand(*shape):
            return torch.rand(shape, generator=g, device="cuda")

        regions = max(N, 8)
        phase = [k % N for k in range(regions)]
        px, py = (rand(regions) * W).tolist(), (rand(regions) * H).tolist()
        base, ramp, angle = rand(N, 3), 0.2 * rand(N, 3), 2 * math.pi * rand(N)
        xs, ys = torch.arange(W, device="cuda") + 0.5, torch.arange(H, device="cuda") + 0.5
        label, best = None, None
        for k in range(regions):
            d = (ys[:, None] - py[k]) ** 2 + (xs[None, :] - px[k]) ** 2
            if k == 0:
                best, label = d, torch.zeros((H, W), dtype=torch.long, device="cuda")
            else:
                label = torch.where(d < best, phase[k], label)
                best = torch.minimum(best, d)
        along = torch.cos(angle)[label] * (xs / W)[None, :] + torch.sin(angle)[label] * (ys / H)[:, None]
        img = base[label] + ramp[label] * along[..., None]
        self.image = (img + noise * torch.randn((H, W, 3), generator=g, device="cuda")).clamp_(0, 1).contiguous()
        Wr, Hr = W << refine, H << refine
        if start == "random":
            u = -torch.log(torch.rand(((Wr + 1) * (Hr + 1), N), generator=g, device="cuda", dtype=torch.float64) + 1e-9)
            u /= u.sum(1, keepdim=True)
        else:
            xn = torch.arange(Wr + 1, device="cuda", dtype=torch.float64) / 2 ** refine
            yn = torch.arange(Hr + 1, device="cuda", dtype=torch.float64) / 2 ** refine
            d = torch.full((N, Hr + 1, Wr + 1), math.inf, device="cuda", dtype=torch.float64)
            for k in range(regions):
                dk = ((yn[:, None] - py[k]) ** 2 + (xn[None, :] - px[k]) ** 2).sqrt_()
                d[phase[k]] = torch.minimum(d[phase[k]], dk)
            u = simplex_rows(-d / (4 * eps)).reshape(N, -1).t()
        self.u0 = u.contiguous()


def segmenter(case, stream):
    kw = {"stream": stream.cuda_stream} if stream is not None else {}
    return ac.Segmenter(case["W"], case["H"], case["N"], case["eps"], case["lam"], case["eps"] ** 2, tol=case["tol"],
                        max_cycles=2000, refine=case["refine"],
                        precision=ac.AC_MIXED if case["precision"] == "mixed" else ac.AC_FP64,
                        projection=ac.AC_PROJ_NODE if case["projection"] == "node" else ac.AC_PROJ_SIMPLEX, **kw)


def one_picture(case, seed):
    return Inputs(case["W"], case["H"], case["N"], seed, 0.05, case["eps"], case["start"], case["refine"])


def batch_pictures(case, seed):
    return [Inputs(W, H, N, seed * 1009 + k, noise, case["eps"], case["start"])
            for k, (W, H, N, noise) in enumerate(batch_images(case))]


def target_labels(case, seed):
    """A piecewise-constant target on the nodes: a Voronoi map of six seeds."""
    rng = random.Random(seed)
    W, H, N = case["W"], case["H"], case["N"]
    xs, ys = torch.arange(W + 1, device="cuda"), torch.arange(H + 1, device="cuda")
    d = torch.stack([(ys[:, None] - rng.uniform(0, H)) ** 2 + (xs[None, :] - rng.uniform(0, W)) ** 2 for _ in range(6)])
    return torch.tensor([rng.randrange(N) for _ in range(6)], device="cuda")[d.argmin(0)].reshape(-1)


def node_mass(W, H):
    """Lumped mass of the nodes, (H + 1) x (W + 1)."""
    m = torch.zeros((H + 1, W + 1), device="cuda", dtype=torch.float64)
    for sy, sx, w in ((0, 0, 2), (1, 1, 2), (0, 1, 1), (1, 0, 1)):
        m[sy:sy + H, sx:sx + W] += w / 6
    return m


def prepare(case, seed):
    stream = torch.cuda.Stream() if case.get("stream") == "own" else None
    state = {"case": case, "stream": stream}
    if case["kind"] == "batch":
        pics = batch_pictures(case, seed)
        b = ac.Batch([dict(W=W, H=H, N=N, eps=case["eps"], tau=case["eps"] ** 2, lam=case["lam"], tol=case["tol"],
                           max_cycles=2000, precision=ac.AC_MIXED) for W, H, N, _ in batch_images(case)],
                     n_streams=case["streams"])
        torch.cuda.synchronize()  # the images are made on torch's stream, the batch reads them on its own
        for k, p in enumerate(pics):
            b.set_image(k, p.image)
        torch.cuda.synchronize()
        state.update(batch=b, u0=[p.u0 for p in pics])
        return state
    pic = one_picture(case, seed)
    torch.cuda.synchronize()
    if case["kind"] == "train":
        state.update(image=pic.image.double().requires_grad_(), u0=pic.u0.requires_grad_(),
                     lam=torch.tensor(case["lam"], dtype=torch.float64, device="cuda", requires_grad=True),
                     eps=torch.tensor(case["eps"], dtype=torch.float64, device="cuda", requires_grad=True),
                     mass=node_mass(case["W"], case["H"]).reshape(-1), target=target_labels(case, seed))
        return state
    seg = segmenter(case, stream)
    state.update(seg=seg, u0=pic.u0)
    if case["kind"] == "segment":
        host = torch.empty(pic.image.shape, dtype=torch.float32, pin_memory=True)
        host.copy_(pic.image)
        state.update(host=host, image=host.numpy(),  # the array shares the pinned buffer
                     labels=np.zeros((case["H"], case["W"]), np.int8))
    else:
        seg.set_image(pic.image)
    torch.cuda.synchronize()
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b, out = state["batch"], []
        for k, u0 in enumerate(state["u0"]):
            b.set_phase(k, u0)
        b.step(case["steps"])
        for k, u0 in enumerate(state["u0"]):
            u = torch.empty_like(u0)
            ac.lib.ac_batch_get_phase(b.b, k, u.data_ptr(), 1)
            out.append(u)
        return out
    if case["kind"] == "train":
        u = adjoint.SegmentationSteps.apply(state["image"], state["lam"], state["eps"], state["u0"], case["eps"] ** 2,
                                            case["steps"], case["every"], case["tol"], ac.AC_FP64)
        loss = adjoint.misfit_loss(u, state["mass"], state["target"])
        grads = torch.autograd.grad(loss, [state["image"], state["lam"], state["eps"], state["u0"]])
        return {"u": u.detach(), "loss": loss.detach(), "image": grads[0], "lam": grads[1], "eps": grads[2], "u0": grads[3]}
    seg, u0 = state["seg"], state["u0"]
    stream = state["stream"] or torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        if case["kind"] == "segment":
            seg.set_image(state["image"])
            seg.set_phase(u0)
            ac.ac_segment(seg.ctx, case["steps"], state["labels"], seg.W, seg.H)
            composite = seg.composite()
            u = torch.empty_like(u0)
            ac.ac_get_phase(seg.ctx, u, seg.n_nodes, seg.N)
            return {"u": u, "labels": state["labels"], "composite": composite}
        seg.set_phase(u0)
        st = seg.step(case["steps"])
        u = torch.empty_like(u0)
        ac.ac_get_phase(seg.ctx, u, seg.n_nodes, seg.N)
        return {"u": u, "energy": st.energy}


def work(case):
    """The field read and written once per time step, the image read once; one colour-mean sum, one right-hand side and
    one projected sweep per step, the least a step can do (about 30 operations per unknown)."""
    if case["kind"] == "batch":
        dof = sum((W + 1) * (H + 1) * N for W, H, N, _ in batch_images(case))
        px = sum(W * H for W, H, _, _ in batch_images(case))
    else:
        r = case["refine"]
        dof = ((case["W"] << r) + 1) * ((case["H"] << r) + 1) * case["N"]
        px = case["W"] * case["H"]
    steps = case["steps"] * (2 if case["kind"] == "train" else 1)  # a gradient solves an adjoint step for each step
    out = {"step": 0, "batch": 0, "segment": 13 * px, "train": 24 * px + 8 * dof}[case["kind"]]
    return {"bytes": 16.0 * dof * steps + 12 * px + out, "flops": 30.0 * dof * steps}


# ---- the same in 64 bits, plain torch -------------------------------------------------------------------------------

class Grid:
    """The step problem of one picture: planes are (..., H + 1, W + 1), phases first."""

    def __init__(self, image, N, eps, lam, tau, refine, projection):
        image = image.repeat_interleave(2 ** refine, 0).repeat_interleave(2 ** refine, 1).permute(2, 0, 1)
        self.H, self.W = image.shape[1:]
        self.N, s = N, 2.0 ** refine
        self.eps, self.tau, self.lam, self.scale = eps * s, tau * s, lam / s, 1 / s
        self.m0 = node_mass(self.W, self.H)
        self.by_node = projection == "node"
        self.m1, self.m2 = self.moments(image)
        ones_x, ones_y = torch.ones(self.H + 1, 1, device="cuda"), torch.ones(1, self.W + 1, device="cuda")
        self.we, self.wn = ones_x.double(), ones_y.double()  # edges to the east by row, to the north by column
        self.we[0] = self.we[-1] = 0.5
        self.wn[:, 0] = self.wn[:, -1] = 0.5

    def moments(self, image):
        """<eta_n, I> (3 planes) and <eta_n, |I|^2>: by simplex of the pixelwise constant image, by node of the nodal
        values with the consistent mass matrix."""
        vals = torch.cat([image, (image * image).sum(0, keepdim=True)])
        H, W = self.H, self.W
        if not self.by_node:
            shifts = ((0, 0, 2 / 6), (1, 1, 2 / 6), (0, 1, 1 / 6), (1, 0, 1 / 6))
            m = sum(w * torch.nn.functional.pad(vals, (sx, 1 - sx, sy, 1 - sy)) for sy, sx, w in shifts)
        else:
            v = torch.cat([vals, vals[:, -1:]], 1)
            v = torch.cat([v, v[:, :, -1:]], 2)
            m = 0
            for tri in (((0, 0), (0, 1), (1, 1)), ((0, 0), (1, 0), (1, 1))):  # the two triangles of a pixel (y, x)
                c = [v[:, a:a + H, b:b + W] for a, b in tri]
                for (a, b), own in zip(tri, c):
                    m = m + torch.nn.functional.pad((own + c[0] + c[1] + c[2]) / 24, (b, 1 - b, a, 1 - a))
        return m[:3], m[3]

    def stiff(self, u):
        """A u (the graph Laplacian of the axis edges)."""
        dx, dy = self.we * (u[..., 1:] - u[..., :-1]), self.wn * (u[..., 1:, :] - u[..., :-1, :])
        out = torch.zeros_like(u)
        out[..., :-1] -= dx
        out[..., 1:] += dx
        out[..., :-1, :] -= dy
        out[..., 1:, :] += dy
        return out

    def means(self, u):
        mass = torch.stack([(p * self.m0).sum() for p in u])
        s = torch.stack([torch.stack([(p * m).sum() for m in self.m1]) for p in u])
        return s / mass[:, None], s, mass

    def energy(self, u):
        c, s, mass = self.means(u)
        fit = sum((p * self.m2).sum() for p in u) - (s * s / mass[:, None]).sum()
        return self.scale * (self.lam * fit + (self.m0 * u * (1 - u)).sum() / self.eps +
                             0.5 * self.eps * sum((p * self.stiff(p)).sum() for p in u))

    def rhs(self, u, eps, lam):
        c = self.means(u)[0]
        f = torch.stack([self.m2 - 2 * (ci[0] * self.m1[0] + ci[1] * self.m1[1] + ci[2] * self.m1[2]) +
                         (ci * ci).sum() * self.m0 for ci in c])
        return self.m0 * u * (1 + 2 * self.tau / eps) - self.tau * lam * f

    def diagonal(self):
        d = torch.zeros_like(self.m0)
        d[:, :-1] += self.we
        d[:, 1:] += self.we
        d[:-1] += self.wn
        d[1:] += self.wn
        return self.m0 + self.tau * self.eps * d

    def minimise(self, b, u):
        """argmin 1/2 u'Su - b'u over the simplices: accelerated projected gradients in the metric of S's diagonal, in
        which S lies between Mhat / diagonal and 2."""
        te, D = self.tau * self.eps, self.diagonal()
        q = math.sqrt(1 / (2 * (1 + 4 * te)))
        beta, old = (1 - q) / (1 + q), u
        for k in range(3000):
            y = u + beta * (u - old)
            old, u = u, simplex_rows(y - (self.m0 * y + te * self.stiff(y) - b) / (2 * D))
            if k % 20 == 19 and float((u - old).abs().max()) < 3e-15:
                break
        return u

    def step(self, u):
        return self.minimise(self.rhs(u, self.eps, self.lam), u)

    def planes(self, rows):
        return rows.t().reshape(self.N, self.H + 1, self.W + 1).contiguous()

    def rows(self, planes):
        return planes.reshape(self.N, -1).t().contiguous()


class ExactStep(torch.autograd.Function):
    """The step's minimiser, differentiated with its active set frozen."""

    @staticmethod
    def forward(ctx, b, eps, u, grid):
        new = grid.minimise(b, u)
        ctx.grid, ctx.new = grid, new
        return new

    @staticmethod
    def backward(ctx, g):
        grid, new = ctx.grid, ctx.new
        free = new > 0
        count = free.sum(0)
        free = free & (count >= 2)
        te, D = grid.tau * grid.eps, grid.diagonal()

        def tangent(v):
            v = torch.where(free, v, 0.0)
            return torch.where(free, v - v.sum(0) / count.clamp(min=1), 0.0)

        r = tangent(g)
        w, z = torch.zeros_like(r), tangent(r / D)
        p, rz, top = z, (r * z).sum(), r.abs().max()
        for _ in range(2000):
            if not float(r.abs().max()) > 1e-15 * float(top):
                break
            q = tangent(grid.m0 * p + te * grid.stiff(p))
            a = rz / (p * q).sum()
            w, r = w + a * p, r - a * q
            z = tangent(r / D)
            rz, old = (r * z).sum(), rz
            p = z + rz / old * p
        return w, -grid.tau * (w * grid.stiff(new)).sum(), None, None


def stored(image, case):
    """The image as the precision keeps it."""
    return image.bfloat16().double() if case["precision"] == "mixed" else image.double()


def exact(case, seed):
    tau = case["eps"] ** 2
    if case["kind"] == "batch":
        out = []
        for (W, H, N, _), p in zip(batch_images(case), batch_pictures(case, seed)):
            g = Grid(stored(p.image, case), N, case["eps"], case["lam"], tau, 0, "simplex")
            u = g.planes(p.u0)
            for _ in range(case["steps"]):
                u = g.step(u)
            out.append(g.rows(u))
        return out
    pic = one_picture(case, seed)
    if case["kind"] == "train":
        image = pic.image.double().requires_grad_()
        lam = torch.tensor(case["lam"], dtype=torch.float64, device="cuda", requires_grad=True)
        eps = torch.tensor(case["eps"], dtype=torch.float64, device="cuda", requires_grad=True)
        u0 = pic.u0.clone().requires_grad_()
        g = Grid(image, case["N"], case["eps"], case["lam"], tau, 0, "simplex")
        u = g.planes(u0)
        for _ in range(case["steps"]):
            u = ExactStep.apply(g.rhs(u, eps, lam), eps, u.detach(), g)
        rows = g.rows(u)
        onehot = torch.nn.functional.one_hot(target_labels(case, seed), case["N"]).double()
        loss = 0.5 * (node_mass(case["W"], case["H"]).reshape(-1, 1) * (rows - onehot) ** 2).sum()
        grads = torch.autograd.grad(loss, [image, lam, eps, u0])
        return {"u": rows.detach(), "loss": loss.detach(), "image": grads[0], "lam": grads[1], "eps": grads[2],
                "u0": grads[3]}
    g = Grid(stored(pic.image, case), case["N"], case["eps"], case["lam"], tau, case["refine"], case["projection"])
    u = g.planes(pic.u0)
    for k in range(case["steps"]):
        energy = float(g.energy(u)) if k == case["steps"] - 1 else None
        u = g.step(u)
    if case["kind"] == "step":
        return {"u": g.rows(u), "energy": energy}
    c = g.means(u)[0]
    mean = (2 * u[:, :-1, :-1] + u[:, :-1, 1:] + u[:, 1:, :-1] + 2 * u[:, 1:, 1:]) / 6
    return {"u": g.rows(u), "labels": None, "composite": torch.einsum("nc,nyx->yxc", c, mean)}
