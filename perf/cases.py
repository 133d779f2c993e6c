"""The framework's work as a user's program has it do, for timing and for comparing results.

listed() names the cases; draw(rng) gives more of the same ranges; prepare(case, seed) makes the
inputs on the GPU; run(state) is one pass through the public entry points; work(case) counts
what a pass cannot do without; exact(case, seed) is the same result from plain torch in 64 bits.

Kinds of case:
  solve   the periodic nDGP solve of one density field and its force (solve_fifth_force): FP64 to
          1e-10 or mixed precision to 1e-8 / 1e-6, as a graph replay or driven from the host, from
          zero, from a full-multigrid start or from the field of the time step before
  batch   many boxes of different sides and couplings in one call (solve_batch)
  truncate  a refinement that is only interpolated from its parent, and its force
  refine  a refinement interpolated from its parent, relaxed, and its force
"""
import math
import random

import torch

import paper_1511_08200_gb300 as mg

BOX = 250.0                 # Mpc/h, the side of the periodic box
H_DOMAIN = BOX / 128        # spacing of the domain grid above a refinement
OMEGA_M0, H0RC = 0.3, 1.0   # background of the nDGP coefficients


def listed():
    return [
        # The truncated level of the paper: phi of a 64^3 refinement interpolated from a 128^3
        # domain and differenced, once per refinement and time step: the smallest call.
        dict(name="truncate_64", kind="truncate", nc=128, p0=32, p1=32, p2=32, sigma=1.5),
        # A small box to 1e-10 by graph replay: all of it fits in L2, launches and latency count.
        dict(name="fp64_32_graph", kind="solve", n=32, precision="fp64", tol=1e-10, sigma=1.0,
             start="zero", graph=True, nu1=2, nu2=2, nu_coarse=500),
        # The domain grid of the refinement step: full-multigrid start, V(3,1), capped bottom.
        dict(name="fp64_128_fmg_graph", kind="solve", n=128, precision="fp64", tol=1e-10, sigma=1.5,
             start="fmg", graph=True, nu1=3, nu2=1, nu_coarse=4),
        # An N-body code's time step: default parameters, driven from the host, warm-started with
        # the field of the step before; a side that is no power of two.
        dict(name="fp64_96_warm", kind="solve", n=96, precision="fp64", tol=1e-10, sigma=1.0,
             start="warm", graph=False, nu1=2, nu2=2, nu_coarse=500),
        # A side that stops halving at 18^3.
        dict(name="fp64_144", kind="solve", n=144, precision="fp64", tol=1e-10, sigma=1.5,
             start="zero", graph=False, nu1=2, nu2=2, nu_coarse=500),
        # The default call on a large grid.
        dict(name="fp64_256", kind="solve", n=256, precision="fp64", tol=1e-10, sigma=1.5,
             start="zero", graph=False, nu1=2, nu2=2, nu_coarse=500),
        # The refinement level solved beside its interpolated form.
        dict(name="refine_64_graph", kind="refine", nc=128, p0=32, p1=32, p2=32, sigma=1.5,
             graph=True, nu_coarse=4),
        # A ragged refinement, default parameters, driven from the host.
        dict(name="refine_ragged", kind="refine", nc=96, p0=24, p1=20, p2=36, sigma=1.0,
             graph=False, nu_coarse=500),
        # The mixed-precision solve of the domain grid.
        dict(name="mixed_128_graph", kind="solve", n=128, precision="mixed", tol=1e-8, sigma=1.5,
             start="zero", graph=True, nu1=2, nu2=2, nu_coarse=500),
        # A served request: loose tolerance, a side that stops halving at 30^3.
        dict(name="mixed_240", kind="solve", n=240, precision="mixed", tol=1e-6, sigma=2.0,
             start="zero", graph=False, nu1=2, nu2=2, nu_coarse=500),
        # The largest grid of the benchmark.
        dict(name="mixed_512", kind="solve", n=512, precision="mixed", tol=1e-8, sigma=2.0,
             start="zero", graph=False, nu1=2, nu2=2, nu_coarse=500),
        # Many boxes in one launch.
        dict(name="batch_24", kind="batch", boxes=24, mix=4, smallest=32, largest=128, sigma=1.0,
             tol=1e-8),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(rng, lo, hi):
    """A side the hierarchy takes: a multiple of 4 whose odd part is at most 15."""
    while True:
        n = 4 * max(1, round(_log_uniform(rng, lo, hi) / 4))
        odd = n
        while odd % 2 == 0:
            odd //= 2
        if odd <= 15 and lo <= n <= hi:
            return n


def draw(rng: random.Random):
    kind = rng.choice(["fp64", "fp64", "fp64", "mixed", "mixed", "refine", "refine", "truncate", "batch"])
    sigma = round(rng.uniform(0.5, 1.5), 3)
    if kind == "fp64":
        start = rng.choice(["zero", "fmg", "warm"])
        nu1, nu2 = rng.choice([(2, 2), (3, 1)])
        return dict(kind="solve", n=_side(rng, 16, 256), precision="fp64", tol=1e-10, sigma=sigma,
                    start=start, graph=start != "warm" and rng.random() < 0.5, nu1=nu1, nu2=nu2,
                    nu_coarse=rng.choice([4, 500]))
    if kind == "mixed":
        start = rng.choice(["zero", "zero", "warm"])
        return dict(kind="solve", n=_side(rng, 16, 384), precision="mixed", tol=rng.choice([1e-6, 1e-8]),
                    sigma=sigma, start=start, graph=start != "warm" and rng.random() < 0.5, nu1=2, nu2=2,
                    nu_coarse=500)
    if kind == "batch":
        return dict(kind="batch", boxes=rng.randrange(2, 25), mix=rng.randrange(1000), smallest=32,
                    largest=rng.choice([64, 96, 128]), sigma=sigma, tol=rng.choice([1e-6, 1e-8]))
    # windows of the parent, each axis its own extent
    p = [2 * max(4, round(_log_uniform(rng, 8, 48) / 2)) for _ in range(3)]
    case = dict(kind=kind, nc=128, p0=p[0], p1=p[1], p2=p[2], sigma=sigma)
    if kind == "refine":
        case.update(graph=rng.random() < 0.5, nu_coarse=rng.choice([4, 500]))
    return case


# ------------------------------------------------------------------ inputs

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _delta(n, sigma, seed, growth=1.0):
    """Lognormal density contrast, P(k) ~ k^-2 up to the Nyquist sphere; `growth` scales the
    Gaussian field (an earlier time of the same realisation)."""
    dev = _device()
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    w = torch.fft.rfftn(torch.randn((n, n, n), generator=g, device=dev, dtype=torch.float64))
    fi = torch.fft.fftfreq(n, 1.0 / n, device=dev, dtype=torch.float64)
    fk = torch.fft.rfftfreq(n, 1.0 / n, device=dev, dtype=torch.float64)
    k = torch.sqrt(fi[:, None, None] ** 2 + fi[None, :, None] ** 2 + fk[None, None, :] ** 2)
    amp = torch.where((k > 0) & (2 * k <= n), 1.0 / torch.clamp(k, min=1.0), torch.zeros_like(k))
    x = torch.fft.irfftn(w * amp, s=(n, n, n))
    x -= x.mean()
    x *= growth * sigma / x.std(unbiased=False)
    x = torch.exp(x - 0.5 * (growth * sigma) ** 2)
    return (x / x.mean() - 1.0).contiguous()


def _coefficients():
    """(beta, alpha, s) of the normal-branch DGP background at a = 1, lengths in Mpc/h."""
    h0 = 1.0 / 2997.92458
    beta = 1.0 + 2.0 * H0RC * (1.0 - 0.5 * OMEGA_M0)
    return beta, (H0RC / h0) ** 2 / (3.0 * beta), OMEGA_M0 * h0 ** 2 / beta


def _batch_boxes(case, seed):
    """(side, factor on alpha, seed of the field) per box; `mix` fixes the sides and the couplings."""
    rng = random.Random(case["mix"])
    sides = [n for n in (32, 48, 64, 96, 128) if case["smallest"] <= n <= case["largest"]]
    return [(rng.choice(sides), 10.0 ** rng.uniform(-1.0, 1.0), seed * 64 + b) for b in range(case["boxes"])]


def _refinement(case, seed):
    """Parent field phi, fine density under the window, window origin, compatibility constant."""
    nc, p = case["nc"], [case["p0"], case["p1"], case["p2"]]
    fine = _delta(2 * nc, case["sigma"], seed)
    coarse = fine.reshape(nc, 2, nc, 2, nc, 2).mean(dim=(1, 3, 5))
    # the window around the densest cell of a smoothed field
    sm = torch.nn.functional.avg_pool3d(coarse[None, None].float(), 8)[0, 0]
    at = int(sm.argmax())
    m = nc // 8
    o = [(c * 8 + 4 - q // 2) % nc for c, q in zip((at // (m * m), at // m % m, at % m), p)]
    idx = [(2 * a + torch.arange(2 * q, device=fine.device)) % (2 * nc) for a, q in zip(o, p)]
    patch = fine[idx[0][:, None, None], idx[1][None, :, None], idx[2][None, None, :]].contiguous()
    _, alpha, s = _coefficients()
    phi, c = _solve(s * coarse, H_DOMAIN, alpha, 1e-11)
    return phi, patch, o, p, c


_context = []


def _shared_context():
    """The one handle that a program keeps: hierarchies and captured solves by size."""
    if not _context:
        _context.append(mg.Context(0))
    return _context[0]


def _params(case, alpha, s, h):
    return mg.default_params(alpha=alpha, s=s, h=h, tol=case["tol"], precision=case["precision"],
                             nu1=case["nu1"], nu2=case["nu2"], nu_coarse=case["nu_coarse"])


def prepare(case, seed):
    kind = case["kind"]
    new = dict(dtype=torch.float64, device=_device())
    _, alpha, s = mg.ndgp_coefficients(1.0, OMEGA_M0, H0RC)
    if kind == "solve":
        n = case["n"]
        st = dict(case=case, ctx=_shared_context(), delta=_delta(n, case["sigma"], seed),
                  params=_params(case, alpha, s, BOX / n), phi=torch.zeros((n, n, n), **new),
                  grad=torch.empty((3, n, n, n), **new))
        if case["start"] == "warm":
            st["before"] = _solve(s * _delta(n, case["sigma"], seed, 0.97), BOX / n, alpha, 1e-8)[0]
        return st
    if kind == "batch":
        boxes = _batch_boxes(case, seed)
        return dict(case=case, ctx=mg.Context(0), deltas=[_delta(n, case["sigma"], sd) for n, _, sd in boxes],
                    params=[mg.default_params(alpha=alpha * a, s=s, h=BOX / n, tol=case["tol"],
                                              precision="mixed") for n, a, _ in boxes],
                    phis=[torch.zeros((n, n, n), **new) for n, _, _ in boxes],
                    grads=[torch.empty((3, n, n, n), **new) for n, _, _ in boxes])
    phi, patch, o, p, c = _refinement(case, seed)
    st = dict(case=case, ctx=_shared_context(), phi=phi, origin=o, pn=p,
              box=torch.empty([2 * q + 2 for q in p], **new), grad=torch.empty([3] + [2 * q for q in p], **new))
    if kind == "refine":
        st.update(patch=patch, compat_c=c,
                  params=mg.default_params(alpha=alpha, s=s, h=H_DOMAIN / 2, tol=1e-10,
                                           nu_coarse=case["nu_coarse"]))
    return st


# ------------------------------------------------------------------ one pass

def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "solve":
        warm = case["start"] == "warm"
        if warm:
            state["phi"].copy_(state["before"])
        phi, grad, _ = ctx.solve_fifth_force(state["delta"], state["params"], phi=state["phi"],
                                             grad=state["grad"], warm=warm, fmg=case["start"] == "fmg",
                                             graph=case["graph"])
        return {"phi": phi, "grad": grad}
    if kind == "batch":
        phis, grads, _ = ctx.solve_batch(state["deltas"], state["params"], phis=state["phis"],
                                         grads=state["grads"])
        return {"phi": phis, "grad": grads}
    box = ctx.refine_interpolate(state["phi"], state["origin"], state["pn"], 1, out=state["box"])
    if kind == "refine":
        ctx.relax_patch(state["patch"], state["params"], state["compat_c"], box, graph=case["graph"])
    grad = ctx.force(box, H_DOMAIN / 2, ghost=1, periodic=False, grad=state["grad"])
    return {"phi": box, "grad": grad}


# ------------------------------------------------------------------ what it cannot do without

# Operations of a cell update and of a cell's residual, counted one by one from the discrete
# equation (a fused multiply-add as two, a root and a quotient as one each).
UPDATE_FLOPS, RESIDUAL_FLOPS = 40, 38


def _solve_work(cells, cycles):
    """V(2,2) cycles over a hierarchy of 8/7 of the finest grid's cells; density in, phi and its
    gradient out."""
    return 5 * 8 * cells, cycles * cells * 8 / 7 * (4 * UPDATE_FLOPS + RESIDUAL_FLOPS)


def work(case):
    kind = case["kind"]
    if kind == "solve":
        cycles = {1e-6: 4, 1e-8: 5, 1e-10: 6}[case["tol"]]
        b, f = _solve_work(case["n"] ** 3, cycles)
        return {"bytes": b + (8 * case["n"] ** 3 if case["start"] == "warm" else 0), "flops": f}
    if kind == "batch":
        cells = sum(n ** 3 for n, _, _ in _batch_boxes(case, 0))
        b, f = _solve_work(cells, 5)
        return {"bytes": b, "flops": f}
    p = [case["p0"], case["p1"], case["p2"]]
    window = math.prod(q + 2 for q in p)
    box, inner = math.prod(2 * q + 2 for q in p), math.prod(2 * q for q in p)
    b, f = 8 * (window + box + 3 * inner), 13 * box + 6 * inner
    if kind == "refine":
        b, f = b + 8 * inner, f + 6 * inner * 8 / 7 * (4 * UPDATE_FLOPS + RESIDUAL_FLOPS)
    return {"bytes": b, "flops": f}


# ------------------------------------------------------------------ the same in plain torch

def _parts(u, h):
    """L and Sigma with L^2 - (d_i d_j phi)^2 = (2/3) L^2 - Sigma on the interior of u (one ghost
    cell a side): Sigma = (1/3) sum (D_aa - D_bb)^2 + 2 sum D_ab^2 holds no centre value."""
    def sh(a, b, c):
        n = u.shape
        return u[1 + a:n[0] - 1 + a, 1 + b:n[1] - 1 + b, 1 + c:n[2] - 1 + c]
    h2 = h * h
    two = 2.0 * sh(0, 0, 0)
    xx = (sh(1, 0, 0) + sh(-1, 0, 0) - two) / h2
    yy = (sh(0, 1, 0) + sh(0, -1, 0) - two) / h2
    zz = (sh(0, 0, 1) + sh(0, 0, -1) - two) / h2
    del two
    lap = xx + yy + zz
    sigma = ((xx - yy) ** 2 + (xx - zz) ** 2 + (yy - zz) ** 2) / 3.0
    del xx, yy, zz
    for a, b in (((1, 0, 0), (0, 1, 0)), ((1, 0, 0), (0, 0, 1)), ((0, 1, 0), (0, 0, 1))):
        pp = [x + y for x, y in zip(a, b)]
        pm = [x - y for x, y in zip(a, b)]
        mm, mp = [-x for x in pp], [-x for x in pm]
        d = (sh(*pp) - sh(*pm) - sh(*mp) + sh(*mm)) / (4.0 * h2)
        sigma += 2.0 * d * d
    return lap, sigma


def _defect(f, u, h, alpha, centred):
    """r = f + c - op(u) (c makes its mean zero if `centred`, else c = 0), and the change of L
    that solves each cell's equation for its own value, its neighbours' combination Sigma held."""
    lap, sigma = _parts(u, h)
    b = f + alpha * sigma
    r = b - lap - (2.0 * alpha / 3.0) * lap * lap
    c = -float(r.mean()) if centred else 0.0
    r += c
    b += c
    root = 2.0 * b / (1.0 + torch.sqrt(torch.clamp(1.0 + (8.0 * alpha / 3.0) * b, min=0.0)))
    return r, root - lap, c


def _wrap(phi):
    for d in range(3):
        n = phi.shape[d]
        phi = torch.cat([phi.narrow(d, n - 1, 1), phi, phi.narrow(d, 0, 1)], dim=d)
    return phi


def _inverse_laplacian(r, h):
    """Periodic 7-point Laplacian, zero mean."""
    n = r.shape[0]
    x = torch.arange(n, device=r.device, dtype=torch.float64)
    e = -4.0 / (h * h) * torch.sin(math.pi * x / n) ** 2
    lam = e[:, None, None] + e[None, :, None] + e[None, None, :n // 2 + 1]
    lam[0, 0, 0] = 1.0
    rk = torch.fft.rfftn(r).div_(lam)
    rk[0, 0, 0] = 0.0
    return torch.fft.irfftn(rk, s=r.shape)


def _sine(x, d):
    """Discrete sine transform of type 1 along d (its own inverse up to 2 / (n + 1))."""
    n = x.shape[d]
    z = torch.zeros_like(x.narrow(d, 0, 1))
    y = torch.fft.rfft(torch.cat([z, x, z, -x.flip(d)], dim=d), dim=d)
    return -0.5 * y.imag.narrow(d, 1, n)


def _inverse_laplacian_box(r, h):
    """7-point Laplacian with zero values on the ghost cells."""
    lam = 0.0
    for d in range(3):
        n = r.shape[d]
        k = torch.arange(1, n + 1, device=r.device, dtype=torch.float64)
        e = -4.0 / (h * h) * torch.sin(0.5 * math.pi * k / (n + 1)) ** 2
        lam = lam + e.reshape([-1 if a == d else 1 for a in range(3)])
        r = _sine(r, d)
    r = r / lam
    for d in range(3):
        r = _sine(r, d) * (2.0 / (r.shape[d] + 1))
    return r


def _accelerate(x, defect, precondition, tol, steps, depth=10):
    """x <- x + precondition(defect) with Anderson's acceleration until the residual has fallen
    below tol or no longer falls."""
    dx, dg, last = [], [], None
    best, best_x, stale = math.inf, x, 0
    for _ in range(steps):
        size, change = defect(x)
        if size < best:
            best, best_x, stale = size, x, 0
        else:
            stale += 1
        if size <= tol or stale > 12:
            break
        g = precondition(change)
        del change
        if last is not None:
            dx.append(x - last[0])
            dg.append(g - last[1])
            dx, dg = dx[-depth:], dg[-depth:]
        last = (x, g)
        new = x + g
        if dg:
            scale = [float(q.norm()) for q in dg]
            a = torch.tensor([[float((p * q).sum()) / (u * v) for q, v in zip(dg, scale)]
                              for p, u in zip(dg, scale)], dtype=torch.float64)
            b = torch.tensor([float((p * g).sum()) / u for p, u in zip(dg, scale)], dtype=torch.float64)
            w = torch.linalg.lstsq(a, b[:, None], driver="gelsd").solution[:, 0]
            for c, p, q, u in zip(w.tolist(), dx, dg, scale):
                new = new - (c / u) * (p + q)
        x = new
    return best_x


def _solve(f, h, alpha, tol, steps=300):
    """The periodic field with op(phi) = f + c, mean(phi) = 0, and c."""
    norm = float(f.norm())
    c = [0.0]

    def defect(phi):
        r, change, c[0] = _defect(f, _wrap(phi), h, alpha, True)
        return float(r.norm()) / norm, change

    phi = _accelerate(torch.zeros_like(f), defect, lambda r: _inverse_laplacian(r, h), tol, steps)
    defect(phi)
    return phi - phi.mean(), c[0]


def _relax(f, box, h, alpha, tol, steps=300):
    """The interior of box with op = f, its ghost cells fixed."""
    norm = float(f.norm())
    out = box.clone()

    def defect(u):
        out[1:-1, 1:-1, 1:-1] = u
        r, change, _ = _defect(f, out, h, alpha, False)
        return float(r.norm()) / norm, change

    u = _accelerate(box[1:-1, 1:-1, 1:-1].clone(), defect, lambda r: _inverse_laplacian_box(r, h), tol, steps)
    out[1:-1, 1:-1, 1:-1] = u
    return out


def _gradient(u, h):
    """Central differences on the interior of u."""
    c = slice(1, -1)
    return torch.stack([u[2:, c, c] - u[:-2, c, c], u[c, 2:, c] - u[c, :-2, c],
                        u[c, c, 2:] - u[c, c, :-2]]) / (2.0 * h)


def _interpolate(phi, o, p):
    """Cell-centred trilinear interpolation onto the window's fine cells and one ghost cell."""
    n = phi.shape[0]
    for d in range(3):
        fine = torch.arange(-1, 2 * p[d] + 1, device=phi.device)
        t4 = 4 * o[d] + 2 * fine - 1
        i0 = torch.div(t4, 4, rounding_mode="floor")
        w = ((t4 - 4 * i0).to(torch.float64) / 4).reshape([-1 if a == d else 1 for a in range(3)])
        phi = phi.index_select(d, i0 % n) * (1 - w) + phi.index_select(d, (i0 + 1) % n) * w
    return phi.contiguous()


def exact(case, seed):
    kind = case["kind"]
    _, alpha, s = _coefficients()
    if kind == "solve":
        n = case["n"]
        phi, _ = _solve(s * _delta(n, case["sigma"], seed), BOX / n, alpha, 1e-13)
        return {"phi": phi, "grad": _gradient(_wrap(phi), BOX / n)}
    if kind == "batch":
        phis = [(_solve(s * _delta(n, case["sigma"], sd), BOX / n, alpha * a, 1e-12)[0], BOX / n)
                for n, a, sd in _batch_boxes(case, seed)]
        return {"phi": [p for p, _ in phis], "grad": [_gradient(_wrap(p), h) for p, h in phis]}
    phi, patch, o, p, c = _refinement(case, seed)
    box = _interpolate(phi, o, p)
    if kind == "refine":
        box = _relax(s * patch + c, box, H_DOMAIN / 2, alpha, 1e-13)
    return {"phi": box, "grad": _gradient(box, H_DOMAIN / 2)}
