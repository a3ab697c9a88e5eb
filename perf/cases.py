"""Timed cases of the functional-map path, through the calls a user's program makes.

A case names one of seven kinds of call and its sizes:

  pair        project + solve of one pair: interactive matching, evaluation one pair at a time
  autograd    FmapFunction inside a torch graph, forward and backward, one pair: the paper's
              training loop (batches of one pair)
  projection  project + project_backward of a set of shapes: the layer around the features
  solver      solve + loss_orth + adjoint from resident descriptors A: the map layer of a
              training step whose features are already spectral
  train       project, solve, loss_orth, solve_backward: the whole differentiable step
  gradfeat    spatial gradient features of a set of shapes (block-diagonal operator)
  overlap     overlap-prediction metrics of a set of segments

Inputs follow the recipe of the repository's synthetic shapes (M-orthonormal Gaussian bases,
masses U[0.5, 1.5]/n, eigenvalues sorted U[0, 100], features N(0, 1)), drawn on the GPU.
Sizes of a ragged set are log-uniform and belong to the case (`sizes` seeds them); the values
belong to the seed.
"""
import math
import random

import numpy as np
import torch

from paper_2604_10377_gb300 import api

DEV = "cuda:0"


# ------------------------------------------------------------------------------ the cases
def listed():
    return [
        # one small pair, forward only, FP32 features: launches and latency are what counts
        dict(name="pair_small_fp32", kind="pair", n=5000, kx=30, d=128, feat="fp32"),
        # the training loop over single pairs at the paper's usual spectral size, through autograd
        dict(name="autograd_pair_k200", kind="autograd", n=5000, kx=200, d=256, feat="bf16"),
        # FP32 features of a ragged batch of 32 pairs: the projection and its gradient
        dict(name="projection_fp32_k50", kind="projection", shapes=64, n_lo=5000, n_hi=50000, sizes=1, k="50", d=256,
             feat="fp32"),
        # dense scans with a large spectrum: the largest bases and widest features
        dict(name="projection_bf16_k200", kind="projection", shapes=8, n_lo=200000, n_hi=200000, sizes=1, k="200",
             d=512, feat="bf16"),
        # the largest spectral sizes of the paper's sweep, one pair
        dict(name="solver_pair_k300", kind="solver", pairs=1, k="300", ky="", d=512, sizes=1, mask=False,
             recompute=False),
        # large spectrum with factors recomputed in the backward pass to bound memory
        dict(name="solver_recompute_k200", kind="solver", pairs=4, k="200", ky="", d=512, sizes=1, mask=False,
             recompute=True),
        # maps between bases of different odd sizes, with an explicit mask
        dict(name="solver_rect_mask", kind="solver", pairs=24, k="77,121,150", ky="65,99,160", d=208, sizes=2,
             mask=True, recompute=False),
        # the map layer of the ragged mixed batch
        dict(name="solver_ragged_256", kind="solver", pairs=256, k="30,50,100,200", ky="", d=256, sizes=4, mask=False,
             recompute=False),
        # a training step on eight pairs of remeshed shapes, BF16 features
        dict(name="train_k100", kind="train", pairs=8, n_lo=20000, n_hi=20000, sizes=1, k="100", d=384, feat="bf16"),
        # the headline step: 256 ragged pairs with mixed spectral sizes
        dict(name="train_ragged_256", kind="train", pairs=256, n_lo=1000, n_hi=100000, sizes=4, k="30,50,100,200",
             d=256, feat="bf16"),
        # gradient features of 64 ragged shapes, written as BF16 projection input
        dict(name="gradfeat_64", kind="gradfeat", shapes=64, n_lo=1000, n_hi=100000, sizes=7, dim=128, out="bf16",
             variant="A"),
        # evaluation of a partial-matching set: one segment per shape
        dict(name="overlap_4096", kind="overlap", segments=4096, n_lo=1000, n_hi=100000, sizes=9),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["pair", "autograd", "projection", "projection", "solver", "solver", "train", "train", "gradfeat",
                       "overlap"])
    feat = rng.choice(["fp32", "bf16"])
    d = 16 * _logu(rng, 2, 32)
    k_top = min(300, 4 * d // 5)     # descriptors outnumber the basis functions
    sizes = rng.randrange(1 << 20)
    if kind in ("pair", "autograd"):
        return dict(kind=kind, n=_logu(rng, 1000, 50000), kx=rng.randint(10, k_top), d=d, feat=feat)
    if kind == "projection":
        n_hi = _logu(rng, 2000, 200000)
        count = max(1, min(_logu(rng, 1, 96), int(3.0e6 / n_hi)))
        ks = ",".join(str(rng.randint(10, k_top)) for _ in range(rng.randint(1, 4)))
        return dict(kind=kind, shapes=count, n_lo=max(1000, n_hi // 20), n_hi=n_hi, sizes=sizes, k=ks, d=d, feat=feat)
    if kind == "solver":
        count = _logu(rng, 1, 96)
        top = k_top if count <= 32 else min(200, k_top)
        ks = [rng.randint(10, top) for _ in range(rng.randint(1, 4))]
        rect = rng.random() < 0.4
        kys = [rng.randint(10, top) for _ in ks] if rect else []
        return dict(kind=kind, pairs=count, k=",".join(map(str, ks)), ky=",".join(map(str, kys)), d=d, sizes=sizes,
                    mask=rng.random() < 0.3, recompute=rng.random() < 0.3)
    if kind == "train":
        n_hi = _logu(rng, 2000, 100000)
        count = max(1, min(_logu(rng, 1, 64), int(2.0e6 / n_hi)))
        ks = ",".join(str(rng.randint(10, min(200, k_top))) for _ in range(rng.randint(1, 4)))
        return dict(kind=kind, pairs=count, n_lo=max(1000, n_hi // 20), n_hi=n_hi, sizes=sizes, k=ks, d=d, feat=feat)
    if kind == "gradfeat":
        n_hi = _logu(rng, 2000, 100000)
        return dict(kind=kind, shapes=_logu(rng, 1, 64), n_lo=1000, n_hi=n_hi, sizes=sizes, dim=16 * rng.randint(2, 8),
                    out=rng.choice(["fp32", "bf16"]), variant=rng.choice(["A", "B"]))
    return dict(kind=kind, segments=_logu(rng, 1, 4096), n_lo=500, n_hi=_logu(rng, 1000, 100000), sizes=sizes)


# ------------------------------------------------------------------------------ sizes
def _ints(text):
    return [int(x) for x in text.split(",") if x]


def _ns(case, count):
    rng = random.Random(case["sizes"])
    return [_logu(rng, case["n_lo"], case["n_hi"]) for _ in range(count)]


def _shapes(case):
    """(n, k, d) of every shape, and (x, y) of every pair."""
    kind = case["kind"]
    if kind in ("pair", "autograd"):
        return [(case["n"], case["kx"], case["d"])] * 2, [(0, 1)]
    if kind == "projection":
        ns = _ns(case, case["shapes"])
        ks = _ints(case["k"])
        shapes = [(n, ks[(i // 2) % len(ks)], case["d"]) for i, n in enumerate(ns)]
        # consecutive shapes of one size are the batch's pairs (a pair may use a shape twice)
        return shapes, [(i, i + 1 if i + 1 < len(shapes) else i) for i in range(0, len(shapes), 2)]
    ks = _ints(case["k"])
    if kind == "solver":
        kys = _ints(case["ky"]) or ks
        pick = random.Random(case["sizes"])
        shapes = []
        for _ in range(case["pairs"]):
            j = pick.randrange(len(ks))
            # the bases themselves are not read by these calls: only their sizes matter
            shapes += [(64, ks[j], case["d"]), (64, kys[j], case["d"])]
    else:
        ns = _ns(case, 2 * case["pairs"])
        pick = random.Random(case["sizes"] + 1)
        kp = [ks[pick.randrange(len(ks))] for _ in range(case["pairs"])]
        shapes = [(n, kp[i // 2], case["d"]) for i, n in enumerate(ns)]
    return shapes, [(2 * p, 2 * p + 1) for p in range(case["pairs"])]


def _lams(case, n_pairs):
    rng = random.Random(31)
    return [float(np.float32(math.exp(rng.uniform(math.log(1e-4), math.log(1e-1))))) for _ in range(n_pairs)]


def _feat_dtype(case):
    return torch.bfloat16 if case.get("feat") == "bf16" else torch.float32


# ------------------------------------------------------------------------------ inputs
def _gen(seed, i):
    g = torch.Generator(device=DEV)
    g.manual_seed((int(seed) * 1000003 + 7919 * i + 17) % (1 << 62))
    return g


def _shape_inputs(case, seed, s, n, k, d, bases=True):
    """phi (n x k), mass (n), evals (k), feat (n x d) of shape s; without the bases, evals alone."""
    g = _gen(seed, 2 * s)
    evals = torch.sort(100.0 * torch.rand(k, generator=g, device=DEV)).values
    if not bases:
        return None, None, evals, None
    mass = (0.5 + torch.rand(n, generator=g, device=DEV)) / n
    phi = torch.randn(n, k, generator=g, device=DEV).double()
    # Phi^T M Phi = I by one Cholesky-QR pass in the M inner product
    chol = torch.linalg.cholesky(phi.T @ (mass.double()[:, None] * phi))
    eye = torch.eye(k, dtype=torch.float64, device=DEV)
    inv = torch.linalg.solve_triangular(chol, eye, upper=False)
    phi = (phi @ inv.T).float()
    feat = torch.randn(n, d, generator=g, device=DEV).to(_feat_dtype(case))
    return phi, mass, evals, feat


def _descriptor(seed, s, k, d):
    """A descriptor matrix as projected features of a 5000-vertex shape have it."""
    return torch.randn(k, d, generator=_gen(seed, 2 * s + 1), device=DEV) / math.sqrt(5000.0)


def _target(seed, p, ky, kx):
    """A target map: the leading block of a random orthogonal matrix."""
    m = max(ky, kx)
    q = torch.linalg.qr(torch.randn(m, m, generator=_gen(seed, 100000 + p), device=DEV)).Q
    return q[:ky, :kx]


def _mask(seed, p, ky, kx):
    return 50.0 * torch.rand(ky, kx, generator=_gen(seed, 200000 + p), device=DEV)


def _gradient_inputs(case, seed):
    """A block-diagonal complex gradient operator in CSR form over all shapes of the case: every
    vertex has itself and six others of its shape within 64 indices; rows sum to zero."""
    ns = _ns(case, case["shapes"])
    g = _gen(seed, 0)
    n = sum(ns)
    start = torch.repeat_interleave(torch.tensor(np.cumsum([0] + ns[:-1]), device=DEV), torch.tensor(ns, device=DEV))
    length = torch.repeat_interleave(torch.tensor(ns, device=DEV), torch.tensor(ns, device=DEV))
    local = torch.arange(n, device=DEV) - start
    # six distinct offsets in six disjoint ranges of +-64, folded back into the shape at its ends
    lanes = torch.tensor([-64, -43, -22, 1, 22, 43], device=DEV)
    off = lanes + torch.randint(0, 21, (n, 6), generator=g, device=DEV)
    nb = local[:, None] + off
    nb = torch.where(nb < 0, nb + 129, nb)
    nb = torch.where(nb >= length[:, None], nb - 129, nb)
    cols = torch.cat([nb, local[:, None]], 1) + start[:, None]
    cols, order = torch.sort(cols, 1)
    vals = torch.randn(n, 7, 2, generator=g, device=DEV) / math.sqrt(6.0)
    own = order == 6
    vals = torch.where(own[..., None], torch.zeros_like(vals), vals)
    vals = torch.where(own[..., None], -vals.sum(1, keepdim=True).expand_as(vals), vals)
    dim = case["dim"]
    row_ptr = torch.arange(0, 7 * n + 1, 7, dtype=torch.int64, device=DEV)
    x = torch.randn(n, dim, generator=g, device=DEV)
    a = torch.randn(2, dim, dim, generator=g, device=DEV) / math.sqrt(dim)
    return (row_ptr, cols.reshape(-1).to(torch.int32), vals.reshape(-1, 2).contiguous(), x, a[0].contiguous(),
            a[1].contiguous())


def _overlap_inputs(case, seed):
    offs = np.concatenate([[0], np.cumsum(_ns(case, case["segments"]))]).astype(np.int64)
    g = _gen(seed, 0)
    n = int(offs[-1])
    scores = torch.rand(n, generator=g, device=DEV)
    # labels agree with thresholded scores on about three vertices of four
    labels = ((scores > 0.5) ^ (torch.rand(n, generator=g, device=DEV) < 0.25)).to(torch.uint8)
    return scores, labels, offs


# ------------------------------------------------------------------------------ prepare, run
def prepare(case, seed):
    kind = case["kind"]
    st = dict(kind=kind)
    if kind == "gradfeat":
        st["in"] = _gradient_inputs(case, seed)
        n = st["in"][3].shape[0]
        st["out"] = torch.empty(n, case["dim"], device=DEV,
                                dtype=torch.bfloat16 if case["out"] == "bf16" else torch.float32)
        st["ws"] = torch.empty(4 * (2 * case["dim"]) ** 2, dtype=torch.uint8, device=DEV)
        st["variant"] = case["variant"]
        return st
    if kind == "overlap":
        st["in"] = _overlap_inputs(case, seed)
        return st
    shapes, pairs = _shapes(case)
    solver = kind == "solver"
    feat = case.get("feat", "fp32")
    lay = api.BatchLayout([n for n, _, _ in shapes], [k for _, k, _ in shapes], [d for _, _, d in shapes], feat)
    kx, ky = [shapes[x][1] for x, _ in pairs], [shapes[y][1] for _, y in pairs]
    masks = None
    if case.get("mask"):
        masks = [_mask(seed, p, ky[p], kx[p]).cpu().numpy() for p in range(len(pairs))]
    b = api.FmapBatch(lay, [(x, y, lam) for (x, y), lam in zip(pairs, _lams(case, len(pairs)))], device=DEV,
                      precision=feat, with_grad=kind not in ("pair", "solver"), masks=masks,
                      store_factors_max_k=0 if case.get("recompute") else 304)
    for s, (n, k, d) in enumerate(shapes):
        phi, mass, evals, f = _shape_inputs(case, seed, s, n, k, d, bases=not solver)
        b.evals[lay.evals_off[s]:lay.evals_off[s] + k] = evals
        if solver:
            b.a_view(b.A, s).copy_(_descriptor(seed, s, k, d))
            continue
        ld = lay.ld_phi[s]
        b.phi[lay.phi_off[s]:lay.phi_off[s] + n * ld].view(n, ld)[:, :k] = phi
        b.mass[lay.mass_off[s]:lay.mass_off[s] + n] = mass
        b.feat[lay.feat_off[s]:lay.feat_off[s] + n * d].view(n, d).copy_(f)
    st["b"] = b
    if kind == "autograd":
        st["feat"] = b.feat.clone().requires_grad_(True)
    if kind == "projection":
        b.dA.copy_(torch.cat([_descriptor(seed, s, k, d).reshape(-1) for s, (_, k, d) in enumerate(shapes)]))
    elif kind != "pair":
        gt = torch.cat([_target(seed, p, ky[p], kx[p]).reshape(-1) for p in range(len(pairs))])
        st["gt"] = gt
        st["loss"] = torch.zeros(len(pairs), device=DEV)
        st["dc"] = torch.empty_like(b.C)
    return st


def run(st):
    kind = st["kind"]
    if kind == "gradfeat":
        row_ptr, col, vals, x, a_re, a_im = st["in"]
        out, status = api.gradient_features(row_ptr, col, vals, x, a_re, a_im, variant=st["variant"], out=st["out"],
                                            ws=st["ws"])
        return dict(out=out, status=status)
    if kind == "overlap":
        counts, metrics = api.overlap_metrics(*st["in"])
        return dict(counts=counts, metrics=metrics)
    b = st["b"]
    if kind == "pair":
        a = b.project()
        c = b.solve(a, keep_factors=False)
        return dict(A=a, C=c, status=b.status)
    if kind == "autograd":
        c = api.FmapFunction.apply(st["feat"], b)
        (df,) = torch.autograd.grad(c, st["feat"], st["gt"])
        return dict(C=c.detach(), dF=df, status=b.status)
    if kind == "projection":
        a = b.project()
        b.project_backward()
        return dict(A=a, dF=b.dfeat)
    if kind == "solver":
        c = b.solve()
        loss, dc = b.loss_orth(c, st["gt"], loss=st["loss"], d_c=st["dc"])
        da = b.adjoint(dc)
        return dict(C=c, loss=loss, dC=dc, dA=da, status=b.status)
    a = b.project()
    c = b.solve(a)
    loss, dc = b.loss_orth(c, st["gt"], loss=st["loss"], d_c=st["dc"])
    da = b.solve_backward(dc, a, c)
    return dict(A=a, C=c, loss=loss, dC=dc, dA=da, dF=b.dfeat, status=b.status)


# ------------------------------------------------------------------------------ work
def work(case):
    kind = case["kind"]
    if kind == "overlap":
        n = sum(_ns(case, case["segments"]))
        return dict(bytes=5 * n + case["segments"] * (8 + 32 + 56), flops=0)
    if kind == "gradfeat":
        n, dim = sum(_ns(case, case["shapes"])), case["dim"]
        out = 2 if case["out"] == "bf16" else 4
        return dict(bytes=n * (8 + 7 * 12 + 4 * dim + out * dim) + 8 * dim * dim,
                    flops=n * (7 * dim * 4 + 8 * dim * dim + 4 * dim))
    shapes, pairs = _shapes(case)
    fb = 2 if case.get("feat") == "bf16" else 4
    nbytes = flops = 0.0
    if kind != "solver":
        for n, k, d in shapes:
            one = n * (4 * k + 4 + fb * d) + 4 * k * d
            passes = 1 if kind == "pair" else 2          # forward, and the gradient of the features
            nbytes += passes * one
            flops += passes * 2.0 * n * k * d
    if kind != "projection":
        for x, y in pairs:
            kx, ky, d = shapes[x][1], shapes[y][1], shapes[x][2]
            # forward: Gram and right-hand sides, ky factorisations, solve and one refinement
            flops += kx * (kx + 1) * d + 2.0 * kx * ky * d + ky * (kx ** 3 / 3.0 + 6.0 * kx * kx)
            nbytes += 4.0 * (kx * d + ky * d + kx * ky + (kx * ky if case.get("mask") else kx + ky))
            if kind != "pair":
                # loss, adjoint solves (factors again where they are recomputed), dA
                if kind != "autograd":
                    flops += 4.0 * ky * ky * kx
                flops += ky * (2.0 * kx * kx + (kx ** 3 / 3.0 if case.get("recompute") else 0.0))
                flops += 4.0 * kx * kx * ky + 2.0 * ky * kx * d + 2.0 * kx * (ky + kx) * d
                nbytes += 4.0 * (3 * kx * ky + 2 * (kx + ky) * d)
    return dict(bytes=nbytes, flops=flops)


# ------------------------------------------------------------------------------ exact
def _exact_map(ax, ay, evx, evy, lam, mask):
    """C and the Cholesky factors of its row systems, in 64 bits."""
    dm = mask.double() if mask is not None else (evy.double()[:, None] - evx.double()[None, :]) ** 2
    s = (ax @ ax.T)[None] + lam * torch.diag_embed(dm)
    chol = torch.linalg.cholesky(s)
    c = torch.cholesky_solve((ay @ ax.T)[..., None], chol)[..., 0]
    return c, chol


def _exact_adjoint(ax, ay, c, chol, dc):
    gam = torch.cholesky_solve(dc[..., None], chol)[..., 0]
    return gam.T @ ay - (gam.T @ c + c.T @ gam) @ ax, gam @ ax


def exact(case, seed):
    kind = case["kind"]
    f64 = torch.float64
    if kind == "overlap":
        scores, labels, offs = _overlap_inputs(case, seed)
        pred, lab = scores > 0.5, labels != 0
        counts = []
        for m in (pred & lab, pred & ~lab, ~pred & lab, ~pred & ~lab):
            run_sum = torch.cat([torch.zeros(1, dtype=torch.int64, device=DEV), torch.cumsum(m, 0)])
            at = run_sum[torch.from_numpy(offs).to(DEV)]
            counts.append(at[1:] - at[:-1])
        tp, fp, fn, tn = [x.to(f64) for x in counts]
        rec, spec = tp / (tp + fn), tn / (tn + fp)
        metrics = torch.stack([tp / (tp + fp + fn), (rec + spec) / 2, (tp + tn) / (tp + fp + fn + tn), tp / (tp + fp),
                               rec, spec, 2 * tp / (2 * tp + fp + fn)], 1)
        return dict(counts=torch.stack(counts, 1), metrics=metrics)
    if kind == "gradfeat":
        row_ptr, col, vals, x, a_re, a_im = _gradient_inputs(case, seed)
        n, dim = x.shape
        out = torch.empty(n, dim, dtype=f64, device=DEV)
        ar, ai = a_re.double(), a_im.double()
        col, vals = col.view(n, 7).long(), vals.view(n, 7, 2)
        for i in range(0, n, 65536):
            rows, v = x[col[i:i + 65536]].double(), vals[i:i + 65536].double()
            zx = (v[:, :, 0, None] * rows).sum(1)
            zy = (v[:, :, 1, None] * rows).sum(1)
            p = zx @ ar.T - zy @ ai.T
            q = zy @ ar.T + zx @ ai.T if case["variant"] == "A" else zx @ ar.T + zy @ ai.T
            out[i:i + 65536] = zx * p + zy * q
        return dict(out=out, status=None)
    shapes, pairs = _shapes(case)
    lams = _lams(case, len(pairs))
    a_len = sum(k * d for _, k, d in shapes)
    a_off = np.concatenate([[0], np.cumsum([k * d for _, k, d in shapes])])
    c_off = np.concatenate([[0], np.cumsum([shapes[x][1] * shapes[y][1] for x, y in pairs])])
    f_off, cur = [], 0
    for n, _, d in shapes:                       # blocks of features start on multiples of 64 elements
        f_off.append(cur)
        cur = (cur + n * d + 63) // 64 * 64
    grads = kind != "pair"
    A = torch.zeros(a_len, dtype=f64, device=DEV)
    dA = torch.zeros(a_len, dtype=f64, device=DEV)
    dF = torch.zeros(cur if kind in ("projection", "train", "autograd") else 0, dtype=f64, device=DEV)
    C = torch.zeros(int(c_off[-1]), dtype=f64, device=DEV)
    dC = torch.zeros_like(C)
    loss = torch.zeros(len(pairs), dtype=f64, device=DEV)

    def at(flat, s):
        return flat[int(a_off[s]):int(a_off[s + 1])].view(shapes[s][1], shapes[s][2])

    evals = []
    for s, (n, k, d) in enumerate(shapes):
        phi, mass, ev, f = _shape_inputs(case, seed, s, n, k, d, bases=kind != "solver")
        evals.append(ev)
        at(A, s).copy_(_descriptor(seed, s, k, d) if kind == "solver"
                       else (phi.double() * mass.double()[:, None]).T @ f.double())
        if kind == "projection":
            at(dA, s).copy_(_descriptor(seed, s, k, d))
    if kind != "projection":
        for p, (x, y) in enumerate(pairs):
            kx, ky = shapes[x][1], shapes[y][1]
            mask = _mask(seed, p, ky, kx) if case.get("mask") else None
            c, chol = _exact_map(at(A, x), at(A, y), evals[x], evals[y], lams[p], mask)
            lo, hi = int(c_off[p]), int(c_off[p + 1])
            C[lo:hi] = c.reshape(-1)
            if not grads:
                continue
            gt = _target(seed, p, ky, kx).double()
            if kind == "autograd":
                dc = gt
            else:
                e = c @ c.T - torch.eye(ky, dtype=f64, device=DEV)
                loss[p] = (e * e).sum() + ((c - gt) ** 2).sum()
                dc = 4 * e @ c + 2 * (c - gt)
            dC[lo:hi] = dc.reshape(-1)
            gx, gy = _exact_adjoint(at(A, x), at(A, y), c, chol, dc)
            at(dA, x).add_(gx)
            at(dA, y).add_(gy)
    if dF.numel():
        for s, (n, k, d) in enumerate(shapes):
            phi, mass, _, _ = _shape_inputs(case, seed, s, n, k, d)
            dF[f_off[s]:f_off[s] + n * d] = (mass.double()[:, None] * (phi.double() @ at(dA, s))).reshape(-1)
    if kind == "pair":
        return dict(A=A, C=C, status=None)
    if kind == "autograd":
        return dict(C=C, dF=dF, status=None)
    if kind == "projection":
        return dict(A=A, dF=dF)
    if kind == "solver":
        return dict(C=C, loss=loss, dC=dC, dA=dA, status=None)
    return dict(A=A, C=C, loss=loss, dC=dC, dA=dA, dF=dF, status=None)
