"""Performance cases: what a program does with the bundle adjuster, through its Python entry points.

Kinds of case
  solve     a bound `binding.Problem`: parameters in from device tensors, one LM + PCG solve,
            parameters out (a reconstruction re-solved from new starting values);
  full      the same from host arrays, with the problem created and bound in the pass (a
            reconstruction solved once);
  evaluate  cost, residuals and Jacobian blocks at given parameters (covariances, outlier
            tests, a caller's own optimiser);
  gradient  cost and gradients through torch.autograd, float32 or float64 (the cost as a
            term of a training loss);
  batch     many small problems in one `binding.Batch` solve (submaps, per-object solves).

Inputs follow the recipe of `synth.py` (ring of cameras, points seen by 2 + Poisson or
2 + geometric cameras, pixel noise, perturbed start), drawn on the GPU so that the largest
takes about a second; pixels are float32 values with half a pixel of noise, as a detector
gives them.  Iteration caps are those of a solve that is still descending, and PCG runs to its
cap or to a tight tolerance, where two runs can be compared.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2605_30583_gb300 import autograd, binding, synth

DEV = "cuda"
F64 = torch.float64


def _case(kind, n_cams, n_pts, views="poisson", mean=3.0, visibility="nearest", lm=5, pcg=20, tol=1e-4, precision="mixed",
          loss=0, loss_scale=1.0, retract=0, schur=0, factors="", dtype="float32", n_problems=1):
    return dict(kind=kind, n_cams=n_cams, n_pts=n_pts, views=views, mean=mean, visibility=visibility, lm=lm, pcg=pcg,
                tol=tol, precision=precision, loss=loss, loss_scale=loss_scale, retract=retract, schur=schur, factors=factors,
                dtype=dtype, n_problems=n_problems)


def listed():
    cases = [
        # a handful of images: latency of the launches and of the grid-wide waits
        ("solve_tiny", _case("solve", 16, 1000, visibility="uniform", lm=5, pcg=20)),
        # a single object, outliers expected: Huber loss and the tangent-space rotation update
        ("solve_robust", _case("solve", 200, 50_000, mean=4.0, lm=5, pcg=20, loss=1, loss_scale=2.0, retract=1)),
        # a video or street sequence, default options
        ("solve_medium", _case("solve", 1000, 200_000, mean=4.0, lm=5, pcg=30)),
        # a sequence with odometry: relative-pose factors between neighbouring cameras
        ("solve_factors", _case("solve", 1000, 200_000, mean=4.0, lm=4, pcg=20, factors="chain+skip")),
        # more points than the chip's shared memory holds, ragged sizes
        ("solve_ragged", _case("solve", 997, 345_679, views="geometric", mean=4.4, lm=3, pcg=20)),
        # a city-scale reconstruction, the largest workload of the benchmark
        ("solve_large", _case("solve", 13_000, 4_500_000, views="geometric", mean=4.4, lm=3, pcg=20)),
        # the camera Schur complement, for scenes whose points are plentiful and cameras few
        ("solve_schur", _case("solve", 331, 70_001, mean=4.0, lm=4, pcg=20, schur=1)),
        # everything in double precision
        ("solve_fp64", _case("solve", 200, 50_000, mean=4.0, lm=3, pcg=15, precision="fp64")),
        # a sequence solved once, from the arrays that a feature matcher leaves on the host
        ("full_medium", _case("full", 1000, 200_000, mean=4.0, lm=4, pcg=20)),
        # residuals and Jacobian blocks of a whole sequence
        ("evaluate_medium", _case("evaluate", 1000, 200_000, mean=4.0)),
        # the cost as a training loss
        ("gradient", _case("gradient", 200, 50_000, mean=4.0)),
        # many submaps at once
        ("batch", _case("batch", 60, 5000, visibility="uniform", lm=3, pcg=20, n_problems=512)),
    ]
    return [dict(c, name=name) for name, c in cases]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["solve", "solve", "solve", "full", "evaluate", "gradient", "batch"])
    lm, pcg = rng.randint(2, 4), rng.randint(10, 30)
    if kind == "batch":
        return _case("batch", rng.randint(20, 60), rng.randint(500, 5000), mean=3.0, visibility="uniform",
                     lm=min(lm, 3), pcg=rng.randint(10, 20), n_problems=size(8, 500))
    views, mean = rng.choice([("poisson", 3.0), ("poisson", 4.0), ("geometric", 4.4)])
    n_cams = size(12, 4000)
    n_pts = max(size(300, 1_200_000), 20 * n_cams)
    c = dict(views=views, mean=mean, visibility="uniform" if n_cams <= 40 and n_pts <= 100_000 else "nearest", lm=lm,
             pcg=pcg)
    if kind == "solve":
        form = rng.choice(["plain", "plain", "huber", "cauchy", "retract", "schur", "factors", "fp64"])
        n_pts = min(n_pts, 200_000) if form == "fp64" else n_pts
        c.update({"huber": dict(loss=1, loss_scale=2.0), "cauchy": dict(loss=2, loss_scale=3.0),
                  "retract": dict(retract=1), "schur": dict(schur=1), "factors": dict(factors="chain"),
                  "fp64": dict(precision="fp64")}.get(form, {}))
    elif kind == "gradient":
        c["dtype"] = rng.choice(["float32", "float64"])
    return _case(kind, n_cams, n_pts, **c)


# ------------------------------------------------------------------------------- inputs ---


def _skew(v):
    o = torch.zeros_like(v[..., 0])
    return torch.stack([o, -v[..., 2], v[..., 1], v[..., 2], o, -v[..., 0], -v[..., 1], v[..., 0], o],
                       -1).reshape(*v.shape[:-1], 3, 3)


def _sinc_terms(th2):
    """sin t / t, (1 - cos t) / t^2 and (t - sin t) / t^3 of t^2, with series near zero."""
    small = th2 < 1e-6
    t = torch.sqrt(torch.where(small, torch.ones_like(th2), th2))
    a = torch.where(small, 1 - th2 / 6 + th2**2 / 120, torch.sin(t) / t)
    b = torch.where(small, 0.5 - th2 / 24 + th2**2 / 720, 2 * torch.sin(t / 2) ** 2 / t**2)
    c = torch.where(small, 1 / 6 - th2 / 120 + th2**2 / 5040, (t - torch.sin(t)) / t**3)
    return a[..., None, None], b[..., None, None], c[..., None, None]


def _exp(w):
    """Rotation matrix and left Jacobian of rotation vectors."""
    k = _skew(w)
    a, b, c = _sinc_terms((w * w).sum(-1))
    eye = torch.eye(3, dtype=w.dtype, device=w.device)
    return eye + a * k + b * (k @ k), eye + b * k + c * (k @ k)


def _quat_mul(p, q):
    p0, p1, p2, p3 = p.unbind(-1)
    q0, q1, q2, q3 = q.unbind(-1)
    return torch.stack([p0 * q0 - p1 * q1 - p2 * q2 - p3 * q3, p0 * q1 + p1 * q0 + p2 * q3 - p3 * q2,
                        p0 * q2 - p1 * q3 + p2 * q0 + p3 * q1, p0 * q3 + p1 * q2 - p2 * q1 + p3 * q0], -1)


def _to_quat(w):
    t = w.norm(dim=-1, keepdim=True).clamp_min(1e-300)
    return torch.cat([torch.cos(t / 2), torch.sin(t / 2) * w / t], -1)


def _to_rotvec(q):
    q = torch.where(q[..., :1] < 0, -q, q)
    n = q[..., 1:].norm(dim=-1, keepdim=True).clamp_min(1e-300)
    return 2 * torch.atan2(n, q[..., :1]) * q[..., 1:] / n


def _project(R, t, intr, X):
    P = (R * X[..., None, :]).sum(-1) + t
    p = -P[..., :2] / P[..., 2:]
    n2 = (p * p).sum(-1)
    s = 1 + intr[..., 1] * n2 + intr[..., 2] * n2 * n2
    return P, p, n2, s, (intr[..., 0] * s)[..., None] * p


def _inputs(case, seed):
    """A scene as CUDA tensors: prob_* give the problem of each camera, point and observation
    (all zero but for a batch), cam and pt are global.  The case alone decides the sizes (of
    every problem, and each point's number of views), the seed everything else."""
    sizes = torch.Generator(device=DEV)
    sizes.manual_seed(1)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def rand(*shape, generator=g):
        return torch.rand(*shape, generator=generator, device=DEV, dtype=F64)

    def randn(*shape):
        return torch.randn(*shape, generator=g, device=DEV, dtype=F64)

    P = case["n_problems"]
    if P > 1:   # uneven problems, up to the stated sizes
        nc = (5 + rand(P, generator=sizes) * (case["n_cams"] - 5)).long()
        npt = (case["n_pts"] // 25 + rand(P, generator=sizes) * (case["n_pts"] * 24 // 25)).long().clamp_min(20)
    else:
        nc = torch.full((1,), case["n_cams"], device=DEV)
        npt = torch.full((1,), case["n_pts"], device=DEV)
    C, N = int(nc.sum()), int(npt.sum())
    prob = torch.arange(P, device=DEV)
    prob_c, prob_p = prob.repeat_interleave(nc), prob.repeat_interleave(npt)
    cam0, pt0 = nc.cumsum(0) - nc, npt.cumsum(0) - npt
    radius = 5.0 * max(1.0, case["n_cams"] / 1000.0) if P == 1 else 5.0
    # cameras: a ring in the z = 0 plane looking inwards, R(az) = R_0 Rz(-az)
    az = 2 * math.pi * (torch.arange(C, device=DEV) - cam0[prob_c]).to(F64) / nc[prob_c]
    z = torch.zeros_like(az)
    q0 = torch.tensor([0.5, -0.5, -0.5, -0.5], device=DEV, dtype=F64).expand(C, 4)
    quat = _quat_mul(q0, torch.stack([torch.cos(az / 2), z, z, -torch.sin(az / 2)], -1))
    w_gt = _to_rotvec(quat)
    R = _exp(w_gt)[0]
    t_gt = -radius * (R @ torch.stack([torch.cos(az), torch.sin(az), z], -1)[..., None])[..., 0]
    intr = torch.stack([500 + 500 * rand(C), 0.01 * randn(C), 0.01 * randn(C)], -1)
    # points: a cloud inside the ring, or a band along a wide ring
    if radius > 8:
        a, r = 2 * math.pi * rand(N), radius - 2 - 6 * rand(N)
        X = torch.stack([r * torch.cos(a), r * torch.sin(a), randn(N).clamp(-3, 3)], -1)
    else:
        X = randn(N, 3)
        X = X * (X.norm(dim=-1, keepdim=True).clamp(max=3.0) / X.norm(dim=-1, keepdim=True))
    # views
    if case["views"] == "poisson":
        extra = torch.poisson(torch.full((N,), float(case["mean"]), device=DEV), generator=sizes)
    else:
        extra = torch.empty(N, device=DEV).geometric_(1.0 / (1.0 + case["mean"]), generator=sizes) - 1
    k = torch.minimum(2 + extra.long(), nc[prob_p])
    pt = torch.arange(N, device=DEV).repeat_interleave(k)
    j = torch.arange(pt.numel(), device=DEV) - (k.cumsum(0) - k).repeat_interleave(k)
    if case["visibility"] == "uniform":
        keys = rand(N, int(nc.max())).float()
        keys[torch.arange(keys.shape[1], device=DEV)[None, :] >= nc[prob_p][:, None]] = 2.0
        cam = keys.argsort(1)[pt, j]
    else:
        u = torch.remainder(torch.atan2(X[:, 1], X[:, 0]), 2 * math.pi) / (2 * math.pi) * nc[prob_p]
        start = torch.round(u - (k - 1) / 2).long()
        cam = torch.remainder(start[pt] + j, nc[prob_p][pt])
    prob_o = prob_p[pt]
    cam = cam + cam0[prob_o]
    # observations of one problem in random order
    order = torch.rand(pt.numel(), generator=g, device=DEV).add_(prob_o).argsort() if P > 1 \
        else torch.randperm(pt.numel(), generator=g, device=DEV)
    cam, pt, prob_o = cam[order], pt[order], prob_o[order]
    px = torch.empty(pt.numel(), 2, device=DEV, dtype=torch.float32)
    for a in range(0, pt.numel(), 1 << 22):
        s = slice(a, a + (1 << 22))
        px[s] = _project(R[cam[s]], t_gt[cam[s]], intr[cam[s]], X[pt[s]])[4].float()
    px += 0.5 * torch.randn(px.shape, generator=g, device=DEV)
    # starting values: a few pixels off, as a reconstruction that is refined once more
    u1, u2 = randn(C, 3), randn(C, 3)
    w0 = _to_rotvec(_quat_mul(_to_quat(0.002 * u1 / u1.norm(dim=-1, keepdim=True)), _to_quat(w_gt)))
    centre = -(R.transpose(1, 2) @ t_gt[..., None]) + 0.01 * (u2 / u2.norm(dim=-1, keepdim=True))[..., None]
    t0 = -(_exp(w0)[0] @ centre)[..., 0]
    s = SimpleNamespace(P=P, nc=nc, npt=npt, cam0=cam0, pt0=pt0, prob_c=prob_c, prob_p=prob_p, prob_o=prob_o, cam=cam,
                        pt=pt, px=px, cams=torch.cat([w0, t0, intr], -1), pts=X + 0.05 * randn(N, 3), factors=None)
    if case["factors"]:
        gt = SimpleNamespace(n_cams=C, cams_gt=torch.cat([w_gt, t_gt, intr], -1).cpu().numpy())
        s.factors = synth.make_pose_factors(gt, pairs=case["factors"], seed=seed)
    return s


def _host(t, dtype):
    return t.cpu().numpy().astype(dtype)


def _options(case):
    return dict(max_lm_iters=case["lm"], max_pcg_iters=case["pcg"], pcg_rel_tol=case["tol"],
                loss=case["loss"], loss_scale=case["loss_scale"], rotation_update=case["retract"], solver=case["schur"])


def prepare(case, seed):
    s = _inputs(case, seed)
    ci, pi, px = _host(s.cam, np.uint32), _host(s.pt, np.uint32), _host(s.px, np.float64)
    st = SimpleNamespace(case=case, options=_options(case))
    if case["kind"] == "batch":
        n_obs = torch.bincount(s.prob_o, minlength=s.P).cpu().numpy()
        cut = np.concatenate([[0], np.cumsum(n_obs)])
        nc, npt, c0, p0 = (t.cpu().numpy() for t in (s.nc, s.npt, s.cam0, s.pt0))
        st.batch = binding.Batch([SimpleNamespace(
            n_cams=int(nc[q]), n_pts=int(npt[q]), cam_idx=ci[cut[q]:cut[q + 1]] - np.uint32(c0[q]),
            pt_idx=pi[cut[q]:cut[q + 1]] - np.uint32(p0[q]), pixels=px[cut[q]:cut[q + 1]]) for q in range(s.P)])
        st.cams, st.pts = _host(s.cams, np.float64), _host(s.pts, np.float64)
        return st
    if case["kind"] == "full":
        st.arrays = (len(s.cams), len(s.pts), ci, pi, px)
        st.cams, st.pts = _host(s.cams, np.float64), _host(s.pts, np.float64)
        return st
    st.problem = binding.Problem(len(s.cams), len(s.pts), ci, pi, px, precision=case["precision"],
                                 pose_factors=s.factors)
    st.cams, st.pts = s.cams, s.pts
    if case["kind"] == "gradient":
        dtype = getattr(torch, case["dtype"])
        st.cams, st.pts = s.cams.to(dtype).requires_grad_(), s.pts.to(dtype).requires_grad_()
    return st


def run(state):
    kind = state.case["kind"]
    if kind == "solve":
        p = state.problem
        p.set_params(state.cams, state.pts)
        r = p.solve(**state.options)
        cams, pts = p.get_params_device()
        return {"initial": r.initial_cost, "final": r.final_cost, "cams": cams, "pts": pts}
    if kind == "full":
        p = binding.Problem(*state.arrays)
        p.set_params(state.cams, state.pts)
        r = p.solve(**state.options)
        cams, pts = (t.cpu() for t in p.get_params_device())
        p.close()
        return {"initial": r.initial_cost, "final": r.final_cost, "cams": cams, "pts": pts}
    if kind == "evaluate":
        state.problem.set_params(state.cams, state.pts)
        cost, r, jac = state.problem.evaluate(residuals=True, jacobian=True)
        return {"cost": cost, "residuals": r, "jacobian": jac}
    if kind == "gradient":
        state.cams.grad = state.pts.grad = None
        loss = autograd.reprojection_cost(state.problem, state.cams, state.pts)
        loss.backward()
        return {"loss": loss.item(), "cams": state.cams.grad, "pts": state.pts.grad}
    b = state.batch
    b.set_params(state.cams, state.pts)
    r = b.solve(**state.options)
    cams, pts = b.get_params()   # the batched mode's parameters are float32 values
    return {"final": np.array([x.final_cost for x in r], dtype=np.float32), "cams": cams.astype(np.float32),
            "pts": pts.astype(np.float32)}


# --------------------------------------------------------------------------------- work ---


def work(case):
    C, N = case["n_cams"], case["n_pts"]
    if case["n_problems"] > 1:
        C, N = case["n_problems"] * (5 + C) // 2, case["n_problems"] * N * 13 // 25
    O = int(N * (2 + case["mean"]))
    size = 8 if case["precision"] == "fp64" or case["dtype"] == "float64" else 4
    n = 9 * C + 3 * N
    seen = 16 * O   # indices and pixel of every observation
    if case["kind"] == "evaluate":
        return {"bytes": seen + 8 * n + size * 26 * O, "flops": 200 * O}
    if case["kind"] == "gradient":
        return {"bytes": seen + 2 * size * n, "flops": 300 * O}
    # per LM iteration: residual and Jacobian blocks (about 500 operations per observation),
    # and per PCG iteration J and J^T of every observation and the vectors' updates
    return {"bytes": seen + 8 * n + size * n, "flops": case["lm"] * (500 * O + case["pcg"] * (150 * O + 12 * n))}


# -------------------------------------------------------------------------------- exact ---


def _mul(a, b):   # products of many tiny matrices
    return sum(a[:, :, k, None] * b[:, None, k, :] for k in range(b.shape[1]))


def _residual_jacobian(s, cams, pts, retract, jacobian=True):
    """r [O, 2] and its Jacobian [O, 2, 12] in 64 bits."""
    R, JL = _exp(cams[:, :3])
    if retract:
        JL = torch.eye(3, device=DEV, dtype=F64).expand_as(JL)
    c, X = s.cam, pts[s.pt]
    P, p, n2, sc, px = _project(R[c], cams[c, 3:6], cams[c, 6:], X)
    r = px - s.px.double()
    if not jacobian:
        return r, None
    f, k1, k2 = cams[c, 6], cams[c, 7], cams[c, 8]
    M = (f * sc)[:, None, None] * torch.eye(2, device=DEV, dtype=F64) \
        + (2 * f * (k1 + 2 * k2 * n2))[:, None, None] * p[:, :, None] * p[:, None, :]
    D = torch.zeros(len(p), 2, 3, device=DEV, dtype=F64)
    D[:, 0, 0] = D[:, 1, 1] = 1
    D[:, :, 2] = p
    A = _mul(M, D) * (-1 / P[:, 2])[:, None, None]
    J = torch.empty(len(p), 2, 12, device=DEV, dtype=F64)
    J[:, :, :3] = _mul(-_mul(A, _skew(P - cams[c, 3:6])), JL[c])
    J[:, :, 3:6] = A
    J[:, :, 6] = sc[:, None] * p
    J[:, :, 7] = (f * n2)[:, None] * p
    J[:, :, 8] = (f * n2 * n2)[:, None] * p
    J[:, :, 9:] = _mul(A, R[c])
    return r, J


def _factor_rows(s, cams, retract, jacobian=True):
    """Rows [F, 6] of the pose factors and their Jacobian [F, 6, 18] over both cameras."""
    a, b = (torch.from_numpy(np.asarray(x).astype(np.int64)).to(DEV) for x in s.factors[:2])
    meas, sq = (torch.from_numpy(np.asarray(x)).to(DEV) for x in s.factors[2:])
    Rm, tm = _exp(meas[:, :3])[0], meas[:, 3:]

    def rows(x):   # x [F, 18]: offsets of both cameras
        ca, cb = cams[a] + (0 if retract else x[:, :9]), cams[b] + (0 if retract else x[:, 9:])
        Ra, Rb, ta, tb = _exp(ca[:, :3])[0], _exp(cb[:, :3])[0], ca[:, 3:6], cb[:, 3:6]
        if retract:
            Ra, Rb = _exp(x[:, :3])[0] @ Ra, _exp(x[:, 9:12])[0] @ Rb
            ta, tb = ta + x[:, 3:6], tb + x[:, 12:15]
        Rba = Rb @ Ra.transpose(1, 2)
        E = Rm.transpose(1, 2) @ Rba
        v = torch.stack([E[:, 2, 1] - E[:, 1, 2], E[:, 0, 2] - E[:, 2, 0], E[:, 1, 0] - E[:, 0, 1]], -1) / 2
        n = v.norm(dim=-1, keepdim=True)
        tr = (E.diagonal(dim1=1, dim2=2).sum(-1, keepdim=True) - 1) / 2
        return sq * torch.cat([torch.atan2(n, tr) / n * v, tb - (Rba @ ta[..., None])[..., 0] - tm], -1)

    x = torch.zeros(len(a), 18, device=DEV, dtype=F64, requires_grad=jacobian)
    with torch.set_grad_enabled(jacobian):
        r = rows(x)
        J = torch.stack([torch.autograd.grad(r[:, i].sum(), x, retain_graph=True)[0] for i in range(6)], 1) \
            if jacobian else None
    return r.detach(), J, a, b


def _exact_solve(case, s):
    """LM + block-Jacobi PCG of every problem at once in 64 bits; returns cost at the start,
    cost at the end (per problem) and the parameters."""
    P, C, N = s.P, len(s.cams), len(s.pts)
    retract, loss, d2, schur = case["retract"], case["loss"], case["loss_scale"] ** 2, case["schur"]
    cams, pts = s.cams.clone(), s.pts.clone()

    def inv3(H):   # symmetric 3 x 3 blocks, by the adjugate
        a, b, c, d, e, f = H[:, 0, 0], H[:, 0, 1], H[:, 0, 2], H[:, 1, 1], H[:, 1, 2], H[:, 2, 2]
        A, B, C_ = d * f - e * e, c * e - b * f, b * e - c * d
        adj = torch.stack([A, B, C_, B, a * f - c * c, b * c - a * e, C_, b * c - a * e, a * d - b * b], -1)
        return (adj / (a * A + b * B + c * C_)[:, None]).reshape(-1, 3, 3)

    def seg(x, prob):   # sum per problem
        return x.sum().reshape(1) if P == 1 else torch.zeros(P, device=DEV, dtype=F64).index_add_(0, prob, x)

    def dot(u, v):
        return seg((u[0] * v[0]).sum(-1), s.prob_c) + seg((u[1] * v[1]).sum(-1), s.prob_p)

    def axpy(a, u, v):   # a u + v, a per problem
        return a[s.prob_c, None] * u[0] + v[0], a[s.prob_p, None] * u[1] + v[1]

    def cost(cams, pts):
        s2 = (_residual_jacobian(s, cams, pts, retract, False)[0] ** 2).sum(-1)
        if loss == 1:
            s2 = torch.where(s2 <= d2, s2, 2 * torch.sqrt(d2 * s2) - d2)
        elif loss == 2:
            s2 = d2 * torch.log1p(s2 / d2)
        F = 0.5 * seg(s2, s.prob_o)
        if s.factors is not None:
            F = F + 0.5 * (_factor_rows(s, cams, retract, False)[0] ** 2).sum()
        return F

    def linearise(cams, pts):
        r, J = _residual_jacobian(s, cams, pts, retract)
        s2 = (r * r).sum(-1)
        if loss:
            w = torch.where(s2 <= d2, torch.ones_like(s2), torch.sqrt(d2 / s2)) if loss == 1 else 1 / (1 + s2 / d2)
            r, J = r * w.sqrt()[:, None], J * w.sqrt()[:, None, None]
        L = SimpleNamespace(J=J, f=None)
        if s.factors is not None:
            rf, Jf, a, b = _factor_rows(s, cams, retract)
            L.f = (Jf, a, b)
        L.g = adjoint(L, r, rf if L.f else None)
        L.Hc = torch.zeros(C, 9, 9, device=DEV, dtype=F64)
        L.Hp = torch.zeros(N, 3, 3, device=DEV, dtype=F64)
        for i in range(0, len(r), 1 << 22):
            k = slice(i, i + (1 << 22))
            for row in (0, 1):
                jc, jp = J[k, row, :9], J[k, row, 9:]
                L.Hc.index_add_(0, s.cam[k], jc[:, :, None] * jc[:, None, :])
                L.Hp.index_add_(0, s.pt[k], jp[:, :, None] * jp[:, None, :])
        if L.f:
            L.Hc.index_add_(0, a, Jf[:, :, :9].transpose(1, 2) @ Jf[:, :, :9])
            L.Hc.index_add_(0, b, Jf[:, :, 9:].transpose(1, 2) @ Jf[:, :, 9:])
        L.D = tuple(H.diagonal(dim1=1, dim2=2).clamp(1e-6, 1e32) for H in (L.Hc, L.Hp))
        return L

    def forward(L, v):
        t = (L.J * torch.cat([v[0][s.cam], v[1][s.pt]], -1)[:, None, :]).sum(-1)
        tf = (L.f[0] @ torch.cat([v[0][L.f[1]], v[0][L.f[2]]], -1)[..., None])[..., 0] if L.f else None
        return t, tf

    def adjoint(L, t, tf):
        u = L.J[:, 0] * t[:, :1] + L.J[:, 1] * t[:, 1:]
        qc = torch.zeros(C, 9, device=DEV, dtype=F64).index_add_(0, s.cam, u[:, :9])
        qp = torch.zeros(N, 3, device=DEV, dtype=F64).index_add_(0, s.pt, u[:, 9:])
        if L.f:
            uf = (L.f[0].transpose(1, 2) @ tf[..., None])[..., 0]
            qc.index_add_(0, L.f[1], uf[:, :9]).index_add_(0, L.f[2], uf[:, 9:])
        return qc, qp

    def sq(L, v):   # |J v|^2
        t, tf = forward(L, v)
        return seg((t * t).sum(-1), s.prob_o) + ((tf * tf).sum() if L.f else 0)

    def step(L, mu):
        muc, mup = mu[s.prob_c, None], mu[s.prob_p, None]
        Mc = torch.linalg.inv(L.Hc + torch.diag_embed(muc * L.D[0]))
        Mp = inv3(L.Hp + torch.diag_embed(mup * L.D[1]))

        def apply(v):
            q = adjoint(L, *forward(L, v))
            return q[0] + muc * L.D[0] * v[0], q[1] + mup * L.D[1] * v[1]

        def solve_p(y):
            return (Mp * y[:, None, :]).sum(-1)

        zero = torch.zeros_like(L.g[0]), torch.zeros_like(L.g[1])
        b = -L.g[0], -L.g[1]
        if schur:   # S = Hcc - Hcp Hpp^-1 Hpc on the cameras
            def op(v):
                q = apply((v[0], zero[1]))
                return q[0] - apply((zero[0], solve_p(q[1])))[0], zero[1]

            r = (b[0] - apply((zero[0], solve_p(b[1])))[0], zero[1])
        else:
            op, r = apply, b

        def prec(r):
            return (Mc * r[0][:, None, :]).sum(-1), zero[1] if schur else solve_p(r[1])

        h, z = zero, prec(r)
        p, rz, rr0 = z, dot(r, z), dot(r, r)
        on = rr0 > 0
        for _ in range(case["pcg"]):
            q = op(p)
            alpha = torch.where(on, rz / dot(p, q), torch.zeros_like(rz))
            h, r = axpy(alpha, p, h), axpy(-alpha, q, r)
            z = prec(r)
            new = dot(r, z)
            on = on & (dot(r, r) > case["tol"] ** 2 * rr0)
            if not bool(on.any()):
                break
            p, rz = axpy(torch.where(on, new / rz, torch.zeros_like(rz)), p, z), torch.where(on, new, rz)
        if schur:
            h = h[0], solve_p(b[1] - apply((h[0], zero[1]))[1])
        return h

    F = F0 = cost(cams, pts)
    mu, nu = torch.full((P,), 0.01, device=DEV, dtype=F64), torch.full((P,), 2.0, device=DEV, dtype=F64)
    L = linearise(cams, pts)
    for it in range(case["lm"]):
        h = step(L, mu)
        new = cams + h[0]
        if retract:
            new = torch.cat([_to_rotvec(_quat_mul(_to_quat(h[0][:, :3]), _to_quat(cams[:, :3]))), new[:, 3:]], -1)
        Fn = cost(new, pts + h[1])
        gain = -dot(L.g, h) - 0.5 * sq(L, h)
        rho = (F - Fn) / gain
        ok = (gain > 0) & (rho > 0)
        mu = torch.where(ok, mu * torch.clamp(1 - (2 * rho - 1) ** 3, min=1 / 3), mu * nu)
        nu = torch.where(ok, torch.full_like(nu, 2.0), 2 * nu)
        F = torch.where(ok, Fn, F)
        cams = torch.where(ok[s.prob_c, None], new, cams)
        pts = torch.where(ok[s.prob_p, None], pts + h[1], pts)
        if it + 1 < case["lm"]:
            L = None
            L = linearise(cams, pts)
    return F0, F, cams, pts


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "evaluate":
        r, J = _residual_jacobian(s, s.cams, s.pts, 0)
        return {"cost": float(0.5 * (r * r).sum()), "residuals": r, "jacobian": J}
    if kind == "gradient":
        dtype = getattr(torch, case["dtype"])
        r, J = _residual_jacobian(s, s.cams.to(dtype).double(), s.pts.to(dtype).double(), 0)
        u = J[:, 0] * r[:, :1] + J[:, 1] * r[:, 1:]
        return {"loss": float(0.5 * (r * r).sum()), "cams": torch.zeros_like(s.cams).index_add_(0, s.cam, u[:, :9]),
                "pts": torch.zeros_like(s.pts).index_add_(0, s.pt, u[:, 9:])}
    F0, F, cams, pts = _exact_solve(case, s)
    if kind == "batch":
        return {"final": F, "cams": cams, "pts": pts}
    return {"initial": float(F0), "final": float(F), "cams": cams, "pts": pts}
