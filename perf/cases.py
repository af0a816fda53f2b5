"""The work this framework is used for, as measurable cases.

A plan is a water phantom with one to three pencil-beam fields, a target and
(up to) three organs at risk.  Its influence pair (D, L) is made on the GPU as
a user's GPU dose engine would hand it over: a voxel row holds the spots whose
lateral window covers the voxel and whose range reaches it, columns ascending.
The geometries are those of the repository's own plans: the tiny one (32^3
voxels at 3 mm, 2250 spots), the lesions of the batch workload, the clinical
one (200 x 200 x 150 voxels at 2 mm, 30000 spots) and its half-resolution form.

Operations (`op`):
  step      one simultaneous feasibility step from x (Fig. 2)
  solve     begin, `iters` superiorized iterations, end: w, dose, LETd (Fig. 3)
  products  D w, L w and D^T a + L^T b, as an outer optimiser calls them
  gradient  objective and gradient with dose and cDL terms (Eq. 2)
  sweep     one block-iterative sweep over `blocks` voxel blocks
  volume    DVH, LVH and cDLVH of every structure, with values at volume
  request   load a plan that lies on the device, set it up, solve it
  csc       transposed product of caller-owned CSC arrays, no allocation
  batch     several uneven plans solved together from one graph
"""
import ctypes
import math

import numpy as np
import torch

from paper_2509_20012_gb300 import fredopt

DEV = "cuda:0"
C_CDL = 0.04
REACH = 15.0  # mm: half width of a pencil beam's lateral window
SIGMA = 4.0
ALPHA, RELAX = 0.99, 1.0
VALUE_BYTES = {"fp32": 4, "bf16": 2, "fp16": 2}


def _tiny(**kw):
    return dict(nx=32, ny=32, nz=32, h=3.0, fields=1, spots=15, pitch=4.0, layers=10, **kw)


def _half(**kw):
    return dict(nx=100, ny=100, nz=75, h=4.0, fields=3, spots=20, pitch=4.0, layers=25, **kw)


def _clinical(**kw):
    return dict(nx=200, ny=200, nz=150, h=2.0, fields=3, spots=20, pitch=4.0, layers=25, **kw)


def listed():
    return [
        # one feasibility step of a small plan: launches and latency count
        _tiny(name="tiny_step_fp32", op="step", fmt="fp32", rows="all"),
        # a whole small plan, 100 iterations
        _tiny(name="tiny_solve_fp32", op="solve", fmt="fp32", rows="all", iters=100),
        # the gradient of the literal Eq. 2 (target dose and OAR cDL terms) on a lesion
        # plan with odd sizes
        dict(name="lesion_gradient_fp16", op="gradient", nx=73, ny=73, nz=61, h=4.1, fields=2, spots=13, pitch=6.0,
             layers=17, fmt="fp16", rows="all"),
        # single products for an optimiser of the caller's own
        _half(name="half_products_bf16", op="products", fmt="bf16", rows="all"),
        # the same transposed product on arrays that the caller owns
        _half(name="half_csc_fp32", op="csc", fmt="fp32", rows="all"),
        # six lesions of uneven size re-optimised together
        dict(name="batch6_bf16", op="batch", nx=75, ny=75, nz=62, h=4.0, fields=1, spots=8, pitch=6.0, layers=10,
             plans=6, fmt="bf16", rows="all", iters=20),
        # the clinical plan, every voxel row streamed every pass, FP32 and 16-bit
        _clinical(name="clinical_solve_fp32", op="solve", fmt="fp32", rows="all", iters=10),
        _clinical(name="clinical_solve_bf16", op="solve", fmt="bf16", rows="all", iters=10),
        # the same over the structure rows only
        _clinical(name="clinical_roi_solve_fp32", op="solve", fmt="fp32", rows="roi", iters=50),
        # one sweep of Fig. 2 over 64 voxel blocks
        _clinical(name="clinical_roi_sweep_fp32", op="sweep", fmt="fp32", rows="roi", blocks=64),
        # plan evaluation: volume histograms and values at volume
        _clinical(name="clinical_volume_fp16", op="volume", fmt="fp16", rows="all"),
        # a served request: the plan is loaded and solved once
        _clinical(name="clinical_request_fp32", op="request", fmt="fp32", rows="all", iters=20),
    ]


def draw(rng):
    """A case of any operation; nonzeros from 1e6 to 4e8 over their logarithm, voxel
    counts, spot grids and layers odd or even as they fall."""
    op = rng.choice(["step", "solve", "solve", "products", "gradient", "sweep", "volume", "request", "csc", "batch"])
    while True:
        h = math.exp(rng.uniform(math.log(2.0), math.log(6.0)))
        target = math.exp(rng.uniform(math.log(1e6), math.log(4e8)))
        extent = rng.uniform(140.0, 400.0)
        case = dict(op=op, nx=int(extent / h), ny=int(rng.uniform(0.8, 1.0) * extent / h),
                    nz=int(rng.uniform(0.7, 1.0) * extent / h), h=round(h, 3), fields=rng.choice([1, 2, 3]),
                    spots=rng.randint(7, 20), pitch=rng.choice([4.0, 5.0, 6.0]), layers=rng.randint(6, 25),
                    fmt=rng.choice(["fp32", "bf16", "fp16"]), rows=rng.choice(["all", "all", "roi"]))
        if op == "csc":
            case.update(fmt="fp32", rows="all")
        if op == "batch":
            case.update(plans=rng.randint(2, 6), fields=1, spots=min(case["spots"], 12), iters=rng.randint(5, 20))
        if op in ("solve", "request"):
            case["iters"] = rng.randint(3, 50) if target < 5e7 else rng.randint(3, 10)
        if op == "sweep":
            case["blocks"] = int(round(math.exp(rng.uniform(math.log(2.0), math.log(64.0)))))
        if target / 3.0 < _nnz(case) < 3.0 * target and _nnz(case) < 4e8:
            return case


# ------------------------------------------------------------------ geometry

AXES = [(2, False, 0, 1), (0, False, 1, 2), (0, True, 1, 2)]  # depth axis, from the far side, lateral axes


def _windows(case):
    """Per field: first spot and spot count per voxel of the two lateral axes, first
    layer and layer count per voxel of the depth axis (layers ascend in range, so the
    layers that reach a depth are the last ones), and the layers' ranges."""
    n = (case["nx"], case["ny"], case["nz"])
    h, s, pitch, layers = case["h"], case["spots"], case["pitch"], case["layers"]
    out = []
    for ax, far, u, v in AXES[:case["fields"]]:
        lat = []
        for a in (u, v):
            x = (np.arange(n[a]) + 0.5) * h - 0.5 * n[a] * h
            pos = (np.arange(s) - 0.5 * (s - 1)) * pitch
            lo = np.searchsorted(pos, x - REACH, side="left")
            lat.append((lo, np.searchsorted(pos, x + REACH, side="right") - lo))
        depth = (np.arange(n[ax]) + 0.5) * h
        if far:
            depth = depth[::-1].copy()
        ranges = 0.5 * n[ax] * h + (np.arange(layers) - 0.5 * (layers - 1)) * min(3.0, 0.6 * n[ax] * h / layers)
        first = np.searchsorted(ranges, depth - 6.0, side="left")
        out.append(dict(ax=ax, u=u, v=v, lat_u=lat[0], lat_v=lat[1], dep=(first, layers - first), depth=depth,
                        ranges=ranges))
    return out


def _sub_cases(case):
    """The plans of a batch: the same phantom, spot grids and layers growing."""
    if case["op"] != "batch":
        return [case]
    return [dict(case, spots=case["spots"] + 2 * i, layers=case["layers"] + 2 * i) for i in range(case["plans"])]


def _nnz(case):
    return sum(int(w["lat_u"][1].sum()) * int(w["lat_v"][1].sum()) * int(w["dep"][1].sum())
               for c in _sub_cases(case) for w in _windows(c))


def _row_counts(case):
    """Nonzeros of every voxel row (voxel = (z * ny + y) * nx + x)."""
    total = 0
    for w in _windows(case):
        f = [None, None, None]
        f[w["u"]], f[w["v"]], f[w["ax"]] = w["lat_u"][1], w["lat_v"][1], w["dep"][1]
        total = total + f[2][:, None, None] * f[1][None, :, None] * f[0][None, None, :]
    return total.reshape(-1)


def _mask(case):
    """Target ellipsoid (bit 0), a cylinder behind it (bit 1), a slab beside it (bit 2),
    two spheres (bit 3): sized by the spot grid, positions in mm from the centre."""
    n = (case["nx"], case["ny"], case["nz"])
    h = case["h"]
    x, y, z = ((np.arange(k) + 0.5) * h - 0.5 * k * h for k in n)
    Z, Y, X = np.meshgrid(z, y, x, indexing="ij", sparse=True)
    a = 0.5 * (case["spots"] - 1) * case["pitch"] * 0.92
    c = min(0.83 * a, 0.25 * n[2] * h)
    m = ((X / a) ** 2 + (Y / a) ** 2 + (Z / c) ** 2 <= 1.0).astype(np.int32)
    m |= ((X ** 2 + (Z - (c + 0.4 * a)) ** 2 <= (0.34 * a) ** 2) & (np.abs(Y) <= 0.71 * a)).astype(np.int32) << 1
    m |= ((np.abs(Y - 1.17 * a) <= max(2.0, 0.5 * h)) & (np.abs(X) <= 0.57 * a) & (np.abs(Z) <= 0.34 * a)).astype(np.int32) << 2
    for sx in (-1.0, 1.0):
        m |= ((X - sx * 1.14 * a) ** 2 + (Y - 0.57 * a) ** 2 + (Z + 1.29 * c) ** 2 <= (0.34 * a) ** 2).astype(np.int32) << 3
    return m.reshape(-1)


def _constraints():
    con = [dict(struct_bit=0, kind="DOSE_MIN", bound=1.9, priority=1.0),
           dict(struct_bit=0, kind="DOSE_MAX", bound=2.14, priority=1.0)]
    for bit, dose, let in ((1, 1.2, 2.5), (2, 1.0, 2.5), (3, 0.5, 3.0)):
        con.append(dict(struct_bit=bit, kind="DOSE_MAX", bound=dose, priority=1.0))
        con.append(dict(struct_bit=bit, kind="LETD_MAX", bound=let, priority=1.0))
    return con


def _objective(case):
    terms = [dict(struct_bit=b, quantity="CDL", target=0.0, weight=1.0) for b in (1, 2, 3)]
    if case["op"] == "gradient":
        terms.append(dict(struct_bit=0, quantity="DOSE", target=2.0, weight=1.0))
    return terms


def _csr(case, seed):
    """row_ptr int64, col int32, D and L float32 on the GPU: Gaussian lateral profile,
    a depth dose that rises to the range, LET that rises with it, 1% noise; D scaled so
    that unit weights give 2 Gy at the centre."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    n = (case["nx"], case["ny"], case["nz"])
    h, s, pitch, layers = case["h"], case["spots"], case["pitch"], case["layers"]
    V = n[0] * n[1] * n[2]
    counts = torch.from_numpy(_row_counts(case)).to(DEV)
    rp = torch.zeros(V + 1, dtype=torch.int64, device=DEV)
    rp[1:] = torch.cumsum(counts, 0)
    nnz = int(rp[-1])
    col = torch.empty(nnz, dtype=torch.int32, device=DEV)
    D = torch.empty(nnz, dtype=torch.float32, device=DEV)
    L = torch.empty(nnz, dtype=torch.float32, device=DEV)
    vox = torch.arange(V, device=DEV)
    idx = (vox % n[0], (vox // n[0]) % n[1], vox // (n[0] * n[1]))
    base = rp[:-1].clone()
    for k, w in enumerate(_windows(case)):
        t = lambda a, dt=torch.int64: torch.from_numpy(np.ascontiguousarray(a)).to(DEV, dt)
        u0, cu = (t(a)[idx[w["u"]]] for a in w["lat_u"])
        v0, cv = (t(a)[idx[w["v"]]] for a in w["lat_v"])
        l0, cl = (t(a)[idx[w["ax"]]] for a in w["dep"])
        cnt = cu * cv * cl
        live = torch.nonzero(cnt).flatten()
        if live.numel() == 0:
            continue
        c = cnt[live]
        row = torch.repeat_interleave(live, c)
        ofs = torch.arange(row.numel(), device=DEV) - torch.repeat_interleave(torch.cumsum(c, 0) - c, c)
        dst = base[row] + ofs
        a, b = cu[row], cv[row]
        iu = u0[row] + ofs % a
        iv = v0[row] + (ofs // a) % b
        il = l0[row] + ofs // (a * b)
        del ofs, a, b
        du = (idx[w["u"]][row] + 0.5 - 0.5 * n[w["u"]]).float() * h - (iu - 0.5 * (s - 1)).float() * pitch
        dv = (idx[w["v"]][row] + 0.5 - 0.5 * n[w["v"]]).float() * h - (iv - 0.5 * (s - 1)).float() * pitch
        res = t(w["ranges"], torch.float32)[il] - t(w["depth"], torch.float32)[idx[w["ax"]][row]]
        col[dst] = (((k * layers + il) * s + iv) * s + iu).int()
        d = torch.exp(-(du * du + dv * dv) / (2.0 * SIGMA * SIGMA))
        del du, dv, iu, iv, il, row
        d *= 0.25 + torch.exp(-((res - 1.0) / 6.0) ** 2)
        d *= 1.0 + 0.01 * (2.0 * torch.rand(d.shape, generator=gen, device=DEV) - 1.0)
        let = 1.0 + 9.0 * torch.exp(-(res.clamp(min=0.0)) / 12.0)
        let *= 1.0 + 0.01 * (2.0 * torch.rand(d.shape, generator=gen, device=DEV) - 1.0)
        D[dst] = d
        L[dst] = let
        del d, let, res, dst
        base += cnt
    mid = ((n[2] // 2) * n[1] + n[1] // 2) * n[0] + n[0] // 2
    D *= (2.0 / D[rp[mid]:rp[mid + 1]].double().sum()).float()
    L *= D
    return rp, col, D, L


def _spots(case):
    return case["fields"] * case["layers"] * case["spots"] ** 2


def _weights(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 1)
    return 0.5 + torch.rand(_spots(case), generator=g, device=DEV)


def _coefs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 2)
    V = case["nx"] * case["ny"] * case["nz"]
    return torch.randn(V, generator=g, device=DEV), torch.randn(V, generator=g, device=DEV) * 0.1


def _to_csc(rp, col, D, L, n):
    """Column pointers, rows and values of the CSC copy."""
    order = torch.sort(col, stable=True).indices
    rows = torch.repeat_interleave(torch.arange(rp.numel() - 1, device=DEV, dtype=torch.int32), rp.diff())
    cp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    cp[1:] = torch.cumsum(torch.bincount(col, minlength=n), 0)
    return cp, rows[order], D[order], L[order]


VOLUME_BITS = (0, 1, 2, 3)


def _volume_requests():
    req = []
    for b in VOLUME_BITS:
        req.append(dict(quantity="DOSE", struct_bit=b, edges=np.linspace(0.0, 4.0, 401), fracs=[0.98, 0.5, 0.02]))
        req.append(dict(quantity="LETD", struct_bit=b, edges=np.linspace(0.0, 12.0, 401)))
        req.append(dict(quantity="CDL", struct_bit=b, edges=np.linspace(0.0, 1.2, 401), fracs=[0.3]))
    return req


# ------------------------------------------------------------------ the cases

def prepare(case, seed):
    st = dict(case=case)
    handles, weights = [], []
    for i, c in enumerate(_sub_cases(case)):
        rp, col, D, L = _csr(c, seed + 1000 * i)
        weights.append(_weights(c, seed + 1000 * i))
        if case["op"] == "csc":
            st["csc"] = _to_csc(rp, col, D, L, _spots(c))
            break
        mask = torch.from_numpy(_mask(c)).to(DEV)
        h = fredopt.Handle(0)
        handles.append(h)
        if case["op"] == "request":
            st["plan"] = (rp, col, D, L, mask)
            break
        h.load_influence(rp, col, D, L, mask, _spots(c), fmt=c["fmt"], rows=c["rows"], shared=case["op"] == "batch")
        h.set_constraints(_constraints())
        h.set_objective(_objective(c))
        del rp, col, D, L, mask
    st["handles"], st["w"] = handles, weights
    if case["op"] in ("products", "csc"):
        st["a"] = _coefs(case, seed)
    if case["op"] == "csc":
        st["u"] = torch.empty(_spots(case), device=DEV)
    if case["op"] == "batch":
        st["w"] = [w.cpu().numpy() for w in weights]
    if case["op"] == "volume":
        st["requests"] = _volume_requests()
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return st


def run(state):
    case = state["case"]
    op = case["op"]
    w = state["w"][0]
    if op == "csc":
        cp, row, D, L = state["csc"]
        a, b = state["a"]
        u = state["u"]
        p = lambda t: ctypes.c_void_p(t.data_ptr())
        rc = fredopt.load_library().fredopt_backward_noalloc(
            a.numel(), u.numel(), row.numel(), p(cp), p(row), p(D), p(L), p(a), p(b), p(u),
            ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if rc != 0:
            raise RuntimeError(f"fredopt_backward_noalloc: {rc}")
        return u
    if op == "batch":
        out = fredopt.superiorize_batch(state["handles"], state["w"], case["iters"], ALPHA, RELAX)
        return [list(o[:3]) for o in out]
    h = state["handles"][0]
    if op == "step":
        return h.feasibility_step(w)
    if op == "products":
        a, b = state["a"]
        return list(h.forward(w)) + [h.backward(a, b)]
    if op == "gradient":
        return list(h.objective(w))
    if op == "sweep":
        return h.sweep_step(w, case["blocks"])
    if op == "volume":
        return h.volume_stats(state["requests"], w)
    if op == "request":
        rp, col, D, L, mask = state["plan"]
        h.load_influence(rp, col, D, L, mask, _spots(case), fmt=case["fmt"], rows=case["rows"])
        h.set_constraints(_constraints())
        h.set_objective(_objective(case))
    return list(h.superiorize(w, case["iters"], ALPHA, RELAX)[:3])


def work(case):
    """Bytes and operations of one pass.  Matrices count at 2-byte indices and their
    stored value width; a matrix is read once per product that the method needs (the
    iterations of a solve cannot share reads: each depends on the one before).  In ROWS
    ALL every voxel row is streamed every pass, by the option's definition; in ROI only
    the structure rows.  The gradient of cDL terms reads L alone."""
    by = fl = 0
    for c in _sub_cases(case):
        op = case["op"]
        counts = _row_counts(c)
        nnz = int(counts.sum())
        roi = int(counts[_mask(c) != 0].sum())
        hot = roi if c["rows"] == "roi" else nnz
        V, n, vb = counts.size, _spots(c), VALUE_BYTES[c["fmt"]]
        both, one = 2 + 2 * vb, 2 + vb
        outputs = 4 * n + 8 * V
        if op == "csc":
            by += nnz * 12 + 8 * (n + 1) + 8 * V + 4 * n
            fl += 4 * nnz
        elif op == "step":
            by += 2 * hot * both + 8 * n
            fl += 8 * hot
        elif op == "products":
            by += (nnz + hot) * both + 16 * V + 8 * n
            fl += 4 * (nnz + hot)
        elif op == "gradient":
            by += 2 * hot * both + 8 * n
            fl += 8 * hot
        elif op == "sweep":
            by += 2 * roi * both + 8 * n
            fl += 8 * roi
        elif op == "volume":
            by += nnz * both + 16 * int((_mask(c) != 0).sum()) + 4 * V
            fl += 4 * nnz
        else:
            it = case["iters"]
            by += it * hot * (3 * both + one) + nnz * both + outputs
            fl += it * hot * 14 + 4 * nnz
            if op == "request":  # the plan is read once and stored in both orders
                by += nnz * 12 + 8 * V + (nnz + hot) * both
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ plain 64-bit values

class _Plain:
    """The method in float64 on plain CSR arrays of the rows that `keep` selects."""

    CHUNK = 1 << 26

    def __init__(self, rp, col, D, L, n, rows=None):
        self.n = n
        if rows is None:
            self.cnt = rp.diff()
            self.col, self.D, self.L = col, D, L
        else:
            self.cnt = rp.diff()[rows]
            start = torch.repeat_interleave(rp[:-1][rows] - (torch.cumsum(self.cnt, 0) - self.cnt), self.cnt)
            at = start + torch.arange(start.numel(), device=DEV)
            self.col, self.D, self.L = col[at], D[at], L[at]
        self.row = torch.repeat_interleave(torch.arange(self.cnt.numel(), device=DEV, dtype=torch.int32), self.cnt)

    def _pieces(self):
        for a in range(0, self.col.numel(), self.CHUNK):
            yield slice(a, a + self.CHUNK)

    def forward(self, w):
        d = torch.zeros(self.cnt.numel(), dtype=torch.float64, device=DEV)
        l = torch.zeros_like(d)
        for s in self._pieces():
            x, r = w[self.col[s].long()], self.row[s].long()
            d.index_add_(0, r, self.D[s].double() * x)
            l.index_add_(0, r, self.L[s].double() * x)
        return d, l

    def backward(self, a, b):
        u = torch.zeros(self.n, dtype=torch.float64, device=DEV)
        for s in self._pieces():
            r = self.row[s].long()
            u.index_add_(0, self.col[s].long(), self.D[s].double() * a[r] + self.L[s].double() * b[r])
        return u

    def moments(self):
        out = [torch.zeros(self.cnt.numel(), dtype=torch.float64, device=DEV) for _ in range(3)]
        for s in self._pieces():
            r, d, l = self.row[s].long(), self.D[s].double(), self.L[s].double()
            for o, v in zip(out, (d * d, l * l, d * l)):
                o.index_add_(0, r, v)
        return out


def _stored(case, rp, v):
    """The values as 16-bit storage keeps them: rounded after a power-of-two row scale."""
    if case["fmt"] == "fp32":
        return v
    if case["fmt"] == "bf16":
        return v.bfloat16().float()
    cnt = rp.diff()
    live = torch.nonzero(cnt).flatten()
    top = torch.segment_reduce(v, "max", lengths=cnt[live]) if live.numel() else v[:0]
    scale = torch.ldexp(torch.ones_like(top), torch.frexp(top).exponent - 14)
    s = torch.repeat_interleave(scale, cnt[live])
    return (v / s).half().float() * s


def _half_space(con, mask, m, d, l):
    """Per row: projection coefficients of D and L, priorities of the violated and of
    the reachable constraint rows."""
    dd, ll, dl = m
    gd, gl = torch.zeros_like(d), torch.zeros_like(d)
    viol, reach = torch.zeros_like(d), torch.zeros_like(d)
    for c in con:
        b = c["bound"]
        if c["kind"].startswith("DOSE"):
            v, norm, cd, cl, lim = d, dd, 1.0, 0.0, b
        else:  # LETD: (L - bound D) w <= 0
            v, norm, cd, cl, lim = l - b * d, ll - 2.0 * b * dl + b * b * dd, -b, 1.0, 0.0
        on = ((mask >> c["struct_bit"]) & 1).bool() & (norm > 0)
        bad = on & ((v > lim) if c["kind"].endswith("MAX") else (v < lim))
        t = torch.where(bad, c["priority"] * (lim - v) / norm, torch.zeros_like(v))
        gd += cd * t
        gl += cl * t
        viol += c["priority"] * bad
        reach += c["priority"] * on
    return gd, gl, viol, reach


def _residual(terms, mask, d, l):
    f, rd, rl = 0.0, torch.zeros_like(d), torch.zeros_like(d)
    for t in terms:
        on = ((mask >> t["struct_bit"]) & 1).double()
        if t["quantity"] == "DOSE":
            q = on * (d - t["target"])
            rd += 2.0 * t["weight"] * q
        else:
            q = on * (C_CDL * l - t["target"])
            rl += 2.0 * t["weight"] * C_CDL * q
        f += float(t["weight"] * (q * q).sum())
    return f, rd, rl


def _letd(d, l):
    return torch.where(d > 0, l / torch.where(d > 0, d, torch.ones_like(d)), torch.zeros_like(d))


def _solve64(case, seed):
    rp, col, D, L = _csr(case, seed)
    D, L = _stored(case, rp, D), _stored(case, rp, L)
    mask = torch.from_numpy(_mask(case)).to(DEV)
    rows = torch.nonzero(mask).flatten()
    P = _Plain(rp, col, D, L, _spots(case), rows)
    mask = mask[rows]
    con, terms, m = _constraints(), _objective(case), P.moments()
    w = _weights(case, seed).double()
    beta0, s = 0.1 * float(w.norm()), 0
    for _ in range(case["iters"]):
        d, l = P.forward(w)
        _, rd, rl = _residual(terms, mask, d, l)
        g = P.backward(rd, rl)
        gn = float(g.norm())
        if gn > 0:
            gd, gl = P.forward(g / -gn)
            B = float(0.5 * (rd * gd + rl * gl).sum())
            Q = sum(float(t["weight"] * ((((mask >> t["struct_bit"]) & 1) *
                                          (gd if t["quantity"] == "DOSE" else C_CDL * gl)) ** 2).sum()) for t in terms)
            for _ in range(50):
                beta = beta0 * ALPHA ** s
                s += 1
                if beta * (2.0 * B + beta * Q) <= 0.0:
                    w, d, l = w - beta / gn * g, d + beta * gd, l + beta * gl
                    break
        gd, gl, _, reach = _half_space(con, mask, m, d, l)
        W = float(reach.sum())
        w = (w + (RELAX / W if W > 0 else 0.0) * P.backward(gd, gl)).clamp(min=0.0)
    del P
    d, l = _Plain(rp, col, D, L, _spots(case)).forward(w)
    return [w, d, _letd(d, l)]


def _volume64(mask, d, l):
    """Values at volume: the ceil(fraction * n)-th largest value of a structure (counts
    and voxel numbers are whole numbers and have no 64-bit counterpart)."""
    out = []
    for r in _volume_requests():
        v = {"DOSE": d, "LETD": _letd(d, l), "CDL": C_CDL * l}[r["quantity"]]
        v = v[((mask >> r["struct_bit"]) & 1).bool()].sort(descending=True).values
        at = None
        if "fracs" in r:
            k = [min(max(math.ceil(f * v.numel() - 1e-9 * max(1.0, f * v.numel())), 1), v.numel()) for f in r["fracs"]]
            at = torch.stack([v[i - 1] for i in k]) if v.numel() else None
        out.append(dict(counts=None, at_volume=at, n_voxels=None))
    return out


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        return [_solve64(dict(c, op="solve"), seed + 1000 * i) for i, c in enumerate(_sub_cases(case))]
    if op in ("solve", "request"):
        return _solve64(case, seed)
    rp, col, D, L = _csr(case, seed)
    D, L = _stored(case, rp, D), _stored(case, rp, L)
    n = _spots(case)
    w = _weights(case, seed).double()
    mask = torch.from_numpy(_mask(case)).to(DEV)
    if op in ("products", "csc"):
        P = _Plain(rp, col, D, L, n)
        a, b = (t.double() for t in _coefs(case, seed))
        if case["rows"] == "roi":
            a, b = a * (mask != 0), b * (mask != 0)
        u = P.backward(a, b)
        return u if op == "csc" else list(P.forward(w)) + [u]
    if op == "volume":
        return _volume64(mask, *_Plain(rp, col, D, L, n).forward(w))
    rows = torch.nonzero((mask != 0) & (rp.diff() > 0)).flatten()
    P = _Plain(rp, col, D, L, n, rows)
    con, m = _constraints(), mask[rows]
    if op == "gradient":
        d, l = P.forward(w)
        f, rd, rl = _residual(_objective(case), m, d, l)
        empty = mask[(mask != 0) & (rp.diff() == 0)]
        f += sum(t["weight"] * t["target"] ** 2 * int(((empty >> t["struct_bit"]) & 1).sum()) for t in _objective(case))
        return [f, P.backward(rd, rl)]
    mom = P.moments()
    if op == "step":
        gd, gl, _, reach = _half_space(con, m, mom, *P.forward(w))
        W = float(reach.sum())
        return (w + (RELAX / W if W > 0 else 0.0) * P.backward(gd, gl)).clamp(min=0.0)
    # sweep: consecutive blocks of structure voxels, each projected from where the last one ended
    size = -(-rows.numel() // case["blocks"])
    for k in range(0, rows.numel(), size):
        sub = slice(k, k + size)
        B = _Plain(rp, col, D, L, n, rows[sub])
        gd, gl, _, reach = _half_space(con, m[sub], [t[sub] for t in mom], *B.forward(w))
        W = float(reach.sum())
        if W > 0:
            w = w + RELAX / W * B.backward(gd, gl)
    return w.clamp(min=0.0)
