"""One handle that loads plan after plan, keeping the buffers that fit: every
output equals that of a fresh handle bit for bit, whatever was loaded before
(larger and smaller plans, within a factor of two and beyond it, other value
formats, row sets, index widths and launch shapes, empty rows, empty plans,
loads that failed)."""
import numpy as np
import pytest

import phantom

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__
    __graft_entry__.build()
    from paper_2509_20012_gb300 import fredopt
    return fredopt


def plan(n_vox, n, density, empty, seed):
    rp, col, D, L = phantom.random_csr(n_vox, n, density, seed=seed, empty_rows=empty)
    mask = np.random.default_rng(seed).choice(np.array([0, 1, 2, 3], np.uint32), n_vox)
    return rp, col, D, L, mask, n


CONS = [dict(struct_bit=0, kind="DOSE_MIN", bound=9.0, priority=1.0),
        dict(struct_bit=1, kind="DOSE_MAX", bound=11.0, priority=0.5),
        dict(struct_bit=1, kind="LETD_MAX", bound=5.0, priority=2.0)]
OBJ = [dict(struct_bit=1, quantity="CDL", target=0.0, weight=1.0),
       dict(struct_bit=0, quantity="DOSE", target=10.0, weight=0.1)]


def outputs(h, args, kw, n_solve=4):
    """Everything that a loaded plan gives."""
    h.load_influence(*args, **kw)
    rng = np.random.default_rng(9)
    x = rng.uniform(0.2, 1.5, h.n_spots).astype(np.float32)
    a, b = (rng.normal(size=h.n_vox).astype(np.float32) for _ in range(2))
    out = {"storage": np.array(h.storage())}
    for k, v in zip(("cp", "row", "D", "L"), h.get_csc()):
        out[k] = v
    for k, v in zip(("dd", "ll", "dl"), h.get_moments()):
        out[k] = v
    out["vox"], out["mask"] = h.get_rows()
    out["tuning"] = np.array(h.tuning())
    h.set_constraints(CONS)
    h.set_objective(OBJ)
    out["dose"], out["lw"] = h.forward(x)
    out["u"] = h.backward(a, b)
    f, g = h.objective(x)
    out["f"], out["g"] = np.array(f), g
    out["step"] = h.feasibility_step(x)
    out["sweep"] = h.sweep_step(x, 5)
    for q in ("DOSE", "CDL", "LETD"):
        out["map" + q] = h.quantity_map(x, q)
    st = h.volume_stats([dict(quantity="DOSE", struct_bit=b, edges=np.linspace(0, 30, 31), fracs=[0.1, 0.9])
                         for b in (0, 1, 5)], x)
    for i, s in enumerate(st):
        out[f"counts{i}"], out[f"at{i}"], out[f"n{i}"] = s["counts"], s["at_volume"], np.array(s["n_voxels"])
    for sweep_blocks in (0, 3):
        w, d, l, rep = h.superiorize(x, n_solve, 0.99, 1.0, sweep_blocks=sweep_blocks)
        out[f"w{sweep_blocks}"], out[f"d{sweep_blocks}"], out[f"l{sweep_blocks}"] = w, d, l
        rep.pop("device_ms")
        out[f"rep{sweep_blocks}"] = np.array([np.atleast_1d(v).astype(np.float64).sum() for v in rep.values()])
        out[f"log{sweep_blocks}"] = np.array([list(e.values()) for e in h.get_log()])
    return out


@pytest.mark.parametrize("device", [False, True])
def test_reload_equals_fresh_handle(lib, device):
    big, mid, small = plan(900, 700, 0.3, 40, 1), plan(700, 601, 0.25, 0, 2), plan(90, 33, 0.4, 5, 3)
    wide = plan(300, 70003, 0.002, 7, 4)
    none = plan(50, 9, 0.0, 50, 5)
    thin = plan(5000, 601, 0.004, 600, 6)
    seq = [(big, {}), (mid, {}), (big, {}), (mid, dict(fmt="bf16")), (big, dict(fmt="fp16", rows="roi")),
           (big, dict(fmt="fp32", rows="roi", index32=True)), (mid, dict(index32=True)), (small, {}),
           (small, dict(fmt="bf16", shared=True)), (wide, {}), (mid, dict(fmt="fp16", shared=True)), (none, {}),
           (mid, dict(rows="roi")), (thin, dict(fmt="bf16")), (big, {}), (thin, dict(rows="roi")),
           (mid, dict(fmt="bf16", rows="roi"))]
    bad = list(mid)
    bad[2] = mid[2].copy()
    bad[2][7] = np.inf

    def put(args):
        if not device:
            return args
        import torch
        t = [torch.from_numpy(a.view(np.int32) if a.dtype == np.uint32 else a).cuda() for a in args[:5]]
        torch.cuda.synchronize()
        return (*t, args[5])

    with lib.Handle(0) as h:
        for i, (args, kw) in enumerate(seq):
            if i % 4 == 3:  # a load that is refused in between
                with pytest.raises(lib.FredoptError):
                    h.load_influence(*put(bad), **kw)
            got = outputs(h, put(args), kw)
            with lib.Handle(0) as fresh:
                want = outputs(fresh, put(args), kw)
            for k in want:
                np.testing.assert_array_equal(got[k], want[k], err_msg=f"load {i}, {kw}: {k}")
