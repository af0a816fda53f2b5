"""Vectors that lie on the device give what the same vectors give as host arrays."""
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


def cuda(x):
    import torch
    return torch.from_numpy(x).cuda()


@pytest.mark.parametrize("n", [1, 255, 2250, 20001])
def test_begin(lib, n):
    """beta0 (a sum over w0, default 0.1 ||w0||) and the solve bit for bit; the
    error of the first bad element."""
    rp, col, D, L = phantom.random_csr(400, n, min(1.0, 60.0 / n), seed=n)
    rng = np.random.default_rng(n)
    mask = rng.choice(np.array([0, 1, 2], np.uint32), 400)
    w0 = rng.uniform(0.1, 2.0, n).astype(np.float32)
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n)
        h.set_constraints([dict(struct_bit=0, kind="DOSE_MAX", bound=1.0, priority=1.0)])
        h.set_objective([dict(struct_bit=1, quantity="CDL", target=0.0, weight=1.0)])
        a = h.superiorize(w0, 5, 0.99, 1.0)
        b = h.superiorize(cuda(w0), 5, 0.99, 1.0)
        assert a[3]["beta0"] == b[3]["beta0"]
        assert abs(a[3]["beta0"] - 0.1 * np.linalg.norm(w0.astype(np.float64))) <= 1e-14 * a[3]["beta0"] * np.sqrt(n)
        for x, y in zip(a[:3], b[:3]):
            np.testing.assert_array_equal(x, y.cpu().numpy())
        for bad, code in (((-1.0, np.nan), -1), ((np.nan, -1.0), -4), ((np.inf, 0.0), -4), ((-0.0, -1e-30), -1)):
            w = w0.copy()
            w[n // 2], w[n - 1] = bad
            if n == 1:  # the second value is the only one
                code = -4 if not np.isfinite(bad[1]) else -1 if bad[1] < 0 else None
            for x in (w, cuda(w)):
                if code is None:
                    h.begin(x, 0.99, 1.0)
                    continue
                with pytest.raises(lib.FredoptError) as e:
                    h.begin(x, 0.99, 1.0)
                assert e.value.code == code


CONS = [dict(struct_bit=0, kind="DOSE_MIN", bound=4.0, priority=1.0),
        dict(struct_bit=1, kind="DOSE_MAX", bound=2.0, priority=0.5),
        dict(struct_bit=1, kind="LETD_MAX", bound=5.0, priority=2.0)]
OBJ = [dict(struct_bit=1, quantity="CDL", target=0.0, weight=1.0),
       dict(struct_bit=0, quantity="DOSE", target=3.0, weight=0.1)]


def at(buf, offset, n):
    """n floats of a device buffer, `offset` floats after a 256-byte boundary."""
    assert buf.data_ptr() % 256 == 0
    return buf[offset:offset + n]


@pytest.mark.parametrize("n", [1, 3, 124, 125, 128, 513])
@pytest.mark.parametrize("rows,n_vox", [("all", 500), ("roi", 501)])
def test_vectors_in_place(lib, n, rows, n_vox):
    """Inputs and outputs at every alignment of a float, an output that is the input,
    and one that overlaps it in part: bit for bit the host arrays' results, the
    inputs unchanged, nothing written beside the outputs."""
    import torch
    rp, col, D, L = phantom.random_csr(n_vox, n, min(1.0, 0.2 + 4.0 / n), seed=n, empty_rows=13)
    rng = np.random.default_rng(n)
    mask = rng.choice(np.array([0, 1, 2, 3], np.uint32), n_vox)
    x = rng.uniform(0.2, 2.0, n).astype(np.float32)
    aD, aL = (rng.normal(size=n_vox).astype(np.float32) for _ in range(2))
    big = 4096
    L_ = lib.load_library()
    with lib.Handle(0) as h:
        h.load_influence(rp, col, D, L, mask, n, rows=rows)
        h.set_constraints(CONS)
        h.set_objective(OBJ)
        import ctypes
        f = ctypes.c_double()
        calls = {  # name: (inputs, output lengths, the call on (inputs, outputs, flags))
            "step": ([x], [n], lambda i, o, fl: L_.fredopt_feasibility_step(h.h, i[0], 1.0, 0.9, 0, o[0], fl)),
            "violated": ([x], [n], lambda i, o, fl: L_.fredopt_feasibility_step(h.h, i[0], 1.0, 0.9, 1, o[0], fl)),
            "sweep": ([x], [n], lambda i, o, fl: L_.fredopt_sweep_step(h.h, i[0], 1.0, 0.9, 0, 3, o[0], fl)),
            "objective": ([x], [n], lambda i, o, fl: L_.fredopt_objective(h.h, i[0], ctypes.byref(f), o[0], fl)),
            "forward": ([x], [n_vox, n_vox], lambda i, o, fl: L_.fredopt_forward(h.h, i[0], o[0], o[1], fl)),
            "backward": ([aD, aL], [n], lambda i, o, fl: L_.fredopt_backward(h.h, i[0], i[1], o[0], fl)),
            "map": ([x], [n_vox], lambda i, o, fl: L_.fredopt_quantity_map(h.h, i[0], 2, o[0], fl)),
        }
        for name, (ins, outs, call) in calls.items():
            want = [np.empty(k, np.float32) for k in outs]
            assert call([a.ctypes.data for a in ins], [o.ctypes.data for o in want], 0) == 0
            f_want = f.value
            for shift_in in range(4):
                for shift_out in range(4):
                    bufs = [torch.full((big,), -7.0, device="cuda") for _ in ins]
                    for b, a in zip(bufs, ins):
                        at(b, 64 + shift_in, len(a)).copy_(torch.from_numpy(a))
                    res = [torch.full((big,), -9.0, device="cuda") for _ in outs]
                    torch.cuda.synchronize()
                    f.value = 0.0
                    rc = call([b.data_ptr() + 4 * (64 + shift_in) for b in bufs],
                              [r.data_ptr() + 4 * (64 + shift_out) for r in res], lib.DEVICE_PTR)
                    assert rc == 0
                    msg = f"{name}, input + {shift_in}, output + {shift_out} floats"
                    for r, w in zip(res, want):
                        got = r.cpu().numpy()
                        np.testing.assert_array_equal(got[64 + shift_out:64 + shift_out + len(w)], w, err_msg=msg)
                        assert np.all(got[:64 + shift_out] == -9.0) and np.all(got[64 + shift_out + len(w):] == -9.0), msg
                    for b, a in zip(bufs, ins):
                        np.testing.assert_array_equal(at(b, 64 + shift_in, len(a)).cpu().numpy(), a, err_msg=msg)
                    if name == "objective":
                        assert f.value == f_want
            # the output over the input: the same vector, and shifted by up to its length
            for d in sorted({0, 1, 2, 4, n // 2, n - 1, -1, -4, -(n // 2), 1 - n} if outs[0] == n and len(ins) == 1 else ()):
                buf = torch.full((big,), -7.0, device="cuda")
                at(buf, 1024, n).copy_(torch.from_numpy(x))
                torch.cuda.synchronize()
                rc = call([buf.data_ptr() + 4 * 1024], [buf.data_ptr() + 4 * (1024 + d)], lib.DEVICE_PTR)
                assert rc == 0
                np.testing.assert_array_equal(at(buf, 1024 + d, n).cpu().numpy(), want[0], err_msg=f"{name}, shift {d}")
        # the statistics take a device fluence too
        req = [dict(quantity=q, struct_bit=b, edges=np.linspace(0, 20, 21), fracs=[0.1, 0.7]) for q in ("DOSE", "LETD")
               for b in (0, 1)]
        want = h.volume_stats(req, x)
        for shift in range(4):
            buf = torch.zeros(big, device="cuda")
            at(buf, shift, n).copy_(torch.from_numpy(x))
            torch.cuda.synchronize()
            for g, w in zip(h.volume_stats(req, at(buf, shift, n)), want):
                np.testing.assert_array_equal(g["counts"], w["counts"])
                np.testing.assert_array_equal(g["at_volume"], w["at_volume"])
