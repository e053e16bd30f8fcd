"""Kernel variants at the sizes and values where they can go wrong, against the oracle."""
import numpy as np
import pytest

import workloads as W
from tests._pair import gpu_f, oracle_of, rel_err, solver_of

pytestmark = pytest.mark.gpu


def _lbs():
    import paper_1702_01335_gb300 as P
    return P


@pytest.mark.parametrize("pattern", ["rest", "jump", "spike", "staircase", "ramp", "scales"])
def test_fp64_weno_weights_at_vanishing_indicators(pattern):
    """The FP64 WENO weights where one, two or all three smoothness indicators vanish or
    differ by tens of orders of magnitude, per velocity: constant stretches next to a jump, a
    single-cell spike, a staircase, an exactly linear ramp and cell values from 1e-300 to 1.
    One step from that state; both sides round the same few dozen operations, so 1e-13 of the
    largest population bounds them."""
    P = _lbs()
    p = dict(W.C1, Nz=24)
    o = oracle_of(p, None)
    s = solver_of(p, o.dt, P.LBS_FP64)
    z, k = np.arange(24)[:, None], np.arange(o.Q)[None, :]
    d = {"rest": 0.0 * (z + k),
         "jump": 0.1 * (z >= 7 + k % 9),
         "spike": 0.1 * (z == 3 + k % 17),
         "staircase": 0.01 * ((z + k) // 5),
         "ramp": (z - 12) * 2.0 ** -8 + 0.0 * k,
         "scales": 0.1 * 10.0 ** (-12.5 * ((z + k) % 24))}[pattern]
    d = np.ascontiguousarray(d, dtype=np.float64)
    s.set_state(0, d)
    o.f[3:-3] = (1.0 + d) * o.weights()[None, :]
    s.step(1)
    o.step(1)
    assert rel_err(gpu_f(s, o), o.f[3:3 + o.Nz]) < 1e-13


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-5)])
@pytest.mark.parametrize("Nz,n", [(9, 1), (4093, 2), (4095, 3), (4093, 7)])
@pytest.mark.parametrize("reduced", [False, True])
def test_finalize_cells_per_cta_agree(Nz, n, reduced, prec, tol):
    """The finalisation at 8, 16 and 32 cells per CTA (batches of 9, 8186, 12285 and 28651
    cells: ragged last groups) gives the states and profiles of four cells per CTA to
    rounding (FP64: a few ulps of the third moments; FP32 storage: the records' FP32)."""
    P = _lbs()
    from paper_1702_01335_gb300 import Instance, Solver
    pr = P.LBS_FP64 if prec == "fp64" else P.LBS_FP32
    inst = [Instance(Qx=3, Qy=0 if reduced else 2, Qz=2 + b % 3, N_eq=3, Nz=Nz - b % 2, Kn=0.2 + 0.1 * b, u_w=0.3,
                     Pr=2.0 / 3.0, visc_law=b % 2, visc_param=0.75, cfl=0.4) for b in range(n)]
    a, b = Solver(inst, precision=pr), Solver(inst, precision=pr)
    assert not a.set_finalize(1) and b.set_finalize(2)
    a.step(9)
    b.step(9)
    for i in range(n):
        assert rel_err(a.populations(i), b.populations(i)) < tol, i
        pa, pb = a.profiles(i), b.profiles(i)
        assert max(np.abs(pa[k] - pb[k]).max() for k in pa) < tol, i


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("Qx,Qy,Qz,Nz,ZT", [(1, 4, 1, 6, 3), (3, 4, 7, 19, 5), (5, 8, 9, 37, 16), (16, 4, 9, 21, 64),
                                             (4, 12, 3, 11, 12), (1, 100, 3, 9, 4)])
@pytest.mark.parametrize("half", [0, 1])
def test_grouped_layout_matches_one_velocity_per_thread(Qx, Qy, Qz, Nz, ZT, half, prec):
    """Four adjacent velocities per thread (V = 4 with Qy a multiple of four) against one per
    thread (V = 1): one or several chunks with ragged last ones (half ranges of 4 to 576
    velocities, 1, 3 or 25 groups of y), tiles of 3 cells up to the whole channel, one or two
    walls.  The two layouts differ by rounding: 1e-12 (FP64) and 1e-5 (FP32 storage) of the
    largest population after 8 steps."""
    P = _lbs()
    from paper_1702_01335_gb300 import Instance, Solver
    pr = P.LBS_FP64 if prec == "fp64" else P.LBS_FP32
    inst = Instance(Qx=Qx, Qy=Qy, Qz=Qz, N_eq=3, Nz=Nz, A=0.8, half=half, Kn=0.3, u_w=0.4, Pr=2.0 / 3.0, visc_law=1,
                    visc_param=0.5, cfl=0.4)
    a, b = Solver(inst, precision=pr), Solver(inst, precision=pr)
    a.set_tiling(4, ZT, 0)
    b.set_tiling(1, 4, 0)
    rng = np.random.default_rng(7)
    z = np.linspace(-1.0, 1.0, Nz)[:, None]
    d = (0.1 * np.sin(2 * z) + 0.02 * rng.standard_normal((1, inst.Q))) * (1 + 0.1 * z * z)
    for s in (a, b):
        s.set_state(0, d.astype(s.dtype))
        s.step(8)
    tol = 1e-12 if prec == "fp64" else 1e-5
    assert rel_err(a.populations(), b.populations()) < tol
    pa, pb = a.profiles(), b.profiles()
    assert max(np.abs(pa[k] - pb[k]).max() for k in pa) < 10 * tol


@pytest.mark.parametrize("sizes,B", [((1, 1, 1, 1), 1), ((6, 31, 31, 33), 65), ((6, 200, 200, 384), 300),
                                     ((7, 40, 40, 40), 20000), ((260, 300, 300, 17), 40),
                                     ((5, 900, 900, 900), 70)])
def test_network_tiles_at_ragged_sizes(sizes, B):
    """The network's products where its tiles are ragged: single entries, sizes one below and
    above a tile, inner sizes above a staged slice of 256, rows that are not 16-byte multiples,
    a batch past the switch to the large tile; outputs, loss and gradients within the bounds of
    the BF16 roundings (test_gpu_mlp.error_bounds) against the oracle."""
    from oracle import mlp as om
    from tests.test_gpu_mlp import _setup, error_bounds
    net, pf, x, t, xd, td = _setup(sizes, B, seed=9)
    E = error_bounds(pf, x, t)
    y = net.forward(xd).cpu().numpy()
    y_ora, _ = om.forward(pf, x)
    floor = 1e-6  # entries whose every term is zero to rounding
    assert np.all(np.abs(y - y_ora) <= E["y"] + floor)
    loss, g = net.loss_grad(xd, td, want_grad=True)
    L_ora, g_ora = om.loss_and_grads(pf, x, t)
    assert abs(loss / L_ora - 1) < 1e-3
    gg = net.unpack(g.astype(np.float64))
    for k in g_ora:
        assert np.all(np.abs(gg[k] - g_ora[k]) <= E[k] + floor * np.abs(g_ora[k]).max()), k
    net.close()


@pytest.mark.parametrize("Qx,Qy,Qz,Nz", [(8, 8, 8, 81), (7, 7, 11, 73), (9, 0, 31, 70), (2, 0, 4, 64), (4, 4, 4, 23)])
@pytest.mark.parametrize("ZT", [3, 5, 16])
@pytest.mark.parametrize("half", [0, 1])
def test_fp64_one_velocity_layouts_agree(Qx, Qy, Qz, Nz, ZT, half):
    """V = 1 in FP64 (warps that split a tile's cells, in the grouped form or, for the small
    batches, with one velocity per thread; tiles of 3 and 5 cells leave them unevenly filled)
    against V = 2, which marches whole tiles: 1e-12 of the largest population after 6 steps."""
    P = _lbs()
    from paper_1702_01335_gb300 import Instance, Solver
    inst = Instance(Qx=Qx, Qy=Qy, Qz=Qz, N_eq=3, Nz=Nz, A=0.7, half=half, Kn=0.4, u_w=0.5, Pr=2.0 / 3.0, cfl=0.4)
    a, b = Solver(inst), Solver(inst)
    a.set_tiling(1, ZT, 0)
    b.set_tiling(2, 7, 0)
    z = np.linspace(-1.0, 1.0, Nz)[:, None]
    d = 0.1 * np.sin(2 * z) + 0.02 * np.random.default_rng(3).standard_normal((1, inst.Q)) * (1 - 0.2 * z)
    for s in (a, b):
        s.set_state(0, d)
        s.step(6)
    assert rel_err(a.populations(), b.populations()) < 1e-12
    pa, pb = a.profiles(), b.profiles()
    assert max(np.abs(pa[k] - pb[k]).max() for k in pa) < 1e-11


def test_default_tiling_follows_the_batch():
    """The tiling a solver starts with: V = 1 for one small channel and for mostly empty
    512-velocity chunks, V = 4 for several channels of full ones, V = 1 for an odd half range."""
    P = _lbs()
    def tiling(p, n, prec):
        s = solver_of([p] * n, 0.0, prec)
        t = s.tiling()
        s.close()
        return t["V"], t["fuse"]
    assert tiling(W.C2, 1, P.LBS_FP32) == (1, 0)
    assert tiling(W.C2, 8, P.LBS_FP32) == (4, 0)
    assert tiling(dict(W.C1, Nz=128), 64, P.LBS_FP32) == (1, 0)
    assert tiling(dict(W.C2, Qx=9, Qy=9, Qz=9), 64, P.LBS_FP32) == (1, 0)
    assert tiling(W.C2, 1, P.LBS_FP64) == (1, 0)
    assert tiling(W.C2, 16, P.LBS_FP64) == (4, 0)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("offset", [0, 2, 8])
def test_checkpoint_to_device_memory_equals_the_host_copy(prec, offset):
    """lbs_get_state to device memory (one gathering launch) gives the bytes of the copy to
    host memory: ragged instances whose buffers are not adjacent, whole batch and single
    instance, destinations that are not 16-byte aligned, states in either buffer."""
    import torch
    P = _lbs()
    pr = P.LBS_FP64 if prec == "fp64" else P.LBS_FP32
    ps = [dict(W.C1, Nz=11), dict(W.C1, Qx=3, Qy=1, Qz=5, Nz=19), dict(W.C2, Nz=30), dict(W.C1, Qx=3, Qy=3, Nz=7)]
    s = solver_of(ps, 1e-3, pr)
    for steps in (0, 1, 3):
        s.step(steps)
        n = s.state_bytes()
        host = np.zeros(n, np.uint8)
        s.get_state_all_ptr(host.ctypes.data)
        dev = torch.full((n + 16,), 7, dtype=torch.uint8, device="cuda")
        torch.cuda.synchronize()
        s.get_state_all_ptr(dev.data_ptr() + offset, to_host=False)
        got = dev.cpu().numpy()
        assert np.array_equal(got[offset:offset + n], host)
        assert np.all(got[:offset] == 7) and np.all(got[offset + n:] == 7)
        st = s.get_state(1)
        one = st.d.view(np.uint8).ravel() if st.r is None else np.concatenate(
            [st.d.view(np.uint8).ravel(), st.r.view(np.uint8).ravel()])
        s.get_state_device(1, dev.data_ptr() + offset)
        assert np.array_equal(dev.cpu().numpy()[offset:offset + one.size], one)
    s.close()


@pytest.mark.parametrize("Qx,Qy,Qz,Nz,half", [(8, 8, 16, 64, 0), (6, 6, 17, 71, 1), (16, 0, 60, 75, 0)])
def test_large_batch_steps_as_a_single_channel(Qx, Qy, Qz, Nz, half):
    """A batch larger than L2, whose tiles fetch their increments ahead (rows of residuals that are
    16-byte multiples and ones that are not, both walls or the centre line), gives every instance
    the bytes that a solver of that instance alone computes with the same layouts."""
    P = _lbs()
    from paper_1702_01335_gb300 import Instance, Solver
    inst = Instance(Qx=Qx, Qy=Qy, Qz=Qz, N_eq=3, Nz=Nz, A=0.8, half=half, Kn=0.3, u_w=0.4, Pr=2.0 / 3.0, cfl=0.4)
    n = int(9.2e6 / (Nz * inst.Q)) + 1
    a, b = Solver([inst] * n, precision=P.LBS_FP32), Solver(inst, precision=P.LBS_FP32)
    z = np.linspace(-1.0, 1.0, Nz)[:, None]
    d = 0.1 * np.sin(2 * z) + 0.02 * np.random.default_rng(5).standard_normal((1, inst.Q)) * (1 + 0.1 * z)
    for s, which in ((a, (0, n - 1)), (b, (0,))):
        s.set_tiling(4, 12, 0)
        s.set_finalize(2)
        for i in which:
            s.set_state(i, d.astype(np.float32))
        s.step(5)
    one = b.get_state(0)
    for i in (0, n - 1):
        st = a.get_state(i)
        assert np.array_equal(st.d, one.d) and np.array_equal(st.r, one.r)


# (precision, Qx, Qy, Qz, Nz, V, ZT): three-cell z-split tiles at the smallest velocity sets (one
# and two nodes per sign of p_z, phi / chi too), longer z-split tiles, the grouped march with
# whole-tile and split warps, ragged chunks and tiles
FOLDED = [("fp64", 1, 1, 1, 6, 1, 3), ("fp64", 1, 1, 2, 9, 1, 3), ("fp64", 1, 2, 1, 6, 1, 4), ("fp64", 2, 1, 1, 6, 1, 4),
          ("fp64", 1, 0, 1, 9, 1, 3), ("fp64", 2, 2, 2, 7, 1, 3), ("fp64", 7, 7, 11, 23, 1, 5), ("fp64", 8, 8, 16, 41, 1, 16),
          ("fp64", 8, 8, 16, 41, 4, 8), ("fp64", 3, 4, 7, 19, 4, 3), ("fp64", 1, 4, 1, 6, 4, 3),
          ("fp32", 1, 4, 1, 6, 4, 3), ("fp32", 8, 8, 16, 41, 4, 13), ("fp32", 5, 8, 9, 23, 4, 5), ("fp32", 1, 1, 1, 6, 1, 3)]


@pytest.mark.parametrize("fuse", [1, 2])
@pytest.mark.parametrize("prec,Qx,Qy,Qz,Nz,V,ZT", FOLDED)
def test_folded_and_split_finalisation_agree_with_separate_launches(prec, Qx, Qy, Qz, Nz, V, ZT, fuse):
    """The finalisation folded into the stage kernel (fuse = 1) and split stepping (fuse = 2) against
    separate launches, same layout.  Folded, the cells are grouped by z-tile, so only the choice
    between the small-drift series and erfc can differ: 1e-12 (FP64) and 1e-5 (FP32 storage) of the
    largest population after 9 steps, as between layouts."""
    P = _lbs()
    from paper_1702_01335_gb300 import Instance, Solver
    pr = P.LBS_FP64 if prec == "fp64" else P.LBS_FP32
    inst = [Instance(Qx=Qx, Qy=Qy, Qz=Qz, N_eq=3, Nz=Nz, A=0.8, half=b % 2, Kn=0.3 + 0.1 * b, u_w=0.4, Pr=2.0 / 3.0,
                     visc_law=1, visc_param=0.5, cfl=0.1) for b in range(3)]
    a, b = Solver(inst, precision=pr), Solver(inst, precision=pr)
    a.set_tiling(V, ZT, 0)
    b.set_tiling(V, ZT, fuse)
    rng = np.random.default_rng(7)
    z = np.linspace(-1.0, 1.0, Nz)[:, None]
    for i in range(3):
        d = (0.1 * np.sin(2 * z) + 0.02 * rng.standard_normal((1, inst[i].Q))) * (1 + 0.1 * z * z)
        for s in (a, b):
            s.set_state(i, d.astype(s.dtype))
    for s in (a, b):
        s.step(9)
    tol = 1e-12 if prec == "fp64" else 1e-5
    for i in range(3):
        assert rel_err(b.populations(i), a.populations(i)) < tol, i
        pa, pb = a.profiles(i), b.profiles(i)
        assert max(np.abs(pa[k] - pb[k]).max() for k in pa) < 10 * tol, i
        assert abs(a.residual(i) - b.residual(i)) <= 100 * tol * max(a.residual(i), 1e-2), i


def _drop_cuda_error():
    """A refused copy stays the CUDA runtime's last error; torch's next check takes and reports it."""
    import torch
    try:
        torch.zeros(1, device="cuda")
    except RuntimeError:
        pass
    torch.zeros(1, device="cuda")


def _short_allocation(nbytes):
    """A device allocation of its own (driver API) of nbytes: address, release."""
    import ctypes

    import torch
    torch.zeros(1, device="cuda")
    cu, p = ctypes.CDLL("libcuda.so.1"), ctypes.c_uint64()
    assert cu.cuMemAlloc_v2(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0
    return p.value, lambda: cu.cuMemFree_v2(p)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_checkpoint_to_a_short_allocation_is_refused(prec):
    """A device allocation of its own that ends before the state does: refused as by a copy, and the
    solver is as before.  (It lies in a mapped page much larger than the state, so that nothing
    could fault in any case.)"""
    P = _lbs()
    s = solver_of(dict(W.C1, Nz=11), 1e-3, P.LBS_FP64 if prec == "fp64" else P.LBS_FP32)
    assert s.state_bytes() < 1 << 17
    p, release = _short_allocation(s.state_bytes() // 2)
    s.step(2)
    before = s.get_state(0)
    with pytest.raises(P.LbsError):
        s.get_state_all_ptr(p, to_host=False)
    release()
    _drop_cuda_error()
    after = s.get_state(0)
    assert np.array_equal(before.d, after.d) and (before.r is None or np.array_equal(before.r, after.r))
    s.close()


def test_checkpoint_after_another_calls_error():
    """A CUDA error that an earlier call left behind (here a refused checkpoint) is not taken for the
    next checkpoint's own."""
    import torch
    P = _lbs()
    s = solver_of(dict(W.C1, Nz=11), 1e-3, P.LBS_FP32)
    n = s.state_bytes()
    host, dev = np.zeros(n, np.uint8), torch.zeros(n, dtype=torch.uint8, device="cuda")
    p, release = _short_allocation(n // 2)
    s.step(2)
    s.get_state_all_ptr(host.ctypes.data)
    torch.cuda.synchronize()
    with pytest.raises(P.LbsError):
        s.get_state_all_ptr(p, to_host=False)
    s.get_state_all_ptr(dev.data_ptr(), to_host=False)
    release()
    _drop_cuda_error()
    assert np.array_equal(dev.cpu().numpy(), host)
    s.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("sizes", [[(7, 7, 11, 65 + 2 * b) for b in range(5)], [(1, 1, 1, 6)],
                                   [(9, 9, 31, 151)] + [(3, 1, 1 + b % 2, 6 + b % 5) for b in range(39)],
                                   [(1, 1 + b % 2, 1, 6 + b % 3) for b in range(1030)]],
                         ids=["odd", "smallest", "uneven", "many"])
def test_checkpoint_at_every_alignment(sizes, prec):
    """A checkpoint to device memory at every even offset from 16 bytes equals the copy to host
    memory: states that are not whole 16-byte words, one large instance among small ones, states
    shorter than a warp's share, more than 32 and more than 1024 instances; nothing beside it is
    written."""
    import torch
    P = _lbs()
    from paper_1702_01335_gb300 import Instance, Solver
    s = Solver([Instance(Qx=x, Qy=y, Qz=z, N_eq=3, Nz=Nz, A=0.5, Kn=0.3, u_w=0.4, Pr=2.0 / 3.0, dt=1e-3)
                for x, y, z, Nz in sizes], precision=P.LBS_FP64 if prec == "fp64" else P.LBS_FP32)
    n = s.state_bytes()
    rng = np.random.default_rng(3)
    host, out = rng.integers(0, 256, n, dtype=np.uint8), np.zeros(n, np.uint8)
    nd = n if prec == "fp64" else n // 6 * 4
    host[:nd] = (0.1 * rng.standard_normal(nd // 8 if prec == "fp64" else nd // 4)).astype(s.dtype).view(np.uint8)
    s.set_state_all_ptr(host.ctypes.data)
    for steps in (0, 1):  # the state in either buffer
        s.step(steps)
        s.get_state_all_ptr(out.ctypes.data)
        assert steps or np.array_equal(out, host)
        for offset in range(0, 16, 2):
            dev = torch.full((n + 64,), 7, dtype=torch.uint8, device="cuda")
            torch.cuda.synchronize()
            s.get_state_all_ptr(dev.data_ptr() + 16 + offset, to_host=False)
            got = dev.cpu().numpy()
            assert np.array_equal(got[16 + offset:16 + offset + n], out)
            assert np.all(got[:16 + offset] == 7) and np.all(got[16 + offset + n:] == 7)
    s.close()
