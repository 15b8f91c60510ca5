"""The forms that the host chooses by size, precision and body: small and large
FP64 tiles, the FP64 march along z, bodies at rest and moving, the field
conversion of a whole batch in one launch, cells below and beyond yield, the
seeding of small and large boxes, and offsets of 64 bits.  Bars as for the
plain parity tests: FP64 relative L1 per plane <= 1e-12 after one step and
<= 1e-8 after several with the device's own dt, FP32 <= 1e-4."""
import numpy as np
import pytest

import workloads as W
from gpu_util import rel_l1, run_both
from test_gpu_3d_marching import CASES as MARCHING

pytestmark = pytest.mark.gpu

B = pytest.importorskip("paper_2111_11806_gb300.binding")

# (dim, size, materials, solid): a tile and one cell more or less, small tiles
# (32, 32 x 4) and, from about 20 000 cells on, large ones (256, 32 x 8)
TILES = [
    (1, (31,), 1, False), (1, (33,), 2, False), (1, (257,), 2, True), (1, (4865,), 1, False), (1, (20001,), 2, False),
    (2, (33, 5), 1, False), (2, (64, 12), 2, False), (2, (31, 9), 3, False), (2, (65, 13), 2, True),
    (2, (161, 131), 1, False), (2, (161, 131), 2, False), (2, (161, 131), 2, True), (2, (161, 131), 3, True),
]


@pytest.mark.parametrize("moving", [False, True], ids=["rest", "moving"])
@pytest.mark.parametrize("dim,n,nmat,solid", TILES)
def test_fp64_tiles(dim, n, nmat, solid, moving):
    wl = W.random_state(dim, n, nmat, solid, seed=601, amp=0.02 if solid else 0.1)
    if moving:
        wl.body_v = (25.0, -15.0, 0.0)[:dim]
    o, g = run_both(wl, 1, B.DFV_FP64)
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= 1e-12), err


@pytest.mark.parametrize("name,make", MARCHING, ids=[c[0] for c in MARCHING])
def test_fp64_marching(name, make):
    wl = make()
    o, g = run_both(wl, 1, B.DFV_FP64)
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= 1e-12), err


# body at the start and from the third step on: values that change under a
# kept step, and motion that begins or ends
BODIES = [((20.0, 5.0), (-30.0, 10.0)), ((0.0, 0.0), (15.0, 0.0)), ((15.0, 0.0), (0.0, 0.0))]


@pytest.mark.parametrize("first,then", BODIES, ids=["other_velocity", "starts", "stops"])
@pytest.mark.parametrize("dim,n", [(2, (50, 41)), (3, (30, 22, 19))])
def test_body_replaced_between_runs(dim, n, first, then):
    from oracle import Oracle
    wl = W.random_state(dim, n, 1, False, seed=602)
    wl.body_v = first + (0.0,) * (dim - 2)
    o, g = Oracle.from_workload(wl), B.Grid.from_workload(wl, precision=B.DFV_FP64)
    for v in (None, then):
        if v is not None:
            o.set_body(v)
            g.set_body(v)
        g.run(3, 0.6)
        for _ in range(3):
            o.step(o.compute_dt(0.6))
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= 1e-8), err


@pytest.mark.parametrize("precision", [B.DFV_FP64, B.DFV_FP32], ids=["fp64", "fp32"])
def test_batch_fields_on_the_device(precision):
    """More instances than one launch's pointers, of 20 to 3201 cells, with
    device pointers: the bits of the per-instance calls, in and out, and the
    step of each instance's own dt as a grid of its own takes it."""
    import torch
    sizes = [(5 + i % 7, 4 + i % 5) for i in range(298)] + [(97, 33), (64, 32)]
    wls = [W.random_state(2, n, 1, False, seed=700 + i, amp=0.02) for i, n in enumerate(sizes)]
    a, b = B.Batch(wls, precision=precision), B.Batch(wls, precision=precision)
    dev = [torch.from_numpy(wl.prim).cuda() for wl in wls]
    ptrs = (B._vp * len(wls))(*[B._vp(t.data_ptr()) for t in dev])
    B._bcheck(B.load().dfv_batch_set_all_fields(a._h, ptrs, 1), a._h, "set")
    for i, wl in enumerate(wls):
        b.set_fields(i, wl.prim)
    for c in (a, b):
        c.run(1, 0.5)
    for which in (B.DFV_FIELDS_CONSERVED, B.DFV_FIELDS_PRIMITIVE):
        outs = [torch.full_like(t, -7.0) for t in dev]
        ptrs = (B._vp * len(wls))(*[B._vp(t.data_ptr()) for t in outs])
        B._bcheck(B.load().dfv_batch_get_all_fields(a._h, ptrs, which, 1), a._h, "get")
        torch.cuda.synchronize()
        for i in range(len(wls)):
            np.testing.assert_array_equal(outs[i].cpu().numpy(), b.get_fields(i, which))
    for i in (0, 17, 298, 299):
        g = B.Grid.from_workload(wls[i], precision=precision)
        assert a.time(i)[0] == pytest.approx(g.run(1, 0.5), rel=1e-12 if precision == B.DFV_FP64 else 1e-6)


@pytest.mark.parametrize("strain", [0.0, 1e-3, 0.03, 0.3, 1.0])
@pytest.mark.parametrize("nmat", [2, 3])
def test_fp32_stretch_below_and_beyond_yield(nmat, strain):
    wl = W.random_state(2, (40, 37), nmat, True, seed=603, amp=0.02)
    L = W.layout(2, nmat, True)
    V = wl.prim[L["iv"]: L["iv"] + L["nv"]]
    one = np.round(V)
    V[:] = one + strain * (V - one)
    o, g = run_both(wl, 1, B.DFV_FP32)
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= 1e-4), err


@pytest.mark.parametrize("n,radius", [(33, 0.05), (200, 0.02), (200, 0.3)])
def test_seeding_of_small_and_large_boxes(n, radius):
    wl = W.cylinder_2d(n, radius=radius)
    o, g = run_both(wl, 1, B.DFV_FP64)
    err = rel_l1(g.cons(), o.cons(), wl)
    assert np.all(err <= 1e-12), err


@pytest.mark.parametrize("n", [(5, 4), (29, 64), (230, 210), (900, 420)])
def test_gas_rows_chosen_by_size_give_the_same_bits(n):
    """The chunk length that the size chooses (1, 2 or 5 rows; 4 in the batch)
    against 8 rows."""
    wl = W.cylinder_2d(n[0], ny=n[1])
    ref = B.Grid.from_workload(wl, precision=B.DFV_FP32, gas_rows=8)
    t = ref.run(4, 0.6)
    g = B.Grid.from_workload(wl, precision=B.DFV_FP32)
    assert g.run(4, 0.6) == t
    np.testing.assert_array_equal(g.cons(), ref.cons())
    b = B.Batch([wl, wl])
    b.set_all_fields()
    b.run(4, 0.6)
    for i in range(2):
        np.testing.assert_array_equal(b.get_fields(i), ref.cons())


def test_gas_planes_of_4_gib_take_64_bit_offsets():
    """An FP32 2-D gas whose five planes take 4 GiB: its first and last cells
    (a seeded disc among these) against the general kernel on the same grid,
    within the bar of that comparison on small grids (relative L1 1e-5)."""
    import torch
    n, h, m = (16400, 13100), 2.0 ** -10, (150, 120)
    ends = [(slice(0, m[1]), slice(0, m[0])), (slice(n[1] - m[1], None), slice(n[0] - m[0], None))]
    x = torch.arange(n[0], dtype=torch.float64, device="cuda")[None, :]
    y = torch.arange(n[1], dtype=torch.float64, device="cuda")[:, None]
    w = torch.empty((5, n[1], n[0]), dtype=torch.float64, device="cuda")
    got = []
    for general in (False, True):
        w[0] = 1.2 + 0.1 * torch.sin(0.13 * x) * torch.cos(0.11 * y)
        w[1] = 40.0 * torch.sin(0.07 * x + 0.05 * y)
        w[2] = 30.0 * torch.cos(0.06 * x) * torch.sin(0.09 * y)
        w[3] = 1e5 * (1.0 + 0.05 * torch.cos(0.08 * x - 0.1 * y))
        w[4] = torch.clamp(20.5 - torch.hypot(x - (n[0] - 60), y - (n[1] - 50)), 0.0, 1.0)
        g = B.Grid(2, n, (0.0, 0.0), (n[0] * h, n[1] * h), [W.AIR], precision=B.DFV_FP32, general_stage=general)
        g.set_fields(w)
        g.set_body()
        for _ in range(2):
            g.step(0.2 * h / 500.0)
        g.get_fields(out=w)
        torch.cuda.synchronize()
        g.check()
        del g
        got.append([w[(slice(None),) + e].cpu() for e in ends])
    for a, b in zip(*got):
        err = (a - b).abs().sum(dim=(1, 2)) / b.abs().sum(dim=(1, 2)).clamp(min=1e-3)
        assert bool((err <= 1e-5).all()), err
