"""The list build, the passes, the resident step and the device-array entry
points at the sizes where they can go wrong: edges of sub-chunks, rows longer
than what a lane or a wave of entries holds, odd and large exponents, blocks
whose rows leave no spare warp, unaligned arrays, positions on the box faces.

Forces, energies and bond counts against the oracle at the tolerances of the
parity tests (FP32 1e-5, FP64 1e-12 of the oracle's error scales, from the
arithmetic); two ways of computing the same thing are held to the same bits.
"""
import numpy as np
import pytest

from gpu_helpers import TOL, assert_forces_match, assert_thermo_match, make_gpu, oracle_pairs
from paper_1912_08569_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1912_08569_gb300.build import build

    build()


def _wl(count, density=0.5, lam=1.0, seed=11, **pair):
    wl = inputs.workload("mix2k", lambda3=lam, n=count, density=density, seed=seed)
    if pair:
        wl["pairs"] = inputs.swap_pairs(lambda3=lam, **pair)
    return wl


def _check(orc, wl, precision, s):
    s.compute_forces()
    ref = orc.forces(wl["x"], wl["types"], wl["n_types"], oracle_pairs(orc, wl), wl["box"], fp32=precision == "fp32")
    assert_forces_match(s.forces(), ref, TOL[precision], precision)
    assert_thermo_match(s.thermo(), ref, TOL[precision], precision)


# ten blocks: 768 (FP32; up to 1,024 in the wide kernel) and 512 (FP64) particles
# fill a sub-chunk
@pytest.mark.parametrize("precision,n", [("fp32", 7680), ("fp32", 7681), ("fp32", 10240), ("fp32", 10241), ("fp32", 15370),
                                         ("fp64", 5120), ("fp64", 5121)])
def test_sub_chunk_edges(orc, precision, n):
    wl = _wl(n)
    s = make_gpu(wl, precision)
    s.set_grid(10)
    _check(orc, wl, precision, s)


# several FP64 sub-chunks per block, all or some of them without a reactive pair: the
# S pass runs no wave of entries there, and the staging is filled again at once
@pytest.mark.parametrize("some", [False, True])
@pytest.mark.parametrize("n", [5121, 12_300])
def test_sub_chunks_without_reactive_pairs(orc, n, some):
    wl = _wl(n)
    wl["n_types"] = 3
    wca = wl["pairs"][(0, 0)]
    wl["types"] = np.where(wl["x"][:, 0] < (0.3 if some else 0.0) * wl["box"][0], wl["types"], 2).astype(np.int32)
    wl["pairs"] = {k: wl["pairs"].get(k, wca) for k in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))}
    if not some:
        wl["pairs"][(0, 1)] = wca
    s = make_gpu(wl, "fp64")
    s.set_grid(10)
    _check(orc, wl, "fp64", s)


# r_cut = 2.4: about 34 reactive and 3 other partners, more than a lane of the
# build holds; on ten blocks of 300 FP64 particles several waves of entries
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("grid", [0, 10])
def test_long_rows(orc, precision, grid):
    wl = _wl(3000, n=10, rcut=2.4)
    s = make_gpu(wl, precision)
    if grid:
        s.set_grid(grid)
    _check(orc, wl, precision, s)


# reactive and other exponents: short products, selected squarings, odd powers
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("n,wca_n", [(10, 6), (12, 6), (9, 5), (1, 7), (100, 12), (128, 127)])
def test_exponents(orc, precision, n, wca_n):
    wl = _wl(900, density=0.3, n=n, wca_n=wca_n)
    if n >= 100:  # no overlaps on the steep walls
        wl["x"] = inputs.rsa_positions(900, wl["box"], 1.0, seed=4)
    _check(orc, wl, precision, make_gpu(wl, precision))


@pytest.mark.parametrize("n,density", [(90, 0.2), (114_000, 0.4)])  # empty blocks; rows in every warp
def test_resident_equals_two_barrier_path_at_the_ends(n, density):
    wl = _wl(n, density, seed=5)
    wl["v"] = inputs.maxwell_velocities(n, 0.2, 1.0, seed=6)
    a, b = make_gpu(wl, "fp32"), make_gpu(wl, "fp32")
    b.set_resident(False)
    logs = []
    for s in (a, b):
        s.set_thermo_log(7, 20)
        s.run(120, 0.001, 0.2, 1.0)
        logs.append(s.thermo_log())
    assert a.thermo()["resident_steps"] == 120 and b.thermo()["resident_steps"] == 0
    for p, q in zip(a.state(), b.state()):
        assert np.array_equal(p, q)
    assert np.array_equal(logs[0]["step"], logs[1]["step"])
    assert np.array_equal(logs[0]["n_bonds"], logs[1]["n_bonds"])
    # FP32 terms, summed in another order: 1e-5 as for the energies against the oracle
    for k in ("U2", "U3", "K"):
        np.testing.assert_allclose(logs[0][k], logs[1][k], rtol=1e-5)


# the energies of equal runs are the same bits (the wave of an FP64 block is lined
# up by 16 warps): forces and a logged run, blocks of one wave, of several, of
# several sub-chunks
@pytest.mark.parametrize("n,grid", [(3000, 0), (3000, 10), (5300, 10)])
def test_fp64_energies_repeat(n, grid):
    wl = _wl(n, 0.5)
    first = None
    for _ in range(12):
        s = make_gpu(wl, "fp64")
        s.set_grid(grid)
        s.compute_forces()
        th = s.thermo()
        s.set_thermo_log(1, 6)
        s.run(6, 0.001, 0.1, 1.0)
        log = s.thermo_log()
        got = [th["U2"], th["U3"], th["W"], *(log[k] for k in ("U2", "U3", "K", "W"))]
        if first is None:
            first = got
        for p, q in zip(first, got):
            assert np.array_equal(p, q)


# list positions are unsigned 32-bit numbers; host calls only, no buffer of that size.
# FP32 rows take max_nn + 6 entries rounded up to a multiple of four
@pytest.mark.parametrize("precision,max_nn,stride", [("fp32", 64, 72), ("fp32", 4096, 4104), ("fp64", 64, 64),
                                                     ("fp64", 4096, 4096)])
def test_lists_beyond_32_bit_positions_are_refused(precision, max_nn, stride):
    import torch
    from paper_1912_08569_gb300 import _abi as A

    blocks = 2 * torch.cuda.get_device_properties(0).multi_processor_count
    limit = (2 ** 32 - 2 ** 16) // stride - min(blocks, 320)
    code = A.SWP_FP64 if precision == "fp64" else A.SWP_FP32
    for n, fits in ((limit, True), (limit + 1, False)):
        ctx = A.swp_create(n, 1, [50.0] * 3, code, 0)
        A.swp_set_nlist(ctx, 0.3, 8)
        if fits:
            A.swp_set_nlist(ctx, 0.3, max_nn)
            assert A.swp_nlist_size(ctx) >= 4 * stride * n
        else:
            with pytest.raises(A.SwpError, match="list entries"):
                A.swp_set_nlist(ctx, 0.3, max_nn)
            assert A.swp_nlist_size(ctx) < 4 * 24 * (n + 1000)  # as before the refused call
        A.swp_destroy(ctx)


# r_cut and the skin move the cell grid, and with it the arrays of the list build
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_a_new_cell_grid_on_a_live_state(orc, precision):
    from paper_1912_08569_gb300 import _abi as A

    wl = _wl(4000, 0.4)
    s = make_gpu(wl, precision)
    s.run(20, 0.001, 0.1, 1.0)
    for rcut, skin in ((2.0, 0.3), (1.5, 0.3), (1.5, 0.6), (1.3, 0.5)):  # (more cells than at first need a larger workspace)
        wl["pairs"] = inputs.swap_pairs(lambda3=1.0, rcut=rcut)
        for (ti, tj), p in wl["pairs"].items():
            A.swp_set_pair(s.ctx, ti, tj, p["kind"], p["eps"], p["sigma"], p["n"], p.get("rcut", 0.0),
                           p.get("lambda3", 0.0), p.get("shift", 0), p.get("rbond", 0.0))
        s.skin = skin
        A.swp_set_nlist(s.ctx, skin, s.max_nn)
        s.run(5, 0.001, 0.1, 1.0)
        wl["x"] = s.state()[0]
        _check(orc, wl, precision, s)


def test_a_velocity_that_is_no_number_leaves_the_others_lists_alone():
    """Device arrays are not looked through: one NaN velocity, a system dilute enough
    that its particle meets nobody, and the list builds the others ask for."""
    import torch

    n = 2000
    wl = _wl(n, 0.02, seed=9)
    wl["v"] = inputs.maxwell_velocities(n, 4.0, 1.0, seed=8)
    wl["v"][700] = np.nan
    got = []
    for resident in (True, False):
        s = make_gpu(wl | dict(v=None), "fp32")
        s.set_state(*(torch.from_numpy(wl[k]).cuda() for k in ("x", "v", "types")))
        s.set_resident(resident)
        s.run(60, 0.005, 0.0, 0.0)
        th = s.thermo()
        assert th["resident_steps"] == (60 if resident else 0)
        got.append((th["n_rebuilds"], *s.state()))
    assert got[0][0] == got[1][0] > 2
    for p, q in zip(got[0][1:], got[1][1:]):
        assert np.array_equal(p, q, equal_nan=p.dtype.kind == "f")


def test_a_halo_that_does_not_fit_costs_little():
    """r_cut = 3.3: a block's second halo shell has more particles than the halo's table
    has places.  The two-barrier path takes over, and finding that out takes no longer
    than the steps themselves (bound: three times the run without the attempt)."""
    import torch

    wl = _wl(50_000, 0.4, n=10, rcut=3.3)
    got, ms = [], []
    for resident in (False, True):
        s = make_gpu(wl, "fp32")
        s.set_resident(resident)
        s.run(5, 0.001, 0.05, 1.0)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(s.stream)
        s.run(30, 0.001, 0.05, 1.0)
        e1.record(s.stream)
        torch.cuda.synchronize()
        ms.append(e0.elapsed_time(e1))
        assert s.thermo()["resident_steps"] == 0
        got.append(s.state())
    for p, q in zip(*got):
        assert np.array_equal(p, q)
    assert ms[1] < 3.0 * ms[0], ms


# a few large particles with rows of 180 entries (the resident step takes rows of up
# to 255) and of 420 (the resident build has to turn them down before it sorts by them)
@pytest.mark.parametrize("big", [1, 9])
@pytest.mark.parametrize("rcut", [4.45, 6.0])
def test_rows_at_the_resident_limit(orc, big, rcut):
    wl = _wl(3000, 0.4)
    wl["types"] = (np.arange(3000) < big).astype(np.int32)
    wl["pairs"] = inputs.swap_pairs(lambda3=1.0, rcut=rcut)
    got = []
    for resident in (True, False):
        s = make_gpu(wl, "fp32")
        s.set_resident(resident)
        _check(orc, wl, "fp32", s)
        s.run(40, 0.001, 0.05, 1.0)
        assert s.thermo()["resident_steps"] == (40 if resident and rcut < 5.0 else 0)
        got.append(s.state())
    for p, q in zip(*got):
        assert np.array_equal(p, q)


class _At:
    """A device address inside a buffer, as the binding takes it."""

    def __init__(self, buf, offset):
        self.buf, self.offset = buf, offset

    def data_ptr(self):
        return self.buf.data_ptr() + self.offset


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_unaligned_device_arrays(precision):
    import torch
    from paper_1912_08569_gb300 import _abi as A

    wl = _wl(1000, 0.3)
    n = wl["n"]

    def at4(a):  # the same bytes four bytes off an 8-byte boundary
        raw = torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).reshape(-1)).cuda()
        buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
        buf[4:4 + raw.numel()] = raw
        return _At(buf, 4)

    got = []
    for shift in (False, True):
        s = make_gpu(wl, precision)
        if shift:
            A.swp_set_state(s.ctx, at4(wl["x"]), at4(wl["v"]), at4(wl["types"].astype(np.int32)), None, None, where=A.SWP_DEVICE)
        s.run(20, 0.001, 0.1, 1.0)
        if shift:
            bufs = [torch.zeros(24 * n + 16, dtype=torch.uint8, device="cuda") for _ in range(3)]
            A.swp_read_forces(s.ctx, _At(bufs[0], 4), where=A.SWP_DEVICE)
            A.swp_read_state(s.ctx, _At(bufs[1], 4), _At(bufs[2], 4), None, where=A.SWP_DEVICE)
            got.append([b[4:4 + 24 * n].cpu().numpy().view(np.float64).reshape(n, 3) for b in bufs])
        else:
            x, v, _ = s.state()
            got.append([s.forces(), x, v])
    for p, q in zip(*got):
        assert np.array_equal(p, q)


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_unaligned_arrays_of_the_static_call(precision):
    import torch
    from paper_1912_08569_gb300 import _abi as A

    wl = _wl(800, 0.3)
    n = wl["n"]
    s = make_gpu(wl, precision)
    x, ty = torch.from_numpy(wl["x"]).cuda(), torch.from_numpy(wl["types"].astype(np.int32)).cuda()
    f = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    A.swp_compute_forces_static(s.ctx, x, ty, f, None, 0)

    def at(t, off):
        raw = t.contiguous().view(torch.uint8).reshape(-1)
        buf = torch.zeros(raw.numel() + 16, dtype=torch.uint8, device="cuda")
        buf[off:off + raw.numel()] = raw
        return _At(buf, off)

    out = at(torch.zeros_like(f), 4)
    A.swp_compute_forces_static(s.ctx, at(x, 4), at(ty, 2), out, None, 0)
    assert torch.equal(out.buf[4:4 + 24 * n].clone().view(torch.float64).view(n, 3), f)
    assert not out.buf[:4].any() and not out.buf[4 + 24 * n:].any()


def test_replayed_launches_are_seen():
    """Steps captured into a graph: every replay advances the state, and the next
    synchronising call reports what the replays did."""
    import torch

    wl = _wl(1500, 0.4)
    a = make_gpu(wl, "fp32")
    a.run(10, 0.001, 0.1, 1.0)
    a.run(10, 0.001, 0.1, 1.0)
    a.run(10, 0.001, 0.1, 1.0)
    st = torch.cuda.Stream()
    from paper_1912_08569_gb300 import SwapSystem
    b = SwapSystem(wl["n"], 2, wl["box"], wl["pairs"], precision="fp32", seed=wl.get("seed", 0), skin=wl["skin"], stream=st)
    b.set_state(wl["x"], wl["v"], wl["types"], wl["mass"])
    b.run(10, 0.001, 0.1, 1.0)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        b.run(10, 0.001, 0.1, 1.0, sync=False)
    with torch.cuda.stream(st):
        g.replay()
    assert b.thermo()["step"] == 20
    with torch.cuda.stream(st):
        g.replay()
    assert b.thermo()["step"] == 30
    for p, q in zip(a.state(), b.state()):
        assert np.array_equal(p, q)


def test_replays_after_a_batch_are_seen():
    """A system whose steps were captured takes part in a batch; a replay after that
    changes its state again."""
    import torch
    from paper_1912_08569_gb300 import SwapBatch

    wl = _wl(1500, 0.4)
    st = torch.cuda.Stream()
    a, b = make_gpu(wl, "fp32", stream=st), make_gpu(wl, "fp32", stream=st)
    b.run(10, 0.001, 0.1, 1.0)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        b.run(10, 0.001, 0.1, 1.0, sync=False)
    SwapBatch([a, b]).run(5, 0.001, 0.1, 1.0, sync=False)
    with torch.cuda.stream(st):
        g.replay()
    assert a.thermo()["step"] == 5
    assert b.thermo()["step"] == 25


@pytest.mark.parametrize("masses", [False, True])
def test_host_arrays_may_be_reused_when_the_call_returns(masses):
    """Pinned arrays, and work ahead on the stream."""
    import torch
    from paper_1912_08569_gb300 import _abi as A

    wl = _wl(1500, 0.4)
    s = make_gpu(wl, "fp32", stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    want = s.state()[:2]
    pinned = [torch.from_numpy(np.ascontiguousarray(wl[k])).pin_memory() for k in ("x", "v", "types", "mass")]
    with torch.cuda.stream(s.stream):
        torch.cuda._sleep(300_000_000)
    A.swp_set_state(s.ctx, pinned[0], pinned[1], pinned[2], pinned[3] if masses else None, None, where=A.SWP_HOST)
    for t in pinned:
        t.zero_()
    for p, q in zip(want, s.state()):
        assert np.array_equal(p, q)


def test_binding_another_workspace_and_stream():
    """Work that is still waiting on the stream bound before changes nothing of
    what the calls on the new binding report."""
    import torch
    from paper_1912_08569_gb300 import _abi as A

    wl = _wl(1500, 0.4)
    a = make_gpu(wl, "fp32")
    a.run(30, 0.001, 0.1, 1.0)
    s = make_gpu(wl, "fp32", stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    with torch.cuda.stream(s.stream):
        torch.cuda._sleep(1_000_000_000)  # about half a second
    s.run(7, 0.001, 0.1, 1.0, sync=False)
    ws, nl, st = torch.empty_like(s.workspace), torch.empty_like(s.nlist_buf), torch.cuda.Stream()
    A.swp_bind_workspace(s.ctx, ws.data_ptr(), ws.numel(), st.cuda_stream)
    A.swp_bind_nlist(s.ctx, nl.data_ptr(), nl.numel())
    s.set_state(wl["x"], wl["v"], wl["types"], wl["mass"])
    s.run(30, 0.001, 0.1, 1.0)
    first = s.state()
    torch.cuda.synchronize()  # the seven steps on the old binding, too
    assert s.thermo()["step"] == 30
    for p, q, r in zip(a.state(), first, s.state()):
        assert np.array_equal(p, q) and np.array_equal(p, r)


def test_destroying_a_context_is_host_work():
    """A context may go while another stream is captured and its own work still runs."""
    import torch

    wl = _wl(1500, 0.4)
    s = make_gpu(wl, "fp32", stream=torch.cuda.Stream())
    s.run(7, 0.001, 0.1, 1.0, sync=False)
    y = torch.zeros(8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        y += 1.0
        s.close()
    g.replay()
    torch.cuda.synchronize()
    assert y.tolist() == [1.0] * 8


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
@pytest.mark.parametrize("device", [False, True])
def test_positions_on_and_outside_the_faces(precision, device):
    import torch
    from paper_1912_08569_gb300 import _abi as A, SwapSystem

    L = 16.0
    below = float(np.nextafter(L, 0.0))
    edge = [0.0, -0.0, below, L, -L, 3.25 * L, -0.5, 1e-30, 2.0 ** -48, L - 2.0 ** -49, 7.5]
    x = np.array([[v, 0.5 + k, 15.5 - k] for k, v in enumerate(edge)])
    s = SwapSystem(len(x), 1, [L] * 3, {}, precision=precision)
    xs = torch.from_numpy(x).cuda() if device else x
    s.set_state(xs)
    got, _, img = s.state()
    q = np.array([round((v - np.floor(v / L) * L) * 2.0 ** 48) for v in edge], dtype=object)  # exact: L is a power of two
    im = np.array([int(np.floor(v / L)) for v in edge])
    for k in range(len(edge)):
        if q[k] >= 2 ** 52:
            q[k], im[k] = q[k] - 2 ** 52, im[k] + 1
    assert np.array_equal(got[:, 0], np.array([float(v) * 2.0 ** -48 for v in q]))
    assert np.array_equal(img[:, 0], im)
    assert np.array_equal(got[:, 1:], x[:, 1:])


# r_cut = 2.4: about 26 partners inside the cut-off, more than the derivative
# passes line up at once.  Central differences of the oracle, h = 1e-4: the
# truncation is below 1e-4 of the derivative (FP64), FP32 terms allow 1e-3.
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-4), ("fp32", 1e-3)])
def test_parameter_derivatives_of_long_rows(orc, precision, tol):
    import torch
    from paper_1912_08569_gb300 import _abi as A

    wl = _wl(1501, 0.5, n=10, rcut=2.4)
    s = make_gpu(wl, precision)
    s.compute_forces()
    dF = torch.empty((3, wl["n"], 3), dtype=torch.float64, device=s.device)
    dU = A.swp_param_grad(s.ctx, 0, 1, dF)
    h, theta = 1e-4, (1.0, 1.0, 1.0)
    x, L = wl["x"], wl["box"]
    d = x[None] - x[:, None]
    d -= L * np.round(d / L)
    r = np.sqrt((d * d).sum(-1))
    near = (wl["types"][:, None] != wl["types"][None]) & (np.abs(r - 2.0 ** 0.1) < 4 * h)
    keep = ~near.any(1)  # vh is only once differentiable where a partner crosses r_min
    for k in range(3):
        r = []
        for sg in (1, -1):
            p = {q: dict(v) for q, v in wl["pairs"].items()}
            th = list(theta)
            th[k] += sg * h
            p[(0, 1)]["lambda3"], p[(0, 1)]["eps"], p[(0, 1)]["sigma"] = th
            r.append(orc.forces(x, wl["types"], 2, orc.pair_table(2, p), L, fp32=precision == "fp32"))
        fd = ((r[0]["U2"] + r[0]["U3"]) - (r[1]["U2"] + r[1]["U3"])) / (2 * h)
        assert abs(dU[k] - fd) <= tol * (abs(fd) + 1.0)
        ref = (r[0]["F"] - r[1]["F"])[keep] / (2 * h)
        assert np.linalg.norm(dF[k].cpu().numpy()[keep] - ref) <= tol * np.linalg.norm(ref)
