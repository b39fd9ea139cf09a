"""The default launch shape (rows per segment from the grid's size): the same
bits as fixed segments, at sizes on both sides of the rule's lines."""
from __future__ import annotations

import numpy as np
import pytest

from paper_1209_6548_gb300 import inputs as I

pytestmark = pytest.mark.gpu


# sizes: one row, rows short of a segment, an even wave, past one wave, and
# past two waves of the longest segments (the fixed shape)
SIZES = [(4, 2), (4, 65), (29, 3), (257, 255), (530, 513), (1030, 1021), (2053, 2049)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("nroots,dim,storage", [(4, 2, 0), (4, 2, 2), (4, 2, 3), (6, 2, 0), (4, 3, 0), (6, 3, 0)])
def test_default_rows_give_the_bits_of_fixed_rows(nx, ny, nroots, dim, storage):
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    if nx * ny * nroots ** dim > 2 ** 26 and (nroots, dim, storage) != (4, 2, 0):
        pytest.skip("large grids with the base set only")
    prob = I.Problem(name="shape", nroots=nroots, dim=dim, nx=nx, ny=ny, bc_y=I.DIFFUSE, kn=0.1, b=-0.5,
                     scheme=I.SPLIT, wall_ux=(0.0, 0.05), g=(1e-3, 0.0))
    p = L.params_from_problem(prob)
    p.storage = storage
    init = I.random_fields(prob, seed=nx + ny)
    got = []
    for rows in (0, 7, ny):
        s = L.Solver(p, h_init=init)
        if rows:
            s.set_launch(0, rows)
        s.step(3)
        got.append((s.populations(), s.info.rows_per_segment))
    assert 1 <= got[0][1] <= ny and got[1][1] == 7 and got[2][1] == ny
    assert np.isfinite(float(got[0][0].double().sum()))
    for other, _ in got[1:]:
        assert torch.equal(got[0][0], other)


@pytest.mark.parametrize("nroots,dim,storage", [(4, 2, 0), (4, 2, 1), (4, 2, 3), (6, 3, 0)])
def test_steps_overlap_safely_on_a_busy_stream_and_in_a_graph(nroots, dim, storage):
    """Each step's kernel may be scheduled while the previous one runs: many
    steps in one call, steps one call at a time between other work on the
    stream, and steps replayed from a captured graph give the same bits."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    prob = I.Problem(name="overlap", nroots=nroots, dim=dim, nx=61, ny=90, bc_y=I.DIFFUSE, kn=0.1, b=-0.5,
                     scheme=I.SPLIT, wall_ux=(0.0, 0.05))
    p = L.params_from_problem(prob)
    p.storage = storage
    init = I.random_fields(prob, seed=1)
    many = L.Solver(p, h_init=init)
    many.step(24)
    single = L.Solver(p, h_init=init)
    noise = torch.zeros(1 << 22, device="cuda")
    for k in range(24):
        if k % 3 == 0:
            noise.add_(1.0)
        single.step(1)
        if k % 5 == 0:
            single.moments()
    assert torch.equal(many.populations(), single.populations())
    if storage == 1:
        return  # the rounding key counts steps on the host: a replayed graph repeats it
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        graphed = L.Solver(p, h_init=init, stream=side)
    side.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        graphed.step(12)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert torch.equal(many.populations(), graphed.populations())


@pytest.mark.parametrize("nx,n,ny_lo,ny_hi,nroots,dim", [
    (4, 5, 2, 60, 4, 2),        # short solves only: the resident kernel
    (4, 40, 2, 300, 4, 2),      # one chain of one-row items
    (4, 150, 16, 1024, 4, 2),   # around a full chip: several chains
    (4, 100, 16, 512, 6, 2),
    (16, 40, 16, 700, 4, 3),
    (1, 300, 16, 500, 4, 2),
])
def test_batch_defaults_give_the_bits_of_fixed_rows(nx, n, ny_lo, ny_hi, nroots, dim):
    """Rows, chains and the resident kernel as the batch's contents choose
    them, through step graphs, single steps, removals and re-admissions,
    against fixed 32-row items without the resident kernel."""
    import torch
    from dataclasses import replace
    from paper_1209_6548_gb300 import lesbgk as L

    probs = [replace(p, nx=nx, nroots=nroots, dim=dim, scheme=I.SPLIT if k % 3 == 0 else I.UNSPLIT)
             for k, p in enumerate(I.batch_mix(n=n, seed=n, ny_lo=ny_lo, ny_hi=ny_hi))]
    params = [L.params_from_problem(p) for p in probs]
    got = []
    for fixed in (False, True):
        bt = L.Batch(capacity=n, nx=nx, pool_bytes=sum(L.batch_slot_bytes(p) for p in params) + (1 << 20))
        if fixed:
            bt.set_resident(False)
            bt.set_rows(32)
        slots = bt.add_many(params)
        bt.step(64 * 2 + 3)
        for k in range(0, n, 3):
            bt.remove(slots[k])
        bt.step(64)
        for k in range(0, n, 6):
            slots[k] = bt.add(params[k])
        bt.step(70)
        keep = [k for k in range(n) if k % 3 or k % 6 == 0]
        got.append([bt.populations(slots[k]) for k in keep])
        assert int(bt.check_guards().sum()) == 0
        bt.close()
    for a, b in zip(*got):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)


@pytest.mark.parametrize("nx,ny", [(4, 64), (1, 4), (2, 5), (3, 33), (4, 1024), (5, 200), (7, 65), (31, 24), (32, 128),
                                   (16, 131), (33, 20), (4, 3)])
@pytest.mark.parametrize("nroots,dim", [(4, 2), (6, 2), (4, 3)])
def test_small_solves_stay_on_chip_with_the_bits_of_single_steps(nx, ny, nroots, dim):
    """Calls of several steps on few columns keep the state in a cluster's
    shared memory; single-step calls and fixed rows take the marching kernel.
    Band edges, ghost rows (periodic, wall), spare lanes, columns that do not
    divide a warp, and sizes just outside the range."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    for bc_y, scheme, spec in ((I.DIFFUSE, I.UNSPLIT, 0.0), (I.DIFFUSE, I.SPLIT, 0.4), (I.PERIODIC, I.SPLIT, 0.0),
                               (I.PERIODIC, I.UNSPLIT, 0.0)):
        prob = I.Problem(name="small", nroots=nroots, dim=dim, nx=nx, ny=ny, bc_y=bc_y, kn=0.1, b=-0.5, scheme=scheme,
                         wall_ux=(-0.05, 0.05), wall_T=(0.97, 1.02), wall_specular=spec, g=(1e-3, 2e-4))
        p = L.params_from_problem(prob)
        init = I.random_fields(prob, amp_u=0.02, amp_T=0.02, amp_rho=0.02, seed=ny)
        got = []
        for mode in ("calls", "single", "rows"):
            s = L.Solver(p, h_init=init)
            if mode == "rows":
                s.set_launch(0, 3)
            if mode == "single":
                for _ in range(11):
                    s.step(1)
            else:
                for n in (3, 1, 5, 2):
                    s.step(n)
            assert s.info.steps_done == 11
            got.append(s.populations())
        assert bool(torch.isfinite(got[0]).all())
        assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])


def test_small_solves_run_past_one_launch_of_steps():
    """More steps than one launch takes (4096), on a stream of its own."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    p = L.params_from_problem(I.couette_4x64())
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        a, b = L.Solver(p, stream=side), L.Solver(p, stream=side)
        a.step(4096 + 100)
        b.set_launch(0, 4)
        b.step(4096 + 100)
        same = torch.equal(a.populations(), b.populations())
    side.synchronize()
    assert same


@pytest.mark.parametrize("capacity,count,ny_hi", [(2, 2, 90), (70, 70, 700), (40, 23, 65), (300, 300, 1024)])
def test_fields_of_many_admissions_arrive_whole(capacity, count, ny_hi):
    """Fields staged in pieces, in slot and class order of their own, larger
    than the staging area (which grows with the capacity), absent for some:
    the populations of single admissions, bitwise."""
    import torch
    from dataclasses import replace
    from paper_1209_6548_gb300 import lesbgk as L

    probs = [replace(p, nroots=6 if k % 4 == 1 else 4, dim=3 if k % 4 == 2 else 2)
             for k, p in enumerate(I.batch_mix(n=count, seed=count, ny_lo=16, ny_hi=ny_hi))]
    if capacity == 2:
        probs[0] = replace(probs[0], ny=1500)  # 192 kB of fields: more than two slots' staging
    params = [L.params_from_problem(p) for p in probs]
    for k, p in enumerate(params):
        p.storage = (0, 1, 2)[k % 3]
    fields = [None if k % 5 == 3 else I.random_fields(p, seed=k) for k, p in enumerate(probs)]
    pool = sum(L.batch_slot_bytes(p) for p in params)
    many = L.Batch(capacity=capacity, nx=4, pool_bytes=pool)
    slots = many.add_many(params, fields)
    one = L.Batch(capacity=capacity, nx=4, pool_bytes=pool)
    for s, p, f in zip(slots, params, fields):
        assert torch.equal(many.populations(s), one.populations(one.add(p, f)))
    assert int(many.check_guards().sum()) == 0
    bad = [f.copy() if f is not None else None for f in fields]
    bad[0][3, 1, 2] = np.nan
    three = L.Batch(capacity=capacity, nx=4, pool_bytes=pool)
    with pytest.raises(L.LesbgkError) as err:
        three.add_many(params, bad)
    assert "node 6 " in str(err.value)
    assert three.pool_free()[1] >= pool  # nothing was kept


@pytest.mark.parametrize("nx,ny,nroots", [(4, 64, 4), (4, 200, 6), (40, 50, 4)])
def test_a_whole_pass_replays_from_a_captured_graph(nx, ny, nroots):
    """Initialisation, steps (on chip for few columns, an odd number of them),
    moments and state as the nodes of one graph: each replay gives the bits of
    the same calls made directly."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    prob = I.Problem(name="pass", nroots=nroots, nx=nx, ny=ny, bc_y=I.DIFFUSE, kn=0.1, b=-0.5, scheme=I.SPLIT,
                     wall_ux=(-0.05, 0.05))
    p = L.params_from_problem(prob)
    fields = torch.from_numpy(I.random_fields(prob, amp_u=0.02, amp_T=0.02, amp_rho=0.02, seed=2)).cuda()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        direct, graphed = L.Solver(p, stream=side), L.Solver(p, stream=side)
        direct.reinit(fields)
        direct.step(9)
        want = direct.moments(), direct.populations()
    side.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        graphed.reinit(fields)
        graphed.step(9)
        got = graphed.moments(), graphed.populations()
    for _ in range(3):
        for t in got:
            t.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


class _PartOfTheDevice:
    """A stream of a green context that holds the fewest SMs the driver gives."""

    def __enter__(self):
        import ctypes as C
        import torch

        class Resource(C.Structure):  # CUdevResource: type, padding, SM counts
            _fields_ = [("type", C.c_int), ("pad", C.c_ubyte * 92), ("sms", C.c_uint), ("rest", C.c_ubyte * 44)]

        torch.zeros(1, device="cuda")
        self.cu = C.CDLL("libcuda.so.1")

        def call(name, *args):
            rc = getattr(self.cu, name)(*args)
            if rc:
                pytest.skip(f"{name}: error {rc}")

        whole, part, rest = Resource(), Resource(), Resource()
        call("cuDeviceGetDevResource", C.c_int(torch.cuda.current_device()), C.byref(whole), C.c_int(1))
        groups = C.c_uint(1)
        call("cuDevSmResourceSplitByCount", C.byref(part), C.byref(groups), C.byref(whole), C.byref(rest), C.c_uint(0),
             C.c_uint(8))
        desc, self.green, self.handle = C.c_void_p(), C.c_void_p(), C.c_void_p()
        call("cuDevResourceGenerateDesc", C.byref(desc), C.byref(part), C.c_uint(1))
        call("cuGreenCtxCreate", C.byref(self.green), desc, C.c_int(torch.cuda.current_device()), C.c_uint(1))
        call("cuGreenCtxStreamCreate", C.byref(self.handle), self.green, C.c_uint(1), C.c_int(0))
        self.sms, self.all_sms = part.sms, whole.sms
        return self

    def __exit__(self, *exc):
        self.cu.cuStreamSynchronize(self.handle)
        self.cu.cuStreamDestroy_v2(self.handle)
        self.cu.cuGreenCtxDestroy(self.green)


def test_small_solves_march_on_a_part_of_the_device():
    """The cluster of an on-chip solve is chosen for the whole device; on a
    stream that has a part of it the call takes one launch per step, with the
    same bits."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    p = L.params_from_problem(I.Problem(name="part", nx=4, ny=1000, bc_y=I.DIFFUSE, kn=0.1, b=-0.5, wall_ux=(0.0, 0.05)))
    whole = L.Solver(p)
    whole.step(9)
    torch.cuda.synchronize()
    assert whole.on_chip_ctas(9) == 16
    with _PartOfTheDevice() as part:
        assert 0 < part.sms < part.all_sms
        s = L.Solver(p)
        torch.cuda.synchronize()
        s.stream = torch.cuda.ExternalStream(part.handle.value)
        assert s.on_chip_ctas(9) == 0
        s.step(9)
        got = s.populations()
        s.stream.synchronize()
        assert s.info.steps_done == 9 and torch.equal(got, whole.populations())


def test_which_calls_keep_the_solve_on_chip():
    """Three or more steps of FP32 solves on up to 32 periodic columns, at one
    node per thread of at most 16 blocks, with steady walls and no rows set."""
    from paper_1209_6548_gb300 import lesbgk as L

    def ctas(n=3, rows=0, storage=0, **kw):
        p = L.params_from_problem(I.Problem(name="path", **{**dict(nx=4, ny=64, bc_y=I.DIFFUSE, kn=0.1, b=-0.5), **kw}))
        p.storage = storage
        s = L.Solver(p)
        if rows:
            s.set_launch(0, rows)
        return s.on_chip_ctas(n)

    assert ctas() > 0 and ctas(ny=1000) == 16 and ctas(nx=32, ny=128) == 16
    assert ctas(nroots=6) > 0 and ctas(dim=3) > 0 and ctas(bc_y=I.PERIODIC) > 0 and ctas(nx=1, ny=4) == 1
    assert ctas(n=2) == 0 and ctas(rows=3) == 0 and ctas(nx=33, ny=20) == 0 and ctas(ny=3) == 0
    assert ctas(storage=1) == 0 and ctas(storage=3) == 0 and ctas(nroots=6, dim=3) == 0
    assert ctas(bc_x=I.DIFFUSE) == 0 and ctas(wall_T_amp=0.02, wall_T_freq=0.5) == 0 and ctas(nx=32, ny=4096) == 0


def _batch(probs, storage=(0,), **kw):
    from paper_1209_6548_gb300 import lesbgk as L

    params = [L.params_from_problem(p) for p in probs]
    for k, p in enumerate(params):
        if p.wall_specular == 0.0:
            p.storage = storage[k % len(storage)]
    bt = L.Batch(capacity=len(params), nx=probs[0].nx, pool_bytes=sum(L.batch_slot_bytes(p) for p in params) + (1 << 20))
    for name, value in kw.items():
        getattr(bt, name)(value)
    return bt, params, bt.add_many(params)


def test_which_work_items_a_batch_makes():
    """One chain of short items for a small batch, four once the items fill the
    chip, the resident kernel for short solves alone; reads in 32-row items."""
    bt, params, slots = _batch(I.batch_mix(n=150, seed=150, ny_lo=16, ny_hi=1024))
    for s, p in zip(slots, params):
        w = bt.work(s)
        assert 1 <= w["step_rows"] <= min(64, p.ny) and w["chains"] == 4 and w["read_rows"] == min(32, p.ny)
    bt, params, slots = _batch(I.batch_mix(n=40, seed=40, ny_lo=2, ny_hi=300))
    assert all(bt.work(s)["chains"] == 1 and bt.work(s)["step_rows"] == 1 for s in slots)
    bt, params, slots = _batch(I.batch_mix(n=20, seed=20, ny_lo=2, ny_hi=64))
    for s, p in zip(slots, params):
        assert bt.work(s) == {"step_rows": 0, "chains": 0, "read_rows": min(32, p.ny)}
    bt.set_resident(False)
    bt.set_rows(5)
    assert all(bt.work(s)["step_rows"] == min(5, p.ny) == bt.work(s)["read_rows"] for s, p in zip(slots, params))


@pytest.mark.parametrize("storage", [(1,), (0, 2)])
def test_four_chains_keep_each_slots_clock(storage):
    """16-bit rounding keys and heated walls follow a slot's own step count:
    four chains against fixed rows, through graphs, single steps, removals and
    re-admissions at another parity."""
    import torch
    from dataclasses import replace

    probs = [replace(p, wall_T_amp=0.02, wall_T_freq=0.5) if k % 2 else p
             for k, p in enumerate(I.batch_mix(n=300, seed=7, ny_lo=16, ny_hi=1024))]
    got = []
    for kw in ({}, {"set_resident": False, "set_rows": 32}):
        bt, params, slots = _batch(probs, storage, **kw)
        if not kw:
            assert max(bt.work(s)["chains"] for s in slots) == 4
        bt.step(64 + 3)
        for k in range(0, 300, 5):
            bt.remove(slots[k])
        bt.step(1)
        for k in range(0, 300, 10):
            slots[k] = bt.add(params[k])
        bt.step(64 + 5)
        got.append([bt.populations(slots[k]) for k in range(300) if k % 5 or k % 10 == 0])
        bt.close()
    for a, b in zip(*got):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)


@pytest.mark.parametrize("storage", [0, 1])
def test_steps_that_fill_the_chip_overlap_safely_with_other_work(storage):
    """On a grid whose steps fill the chip even single-step calls overlap what
    runs before them: foreign kernels, moments and state reads between."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    prob = I.Problem(name="fills", nx=1030, ny=1021, bc_y=I.DIFFUSE, kn=0.1, b=-0.5, scheme=I.SPLIT,
                     wall_ux=(0.0, 0.05))
    p = L.params_from_problem(prob)
    p.storage = storage
    init = I.random_fields(prob, seed=1)
    many = L.Solver(p, h_init=init)
    many.step(18)
    blocks = 37 * -(-1021 // many.info.rows_per_segment) / 4  # 28 columns per warp, four warps per block
    assert blocks >= 3.5 * torch.cuda.get_device_properties(0).multi_processor_count
    single = L.Solver(p, h_init=init)
    noise = torch.zeros(1 << 22, device="cuda")
    for k in range(18):
        if k % 3 == 0:
            noise.add_(1.0)
        single.step(1)
        if k % 5 == 0:
            single.moments()
        if k % 7 == 0:
            single.populations()
    assert torch.equal(many.populations(), single.populations())


def test_reads_of_resident_solves_go_by_the_callers_rows():
    """Rows set by the caller hold for the reads of solves that the resident
    kernel steps, whatever rows their class had before, and the reads give the
    same bits."""
    import numpy as np
    import torch

    probs = I.batch_mix(n=24, seed=3, ny_lo=16, ny_hi=64)
    bt, params, slots = _batch(probs, set_resident=True)
    other, _, slots2 = _batch(probs, set_resident=False)
    other.set_rows(32)
    other.set_rows(4)
    other.set_resident(True)
    for x in (bt, other):
        x.set_rows(32)
    for s, t, p in zip(slots, slots2, params):
        assert bt.work(s) == other.work(t) == {"step_rows": 0, "chains": 0, "read_rows": min(32, p.ny)}
    free, _, slots3 = _batch(probs)  # the rules: items of 32 rows
    for x in (bt, other, free):
        x.step(64)
    first = [x.residuals(mass=True)[1] for x in (bt, other, free)]
    for x in (bt, other, free):
        x.step(64)
    second = [x.residuals(mass=True) for x in (bt, other, free)]
    for m, (r, m2) in zip(first[1:], second[1:]):
        assert np.array_equal(m, first[0]) and np.array_equal(r, second[0][0]) and np.array_equal(m2, second[0][1])
    outs = [[torch.empty((9, p.ny, 4), device="cuda") for p in params] for _ in range(3)]
    for x, sl, o in zip((bt, other, free), (slots, slots2, slots3), outs):
        x.moments_many(sl, o)
    for a, b, c in zip(*outs):
        assert torch.equal(a, b) and torch.equal(a, c)


@pytest.mark.parametrize("ny", [4, 5, 6, 7, 33])
def test_a_bad_field_is_found_at_its_node(ny):
    """The check of a batched solve's fields names the first bad node wherever
    it lies among the lanes of the check, and takes huge finite values."""
    from paper_1209_6548_gb300 import lesbgk as L

    prob = I.Problem(name="bad", nx=1, ny=ny, bc_y=I.DIFFUSE, kn=0.1, b=-0.5)
    p = L.params_from_problem(prob)
    bt = L.Batch(capacity=2, nx=1, pool_bytes=4 * L.batch_slot_bytes(p))
    rest = np.zeros((4, ny, 1))
    rest[0] = rest[3] = 1.0
    for field, value in ((0, 0.0), (0, -1.0), (0, np.nan), (0, np.inf), (1, np.nan), (1, -np.inf), (2, np.inf), (3, 0.0),
                         (3, np.nan), (3, np.inf)):
        for node in {0, 1, ny // 2, ny - 2, ny - 1}:
            f = rest.copy()
            f[field, node:, 0] = value
            f[2, ny - 1, 0] = np.inf  # a later one is not named
            with pytest.raises(L.LesbgkError) as err:
                bt.add(p, f)
            assert f"node {node} " in str(err.value)
    f = rest.copy()
    f[1, :, 0], f[2, :, 0] = 1.5e308, 1.5e308
    bt.remove(bt.add(p, f))  # finite, though their sum is not


@pytest.mark.parametrize("capacity,sizes", [
    (3, (40, 40, 700)),                      # three solves: straight to their buffers
    (16, (31, 32, 33, 64, 100, 255, 256)),   # staging room 16 kdoubles: staged up to 1024 of them, 8 rows of 32 columns
    (512, (159, 160, 161, 8, 1200, 700, 64)),  # staged up to 160 kB: 160 rows
])
@pytest.mark.parametrize("pinned", [False, True])
def test_large_and_pinned_fields_arrive_whole(capacity, sizes, pinned):
    """Fields on both sides of the size from which they go straight to the
    solve's own buffer, in one call, repeated: the populations of single
    admissions, bitwise."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    probs = [I.Problem(name="f", nx=32, ny=ny, nroots=6 if k % 3 == 2 else 4, bc_y=I.DIFFUSE, kn=0.1, b=-0.5)
             for k, ny in enumerate(sizes * 2)]
    if capacity == 16:
        probs = [I.Problem(name="f", nx=32, ny=ny, bc_y=I.DIFFUSE, kn=0.1, b=-0.5) for ny in (7, 8, 9, *sizes)]
    if capacity == 3:
        probs = probs[:3]
    params = [L.params_from_problem(p) for p in probs]
    fields = []
    for k, p in enumerate(probs):
        t = torch.from_numpy(I.random_fields(p, seed=k))
        fields.append((t.pin_memory() if pinned else t).numpy())
    pool = sum(L.batch_slot_bytes(p) for p in params)
    many, one = (L.Batch(capacity=capacity, nx=32, pool_bytes=pool) for _ in range(2))
    want = [one.populations(one.add(p, f)) for p, f in zip(params, fields)]
    for _ in range(2):
        slots = many.add_many(params, fields)
        for s, w in zip(slots, want):
            assert torch.equal(many.populations(s), w)
        assert int(many.check_guards().sum()) == 0
        for s in slots:
            many.remove(s)


def test_autotune_may_keep_the_rules_and_a_failed_one_changes_nothing():
    """Without candidates of the caller's the tuner keeps the batch's own rules
    where they win (they do against rows no solve here should run with), with
    the state untouched; a call that fails leaves the configuration as it was;
    set_auto returns to the rules."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    probs = I.batch_mix(n=150, seed=150, ny_lo=600, ny_hi=1024)
    bt, params, slots = _batch(probs)
    ref, _, slots2 = _batch(probs)
    bt.step(3)  # an odd parity
    rules = bt.work(slots[0]), bt.launch()
    before = [bt.populations(s) for s in slots]
    assert bt.autotune() == rules[1]["rows_per_item"]
    assert (bt.work(slots[0]), bt.launch()) == rules
    assert all(torch.equal(bt.populations(s), x) for s, x in zip(slots, before))
    for rows in ((64, 0), (64, 5000), (64, -1)):
        with pytest.raises(L.LesbgkError) as err:
            bt.autotune(rows)
        assert err.value.code == L.EINVAL and (bt.work(slots[0]), bt.launch()) == rules
    assert bt.autotune((64, 128)) in (64, 128)
    fixed = bt.work(slots[0]), bt.launch()
    assert fixed[0]["step_rows"] in (0, 64, 128) and fixed[1] != rules[1]
    with pytest.raises(L.LesbgkError):
        bt.autotune((32, 4097))
    assert (bt.work(slots[0]), bt.launch()) == fixed
    bt.set_auto()
    assert (bt.work(slots[0]), bt.launch()) == rules
    bt.step(64 + 6)
    ref.step(73)
    for s, t in zip(slots, slots2):
        assert torch.equal(bt.populations(s), ref.populations(t))
    empty = L.Batch(capacity=2, nx=4, pool_bytes=1 << 20)
    assert empty.autotune((8, 16)) in (8, 16)


@pytest.mark.parametrize("classes,chains", [(1, 4), (2, 4), (3, 2), (6, 1)])
def test_chains_are_shared_among_the_classes(classes, chains):
    """However many classes a batch holds, about eight chains step it, with the
    bits of fixed rows."""
    import torch
    from dataclasses import replace
    from paper_1209_6548_gb300 import lesbgk as L

    kinds = [(4, 2, 0), (6, 2, 0), (4, 3, 0), (4, 2, 1), (6, 2, 1), (4, 3, 2)][:classes]
    probs = [replace(p, nroots=kinds[k % classes][0], dim=kinds[k % classes][1])
             for k, p in enumerate(I.batch_mix(n=192, seed=9, ny_lo=200, ny_hi=1024))]
    got = []
    for kw in ({}, {"set_resident": False, "set_rows": 32}):
        bt, params, slots = _batch(probs, storage=[k[2] for k in kinds], **kw)
        if not kw:
            assert {bt.work(s)["chains"] for s in slots} == {chains}
        bt.step(64 + 1)
        got.append([bt.populations(s) for s in slots])
        bt.close()
    for a, b in zip(*got):
        assert bool(torch.isfinite(a).all()) and torch.equal(a, b)


@pytest.mark.parametrize("nx,ny,resident", [(1, 128, True), (1, 129, False), (2, 128, True), (2, 129, False), (4, 64, True),
                                            (4, 65, False), (8, 32, True), (8, 33, False), (32, 8, True), (32, 9, False)])
def test_which_batches_are_resident(nx, ny, resident):
    """Solves of at most 256 nodes and 128 rows go to the resident kernel by
    themselves, with the bits of the per-step kernel; one that does not keeps
    all of them from it."""
    import torch
    from dataclasses import replace

    probs = [replace(I.batch_mix(n=1, seed=1)[0], nx=nx, ny=h) for h in (ny, max(4, ny // 2), 4)]
    bt, _, slots = _batch(probs)
    ref, _, slots2 = _batch(probs, set_resident=False)
    for s in slots:
        assert (bt.work(s)["step_rows"] == 0) == resident
    for x in (bt, ref):
        x.step(64 + 3)
    for s, t in zip(slots, slots2):
        assert torch.equal(bt.populations(s), ref.populations(t))


@pytest.mark.parametrize("nx,n,ny_hi", [(1, 70, 300), (2, 40, 200), (4, 60, 500), (8, 30, 200), (16, 24, 150), (32, 20, 120)])
@pytest.mark.parametrize("nroots,dim,storage,amp", [(4, 2, 0, 0.0), (4, 2, 1, 0.0), (4, 2, 0, 0.02), (4, 2, 2, 0.02),
                                                    (6, 2, 0, 0.0), (4, 3, 1, 0.0)])
def test_any_rows_of_the_callers_give_the_bits_of_the_solve_alone(nx, n, ny_hi, nroots, dim, storage, amp):
    """Rows from one to more than a solve has, which choose kernels, chains and
    how steps follow one another: through graphs and single steps, every slot
    as its solve alone, value for value and, where a solve diverges (some of the
    shortest do), NaN for NaN."""
    import torch
    from dataclasses import replace
    from paper_1209_6548_gb300 import lesbgk as L

    probs = [replace(p, nx=nx, nroots=nroots, dim=dim, scheme=I.SPLIT if k % 3 == 0 else I.UNSPLIT, wall_T_amp=amp,
                     wall_T_freq=0.5 if amp else 0.0)
             for k, p in enumerate(I.batch_mix(n=n, seed=n, ny_lo=3, ny_hi=ny_hi))]
    bt, params, slots = _batch(probs, storage=(storage,), set_resident=False)
    done = 0
    for rows in (1, 2, 7, 16, 32, 64, 600):
        bt.set_rows(rows)
        bt.step(64 + 2)
        done += 66
    for k in range(0, n, 7):
        ref = L.Solver(params[k])
        ref.step(done)
        got, want = bt.populations(slots[k]), ref.populations()
        assert bool(((got == want) | (torch.isnan(got) & torch.isnan(want))).all()), (k, params[k].ny)


@pytest.mark.parametrize("nroots,dim,nx,ny", [(6, 2, 2524, 1703), (6, 3, 2048, 1024), (4, 3, 2433, 1730)])
def test_grids_just_past_a_wave_keep_long_segments(nroots, dim, nx, ny):
    """Grids whose long segments take little more than whole waves keep them
    (many short ones took 1 to 14% longer), with the bits of other rows."""
    import torch
    from paper_1209_6548_gb300 import lesbgk as L

    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the waves are those of 152 SMs")
    prob = I.Problem(name="wave", nroots=nroots, dim=dim, nx=nx, ny=ny, bc_y=I.PERIODIC, kn=0.1, b=-0.5, scheme=I.SPLIT)
    p = L.params_from_problem(prob)
    s = L.Solver(p, h_init=I.random_fields(prob, seed=1))
    assert s.info.rows_per_segment >= 64
    start = s.populations()
    s.step(2)
    got = s.populations()
    s.set_populations(start, 0)
    s.set_launch(0, 32)
    s.step(2)
    assert torch.equal(s.populations(), got)
