"""The library's host side on a stand-in runtime (tests/fake_cudart.c): which buffers its launches
and captured graphs point to, and what it does when device memory runs out."""
import pytest

from fakert import run


@pytest.mark.parametrize("side,calls", [
    # the workspace grows through an FP32 cycle
    (128, "cycle(9, 0) cycle(16, 1) cycle(9, 0) cycle(5, 0) cycle(9, 0)"),
    # through a solve in two lanes, which takes other sweeps
    (128, "cycle(5, 0) solve(32) cycle(5, 0) cycle(12, 0) cycle(5, 0) solve(32)"),
    # through a server that gets the hierarchy after a solve
    (512, "cycle(1, 0) serve(3) cycle(1, 0) cycle(3, 0)"),
])
def test_graphs_keep_their_buffers(side, calls):
    """One FP64 hierarchy used at changing widths: no launch and no replayed graph points to
    memory that was freed."""
    out = run("""
F = fake()
F.fake_times(1e4, -1.0)  # each timed candidate beats those before it: the row-block forms win
h = Hier([%d, %d, 32, 16], overlap=1, fgmres_m=2)
for c in %r.replace(") ", ");").split(";"):
    h.ok(eval("h." + c))
    assert F.fake_dead() == 0, (c, F.fake_dead_what())
assert "k_ring" in F.fake_captured().decode()
print("ok")
""" % (side, side // 4 if side > 256 else 64, calls))
    assert "ok" in out


def test_form6_entry_keeps_graph_buffers():
    """amg_kaczmarz_form with the FP64 row-block form between two cycles of one width."""
    out = run("""
F = fake()
F.fake_times(1e4, -1.0)
h = Hier([128, 64, 32, 16])
h.ok(h.cycle(9, 0))
h.ok(h.cycle(16, 1))
h.ok(h.cycle(9, 0))
h.ok(h.lib.amg_kaczmarz_form(h.amg, 0, h.v, h.v, 12, 1, 0, 6, 0))
h.ok(h.cycle(9, 0))
assert F.fake_dead() == 0, F.fake_dead_what()
print("ok")
""")
    assert "ok" in out


def test_no_memory_for_the_row_block_forms():
    """Device memory that runs out while a wider cycle is prepared: the cycles of the widths known
    before run on buffers that exist."""
    out = run("""
F = fake()
F.fake_times(1e4, -1.0)
h = Hier([128, 64, 32, 16])
h.ok(h.cycle(9, 0))
h.ok(h.cycle(16, 1))
n = 16 * (128 * 128 // 2 // 2)
F.fake_fail(n, n * 16, 0, 1)  # what inner products of the ring passes of 1 to 16 would take on level 0
rc = h.cycle(12, 0)
F.fake_fail(1, 0, 0, 0)
assert rc in (0, h.W.WL_OOM), rc
h.ok(h.cycle(9, 0))
assert F.fake_dead() == 0, F.fake_dead_what()
print("ok")
""")
    assert "ok" in out


@pytest.mark.parametrize("order,prec,sides", [
    (0, 0, [256, 128, 64, 32, 16]), (0, 1, [128, 64, 32, 16, 8]), (1, 0, [128, 64, 32, 16]),
    (1, 1, [256, 128, 64, 32, 16]), (1, 2, [128, 64, 32, 16])])
def test_what_a_cycle_computes_does_not_hang_on_timings(order, prec, sides):
    """Whatever the tuner measures, the kernels that a cycle captures are the same but for those
    that agree bit for bit: one family of forms 0 to 3, and k_kacz_rows with any chunks."""
    out = run("""
F = fake()
def captured(start, step, nrhs):
    F.fake_times(start, step)
    h = Hier(%r, kacz_order=%d, precision=%d, fgmres_m=1)
    h.ok(h.cycle(nrhs, %d))
    out = []
    for n in F.fake_captured().decode().split():
        old = "k_kacz" in n and "k_kacz_r" not in n
        k = "old" if old else "k_kacz_rows" if "k_kacz_rows" in n else n
        if k != "old" or not out or out[-1] != k:  # a sweep of forms 0 to 3 is one to 64 launches
            out.append(k)
    return out
for nrhs in (1, 2, 5, 9, 16, 30):
    a, b = captured(1.0, 1.0, nrhs), captured(1e4, -1.0, nrhs)
    assert a == b, (nrhs, set(a) ^ set(b))
print("ok")
""" % (sides, order, prec, prec))
    assert "ok" in out


@pytest.mark.parametrize("order,prec,sides", [(0, 0, [256, 128, 64, 32, 16]), (1, 1, [256, 128, 64, 32, 16, 8]),
                                              (0, 2, [64, 32, 16])])
def test_cycle_forms_are_reported_and_pinned(order, prec, sides):
    """amg_cycle_form names what the cycle's graph holds; those forms, pinned on a second hierarchy
    whose tuner would choose otherwise, give the same kernels; a pinned form of the other kind
    takes their place."""
    out = run("""
F = fake()
sides, prec = %r, %d
def hier():
    return Hier(sides, kacz_order=%d, precision=prec, fgmres_m=1)
def form(h, l, nrhs):
    f, p, u = C.c_int(), C.c_int(), C.c_float()
    h.ok(h.lib.amg_cycle_form(h.amg, l, nrhs, prec, C.byref(f), C.byref(p), C.byref(u)))
    return f.value, p.value
def captured(h, nrhs):
    h.ok(h.cycle(nrhs, prec))
    return F.fake_captured().decode().split()
KERNEL = {0: "k_kacz", 1: "k_kacz_coop", 2: "k_kacz_tile", 3: "k_kacz_block", 4: "k_kacz_rows", 5: "k_kacz_rings"}
for nrhs in (1, 3, 9, 12):
    F.fake_times(1.0, 1.0)
    a = hier()
    names = captured(a, nrhs)
    forms = [form(a, l, nrhs) for l in range(len(sides) - 1)]
    for l, (f, p) in enumerate(forms):
        k = KERNEL[f] if f < 6 else ("k_ring_dots", "k_ring64_cluster", "k_ring_pass")[p]
        assert any(k in n for n in names), (l, f, p, names)
    assert ("k_ring_" in " ".join(names)) == any(f == 6 and p != 1 for f, p in forms)
    F.fake_times(1e4, -1.0)  # the last candidate wins
    b = hier()
    for l, (f, p) in enumerate(forms):
        b.ok(b.lib.amg_pin_sweep_form(b.amg, l, nrhs, prec, f, p))
    assert captured(b, nrhs) == names and [form(b, l, nrhs) for l in range(len(sides) - 1)] == forms
    c = hier()  # a row-block form pinned, then an old one: the old one runs
    for l, (f, p) in enumerate(forms):
        if f >= 4:
            old = (2, 8) if f == 4 else (0, 0)
            c.ok(c.lib.amg_pin_sweep_form(c.amg, l, nrhs, prec, f, p))
            c.ok(c.lib.amg_pin_sweep_form(c.amg, l, nrhs, prec, *old))
    assert not any("k_ring" in n or "k_kacz_r" in n for n in captured(c, nrhs))
    for f, p in ((4, 3 | 1 << 8), (5, 1), (6, 3), (7, 0), (6 if prec else 5, 0)):
        assert c.lib.amg_pin_sweep_form(c.amg, 0, nrhs, prec, f, p) == c.W.WL_EINVAL, (f, p)
print("ok")
""" % (sides, prec, order))
    assert "ok" in out


def test_two_lanes_take_a_pinned_row_block_form():
    """A form pinned for the lanes' width is the second lane's too, with constants of its own."""
    out = run("""
F = fake()
h = Hier([128, 64, 32, 16], overlap=1, fgmres_m=1)
h.ok(h.lib.amg_pin_sweep_form(h.amg, 0, 16, 0, 6, 0))
h.ok(h.solve(32))
assert "k_ring_dots" in F.fake_captured().decode()  # the second lane's graph is captured last
h.ok(h.lib.amg_pin_sweep_form(h.amg, 0, 17, 0, 0, 0))
h.ok(h.solve(34))
assert "k_ring_dots" not in F.fake_captured().decode() and F.fake_dead() == 0
print("ok")
""")
    assert "ok" in out


@pytest.mark.parametrize("clusters", [4, 0])
def test_clusters_are_used_where_the_device_holds_them(clusters):
    """A device that cannot hold the kernels' clusters (a partition, say) gets the two-launch form,
    in cycles, in the setup and where a form is named."""
    out = run("""
F = fake()
F.fake_clusters(%d)
F.fake_times(1e4, -1.0)
h = Hier([128, 64, 32, 16], fgmres_m=1)
for nrhs in (1, 3, 5, 9):
    h.ok(h.cycle(nrhs, 0))
    names = F.fake_captured().decode()
    assert ("k_ring64_cluster" in names or "k_ring_pass" in names) == (%d > 0), names
    for l, param in ((1, 1), (2, 1), (0, 2)):
        rc = h.lib.amg_kaczmarz_form(h.amg, l, h.v, h.v, 1, 1, 0, 6, param)
        assert rc == (0 if %d else h.W.WL_EINVAL), (rc, l, param)
F.fake_clear()
h.ok(h.setup())
names = F.fake_launched().decode()
assert ("k_ring64_cluster" in names) == (%d > 0) and "k_ring_dots" in names
print("ok")
""" % ((clusters,) * 4))
    assert "ok" in out


@pytest.mark.parametrize("level,coarsest", [(0, 8), (1, 16), (2, 16)])  # no other buffer of that size
def test_setup_without_memory_for_the_row_block_forms(level, coarsest):
    """amg_setup does with the other sweeps on a level whose triangular inverses find no memory."""
    out = run("""
F = fake()
h = Hier([128, 64, 32, %d], fgmres_m=1)
n = h.Nl[%d] ** 2 // 2
F.fake_fail(n * 384, n * 384, 0, 1000)
F.fake_clear()
h.ok(h.setup())
names = F.fake_launched().decode()
assert "k_ring" in names and "k_kacz" in names and F.fake_dead() == 0, F.fake_dead_what()
print("ok")
""" % (coarsest, level))
    assert "ok" in out


@pytest.mark.parametrize("at", [0, 3, 8, 17])
def test_no_memory_for_a_wider_batch(at):
    """A batch whose workspace does not fit is refused with WL_OOM at whichever buffer; the widths
    before it, and a server that holds the hierarchy, go on."""
    out = run("""
F = fake()
h = Hier([128, 64, 32, 16], fgmres_m=1)
h.ok(h.cycle(9, 0))
for prec in (0, 1):
    F.fake_fail(40 * 16 * 2, 1 << 40, %d, 1)  # one of the buffers that grow
    assert h.cycle(40, prec) == h.W.WL_OOM
    assert b"failed" in h.lib.wl_last_error()
    F.fake_fail(1, 0, 0, 0)
    h.ok(h.cycle(9, prec))
    h.ok(h.cycle(4, prec))
    assert F.fake_dead() == 0, F.fake_dead_what()
h.ok(h.cycle(40, 0))
F.fake_fail(1, 1 << 40, 0, 1 << 30)  # no memory at all: refused until there is some
assert h.cycle(50, 0) == h.W.WL_OOM and h.cycle(9, 0) == h.W.WL_OOM
F.fake_fail(1, 0, 0, 0)
h.ok(h.cycle(9, 0))
assert F.fake_dead() == 0, F.fake_dead_what()
print("ok")
""" % at)
    assert "ok" in out


def test_a_wait_that_ran_out_is_reported():
    """A cycle whose sweeps gave up on a bounded wait (the flag that their kernels set) is not passed
    off as valid, by amg_cycle or amg_rho, and the next one is."""
    out = run("""
F = fake()
h = Hier([64, 32, 16], fgmres_m=1, precision=1)
rho, it = C.c_double(), C.c_int()
for call in (lambda: h.cycle(1, 1), lambda: h.lib.amg_rho(h.amg, h.v, h.v, 1, 0.5, 1, C.byref(rho), C.byref(it), None)):
    F.fake_symbol(1)
    assert call() == h.W.WL_TIMEOUT
    assert call() in (h.W.WL_OK, h.W.WL_NOT_CONVERGED)
print("ok")
""")
    assert "ok" in out


@pytest.mark.parametrize("m", [1, 2, 4, 5, 6, 7, 8, 11, 12, 32])
def test_krylov_workspace_holds_every_restart_length(m):
    """FGMRES(m) with few right-hand sides: the solver's scalars and the partial sums of its dot
    products (FP64 and double-float) lie within their buffers."""
    out = run("""
F = fake()
for Nl, params, prec in (([16, 8], {}, 0), ([512, 128, 32, 16], {}, 0),
                         ([512, 128, 32, 16], dict(precision=1, arnoldi_matvec=1, gs_arith=1), 1)):
    ms = C.c_double()
    for nrhs in (1, 7):
        h = Hier(Nl, fgmres_m=%d, max_restarts=1, **params)
        assert h.lib.amg_fgmres(h.amg, h.v, h.v, nrhs, 1e-3, None) in (0, 1)
        h.ok(h.lib.wl_time_kernel(h.amg, h.W.WL_K_GS_DOT, 0, nrhs, prec, 1, C.byref(ms)))
        assert F.fake_dead() == 0, (Nl, nrhs, F.fake_dead_what())
        h.close()
print("ok")
""" % m)
    assert "ok" in out
