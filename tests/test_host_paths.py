"""Host code of the library on a pretended CUDA runtime: order of copies and kernels, failed
calls, several devices (no GPU; host_harness.py)."""
from host_harness import run  # noqa: F401


def test_uploads_are_ordered_before_the_kernels_that_read_them(run):  # noqa: F811
    """A copy from pageable memory may still be in flight when cudaMemcpy returns, and the
    context's stream does not wait for the legacy stream: clouds of few and many points, loaded
    again on one context, with and without scanner ids, then each kind of call."""
    run(r"""
r = renderer()
for n in (1, 100, 50_000):
    xyz, rgb, sid = cloud(n, seed=n)
    for s in (sid, None):
        r.load_cloud(xyz, rgb, s)
        assert get("unordered") == 0, ("load_cloud", n)
        r.build_grid(0.5)
        assert get("unordered") == 0, ("build_grid", n)
r.render(VIEW, INTR, W, H, 2, 1.0)
assert get("unordered") == 0, "fp32 frame"
for stage in range(5):
    r.render_stage(VIEW, INTR, W, H, 2, 1.0, stage)
    out = Dev(20 * W * H)
    assert fk.lnr_render_stage(r._c, ctypes.byref(_lib.make_view(VIEW)), ctypes.byref(_lib.make_intr(INTR)), W, H, 2,
                               ctypes.c_float(1.0), stage, ctypes.c_void_p(out.data_ptr()), 1) == 0
    assert get("unordered") == 0, ("stage", stage)
r.set_precision("bf16")
r.render(VIEW, INTR, W, H, 2, 1.0)
r.calibrate(VIEW, INTR, W, H, 2, 1.0)
r.set_precision("fp8")
r.render(VIEW, INTR, W, H, 2, 1.0)
assert get("unordered") == 0, "fp8 frame"
assert get("launches") > 40
""")


def test_a_frame_that_gave_up_waiting_is_reported_to_its_own_caller(run):  # noqa: F811
    """Contexts share no error word: a frame whose kernels' bounded waits ran out fails the call
    that waits for it (also a served request), and no other context's."""
    run(r"""
for prec, kernel in (("fp32", b"k_conv_split"), ("bf16", b"k_conv_halo")):
    a, b = renderer(prec=prec), renderer(prec=prec)
    out = Dev(12 * W * H)
    fk.fk_give_up(kernel, 6)
    assert status(a.render, VIEW, INTR, W, H, 2, 1.0, out=out) == 0   # returns without waiting
    fk.fk_give_up(b"", 0)
    assert status(b.render, VIEW, INTR, W, H, 2, 1.0) == 0, prec      # another context's frame is fine
    assert status(a.render, VIEW, INTR, W, H, 2, 1.0) == -5, prec     # the next call of a that waits
    assert status(a.render, VIEW, INTR, W, H, 2, 1.0) == 0, prec
    a.serve_start(max_batch=2, slots=2)
    def served():
        res = np.empty((H, W, 3), np.float32)
        t = a.submit(VIEW, INTR, W, H, 2, 1.0)
        while True:
            try:
                if a.poll(t, res)[1] is not None:
                    return 0
            except lnr.LnrError as e:
                return e.status
    fk.fk_give_up(kernel, 6)
    assert served() == -5, prec
    fk.fk_give_up(b"", 0)
    assert served() == 0, prec
    assert status(b.render, VIEW, INTR, W, H, 2, 1.0) == 0, prec
    a.serve_stop()
    a.close(), b.close()
""")


def test_every_precision_runs_on_a_second_device(run):  # noqa: F811
    """A kernel's shared-memory allowance belongs to a device, as do an SM count and the buffers
    that a launch points to: contexts on two devices of one process, results left on the device."""
    run(r"""
for device in (0, 1, 0):
    r = renderer(device)
    for prec in ("fp32", "bf16", "fp8"):
        if prec == "fp8":
            r.calibrate(VIEW, INTR, W, H, 2, 1.0)
        r.set_precision(prec)
        for _ in range(4):                       # eager, captured, replayed
            r.render(VIEW, INTR, W, H, 2, 1.0, out=Dev(12 * W * H))
        assert get("refused") == 0, (device, prec)
        assert get("foreign") == 0, (device, prec)
        r.render(VIEW, INTR, W, H, 2, 1.0)
    r.close()
assert get("conv_split") > 0 and get("conv_halo") > 0
""")


def test_a_refused_launch_fails_the_call_that_made_it(run):  # noqa: F811
    """Whatever the call: into host or device memory, eager, captured or replayed, timed, served,
    calibration, a shard's frame.  Once launches succeed again, so do the calls, and no graph
    without the refused launch is kept."""
    run(r"""
for prec, kernel in (("fp32", b"k_conv_split"), ("bf16", b"k_conv_halo")):
    keys, rgba = Dev(8 * W * H), Dev(4 * W * H)
    for runs in range(3):                        # eager, eager, captured
        for host in (False, True):
            a = renderer(prec=prec)
            out = None if host else Dev(12 * W * H)
            for _ in range(2 * runs):            # two view blocks in turn, each with its graph
                a.render(VIEW, INTR, W, H, 2, 1.0, out=out)
            fk.fk_refuse(kernel)
            assert status(a.render, VIEW, INTR, W, H, 2, 1.0, out=out) == -4, (prec, runs, host)
            fk.fk_refuse(b"")
            for k in range(8):
                convs = get("conv_split") + get("conv_halo")
                graphs = get("graphs")
                assert status(a.render, VIEW, INTR, W, H, 2, 1.0, out=out) == 0
                if k == 0:                       # launched anew, not a graph without the launch
                    assert get("conv_split") + get("conv_halo") > convs
            assert get("graphs") > graphs
            a.close()
    a = renderer(prec=prec)
    b = renderer(prec=prec)
    fk.fk_refuse(kernel)
    a.set_timing(True)
    assert status(a.render, VIEW, INTR, W, H, 2, 1.0, out=Dev(12 * W * H)) == -4
    a.set_timing(False)
    assert status(a.shard_finish, VIEW, INTR, W, H, 2, 1.0, keys, rgba, out=Dev(12 * W * H)) == -4
    if prec == "bf16":
        assert status(a.calibrate, VIEW, INTR, W, H, 2, 1.0) == -4
    a.serve_start(max_batch=2, slots=2)
    t = a.submit(VIEW, INTR, W, H, 2, 1.0)
    def poll():
        while True:
            try:
                if a.poll(t, np.empty((H, W, 3), np.float32))[1] is not None:
                    return 0
            except lnr.LnrError as e:
                return e.status
    assert poll() == -4
    fk.fk_refuse(b"")
    t = a.submit(VIEW, INTR, W, H, 2, 1.0)
    assert poll() == 0
    a.serve_stop()
    assert status(b.render, VIEW, INTR, W, H, 2, 1.0) == 0
    a.close(), b.close()
""")


def test_a_failed_call_leaves_no_error_for_the_next(run):  # noqa: F811
    """An allocation that fails is that call's error alone: the same context's and another one's
    next calls succeed."""
    run(r"""
for prec in ("fp32", "bf16"):
    a, b = renderer(prec=prec), renderer(prec=prec)
    failed = 0
    for k in range(1, 100):
        B = 8 * k                                # every buffer has to grow
        fk.fk_fail_alloc(k)
        st = status(a.render_batch, [VIEW] * B, INTR, W, H, 2, 1.0)
        fk.fk_fail_alloc(0)
        if st == 0:
            break
        failed += 1
        assert st == -3, st
        assert status(b.render, VIEW, INTR, W, H, 2, 1.0) == 0, k
        assert status(a.render, VIEW, INTR, W, H, 2, 1.0) == 0, k
    assert failed > 10, failed
    for k in range(1, 100):
        fk.fk_fail_alloc(k)
        st = status(a.set_unet, CH, synth.unet_weights(CH, seed=1), prec)
        fk.fk_fail_alloc(0)
        if st == 0:
            break
        assert st == -3 and status(b.render, VIEW, INTR, W, H, 2, 1.0) == 0, k
        assert status(a.render, VIEW, INTR, W, H, 2, 1.0) == -2
    assert status(a.render, VIEW, INTR, W, H, 2, 1.0) == 0
    assert k > 5
    a.close(), b.close()
""")


def test_a_failed_upload_or_grid_build_leaves_no_usable_cloud(run):  # noqa: F811
    """Every allocation of a load and of a grid build fails once: what needs the cloud or the grid
    then answers LNR_E_STATE until a load and a build succeed.  Refused arguments change nothing."""
    run(r"""
frame = lambda r: status(r.render, VIEW, INTR, W, H, 2, 1.0)
r = renderer()
assert frame(r) == 0
assert status(r.build_grid_frame, 0.5, [0, 0, 0], [0, 1, 1]) == -1 and frame(r) == 0
assert status(r.build_grid, 0.0) == -1 and frame(r) == 0
assert status(r.load_cloud, np.full((1, 3), np.nan), np.zeros((1, 3))) == -1 and frame(r) == 0
failed, cells, n = 0, 4, 1000
for what in ("grid", "cloud"):
    for k in range(1, 100):
        cells, n = cells + 3, n + 5000           # every buffer has to grow
        if what == "grid":
            r.load_cloud(*cloud(n))
            r.build_grid(0.5)
            fk.fk_fail_alloc(k)
            st = status(r.build_grid_frame, 0.5, [0, 0, 0], [cells, cells, cells])
        else:
            fk.fk_fail_alloc(k)
            st = status(r.load_cloud, *cloud(n))
        fk.fk_fail_alloc(0)
        if st == 0:
            break
        failed += 1
        assert st == -3
        assert frame(r) == -2, (what, k)
        assert status(r.grid_info) == -2
        assert status(r.serve_start) == -2
        assert status(r.render_stage, VIEW, INTR, W, H, 2, 1.0, 0) == -2
        if what == "cloud":
            assert status(r.build_grid, 0.5) == -2, k
            assert status(r.build_grid_frame, 0.5, [0, 0, 0], [2, 2, 2]) == -2
            r.load_cloud(*cloud(10))
        r.build_grid(0.5)
        assert frame(r) == 0
assert failed >= 4, failed
""")


def test_outputs_are_as_large_as_the_network_writes_them(run):  # noqa: F811
    """A fourth output would be written past the frame buffers, which hold three floats a pixel:
    refused, the network before it stays.  One or two outputs fill that many floats a pixel and
    nothing after them, whichever call delivers them."""
    run(r"""
def weights(o): return synth.unet_weights(CH, seed=1, out_ch=o)
for prec in ("fp32", "bf16"):
    r = renderer(prec=prec)
    for o in (0, 4, 5):
        assert status(r.set_unet, CH, weights(max(o, 1)), prec, out_ch=o) == -1, o
    assert status(r.render, VIEW, INTR, W, H, 2, 1.0) == 0
    for o in (1, 2, 3):
        r.set_unet(CH, weights(o), prec, out_ch=o)
        P = W * H
        def check(buf, n):
            assert (buf[:n] == 0.0).all() and (buf[n:] == -7.0).all(), (prec, o)
        def fresh(views=1):
            return np.full(views * P * 3, -7.0, np.float32)
        buf = fresh()
        r.render(VIEW, INTR, W, H, 2, 1.0, out=buf)
        check(buf, o * P)
        buf = fresh(4)
        r.render_batch([VIEW] * 4, INTR, W, H, 2, 1.0, out=buf)
        check(buf, 4 * o * P)
        buf = fresh()
        assert fk.lnr_shard_finish(r._c, ctypes.byref(_lib.make_view(VIEW)), ctypes.byref(_lib.make_intr(INTR)), W, H, 2,
                                   ctypes.c_float(1.0), ctypes.c_void_p(Dev(8 * P).data_ptr()),
                                   ctypes.c_void_p(Dev(4 * P).data_ptr()), _lib._ptr(buf), 0) == 0
        check(buf, o * P)
        assert r.render(VIEW, INTR, W, H, 2, 1.0).shape == (H, W, o)
        assert r.render_batch([VIEW] * 2, INTR, W, H, 2, 1.0).shape == (2, H, W, o)
        r.serve_start(max_batch=4, slots=2)
        bufs = [fresh() for _ in range(6)]
        tickets = [r.submit_into(VIEW, INTR, W, H, 2, 1.0, b) for b in bufs]
        while tickets:
            tickets = [t for t in tickets if r.poll(t)[1] is None]
        for b in bufs:
            check(b, o * P)
        r.serve_stop()
    r.close()
""")


def test_filter_without_allocation_takes_the_same_images(run):  # noqa: F811
    """The images that lnr_filter_static takes: those whose levels 1..n, twice over and 64 floats,
    come to at most 3 Mi floats."""
    run(r"""
def levels(w, h, n):
    total = 0
    for _ in range(n):
        w, h = (w + 1) // 2, (h + 1) // 2
        total += w * h
    return total
buf = Dev(64)
p = ctypes.c_void_p(buf.data_ptr())
taken = 0
for w, h in [(64, 64), (1920, 1080), (2560, 1440), (4096, 4096)] + [(2048, h) for h in range(2289, 2313)]:
    for n in range(1, 7):
        want = 0 if 64 + 2 * levels(w, h, n) <= 3 << 20 else -1
        taken += want == 0
        assert fk.lnr_filter_static(p, w, h, n, ctypes.c_float(1.0), p, None) == want, (w, h, n)
assert 18 < taken < 150, taken
""")
