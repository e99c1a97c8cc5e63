"""Schedules left in host memory, and the copy of logits, against the calls they stand in for."""
import ctypes as C
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def _step(n_mb, tokens, E=12, K=3, D=5):
    from paper_2608_07964_b200 import binding as B
    step = B.MoEStep(3, E, K, 1, 64, 64, D, [e % D for e in range(E)], n_mb * tokens)
    g = torch.Generator(device="cuda").manual_seed(7)
    step.logits.normal_(generator=g)
    step.x.normal_(generator=g)
    w = [torch.empty(s, dtype=torch.bfloat16, device="cuda").normal_(0, 0.05, generator=g) for s in ((3, E + 1, 64, 64),) * 3]
    step.bind_weights(*w)
    return B, step


def _copy(step, dst, src):
    step.copier(dst)[0](src)


@pytest.mark.parametrize("n_mb,m,policy", [(1, 1, 0), (4, 3, 0), (11, 8, 0), (16, 12, 0), (16, 1, 0), (9, 2, 1), (9, 2, 2), (5, 1, 3)])
def test_a_watched_schedule_is_the_one_on_the_device(n_mb, m, policy):
    B, step = _step(n_mb, 37)
    batch = B.Batch([37 * j for j in range(n_mb + 1)], [j % 3 for j in range(n_mb)])
    step.watch_schedule(5)
    step.eb_step(batch, m, policy)
    got = step.schedule_wait(5, n_mb)
    loads = got.pop("loads")
    assert got == step.sched_result() and loads == step.mb_load[:n_mb].cpu().tolist()
    step.watch_schedule(6)
    step.eb_route(batch)
    step.eb_schedule(batch, m, policy)
    again = step.schedule_wait(6, n_mb)
    assert again.pop("loads") == loads and again == got
    # nothing is watched: the wait falls back on the device's record once the stream is idle
    step.watch_schedule(9)
    step.watch_schedule(0)
    step.eb_step(batch, m, policy)
    last = step.schedule_wait(9, n_mb)
    assert last.pop("loads") == loads and last == got


def test_a_watched_graph_marks_every_replay():
    B, step = _step(4, 16)
    batch = B.Batch([0, 16, 32, 48, 64], [0, 1, 2, 0])
    step.eb_step(batch, 3)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    step.watch_schedule(3)
    with torch.cuda.graph(graph):
        step.eb_step(batch, 3)
    for seed in range(4):
        step.logits.normal_(generator=torch.Generator(device="cuda").manual_seed(seed))
        step.watch_schedule(3)
        step.watch_schedule(0)
        graph.replay()
        got = step.schedule_wait(3, 4)
        assert got.pop("loads") == step.mb_load[:4].cpu().tolist() and got == step.sched_result()


def test_a_schedule_is_waited_for_from_any_stream():
    """The stream that asks is idle while the schedule is still behind other work on the one that makes it."""
    B, step = _step(4, 16)
    batch = B.Batch([0, 16, 32, 48, 64], [0, 1, 2, 0])
    step.eb_step(batch, 3)
    before = step.sched_result(), step.mb_load[:4].cpu().tolist()
    busy = torch.randn(8192, 8192, device="cuda")
    for alone in (False, True):   # a whole step, eb_schedule alone
        step.logits.normal_(generator=torch.Generator(device="cuda").manual_seed(11 + alone))
        launching, asking = torch.cuda.Stream(), torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(launching):
            for _ in range(10):
                busy @ busy
            step.watch_schedule(21 + alone)
            if alone:
                step.eb_route(batch)
                step.eb_schedule(batch, 3)
            else:
                step.eb_step(batch, 3)
            step.watch_schedule(0)
        with torch.cuda.stream(asking):
            got = step.schedule_wait(21 + alone, 4)
        loads = got.pop("loads")
        torch.cuda.synchronize()
        now = step.sched_result(), step.mb_load[:4].cpu().tolist()
        assert (got, loads) == now and now[1] != before[1]
        before = now


@pytest.mark.parametrize("same", [True, False])
def test_replays_in_a_row_give_the_last_ones_schedule(same):
    """Steps replayed without waiting for the ones before, of one graph and of two."""
    from paper_2608_07964_b200 import driver
    B, step = _step(4, 16)
    graphs = driver.StepGraphs(step, [0, 16, 32, 48, 64])
    layers = [[0, 1, 2, 0], [0, 1, 2, 0] if same else [1, 1, 2, 0]]
    for lay in layers:
        ticket = graphs.run(lay, 15, 15, 3, 0)
        step.schedule_wait(ticket, 4)
    busy = torch.randn(8192, 8192, device="cuda")
    for trial in range(4):
        other = torch.randn(step.logits.shape, device="cuda", generator=torch.Generator(device="cuda").manual_seed(trial))
        torch.cuda.synchronize()
        for _ in range(4):
            busy @ busy
        first = graphs.run(layers[0], 15, 15, 3, 0)
        step.logits.copy_(other)
        for _ in range(4):
            busy @ busy
        last = graphs.run(layers[1], 15, 15, 3, 0)
        got = step.schedule_wait(last, 4)
        loads = got.pop("loads")
        torch.cuda.synchronize()
        assert got == step.sched_result() and loads == step.mb_load[:4].cpu().tolist(), trial
        with pytest.raises(B.EbError):   # its record is gone
            step.schedule_wait(first, 4)
        again = graphs.run(layers[0], 15, 15, 3, 0)   # waited for: marked like any other
        assert again == graphs.graphs[(15, tuple(layers[0]), 15, 3, 0)][2]
        got = step.schedule_wait(again, 4)
        assert got.pop("loads") == loads and got == step.sched_result()


@pytest.mark.parametrize("rows,cols,lead", [(1, 1, 0), (3, 5, 1), (77, 64, 4), (1000, 8, 2), (4097, 64, 0), (31, 12, 3)])
def test_copy_equals_torch(rows, cols, lead):
    B, step = _step(1, 1)
    src = torch.randn(lead + rows * cols, device="cuda")[lead:].view(rows, cols)
    for d in (0, 1):
        buf = torch.zeros(d + rows * cols + 8, device="cuda")
        _copy(step, buf[d:d + rows * cols].view(rows, cols), src)
        assert torch.equal(buf[d:d + rows * cols].view(rows, cols), src)
        assert not buf[:d].any() and not buf[d + rows * cols:].any()
    for other in (src.double(), src.cpu(), src.t().contiguous().t(), src[:1].expand(rows, cols)):   # the general way
        dst = torch.zeros(rows, cols, device="cuda")
        _copy(step, dst, other)
        assert torch.equal(dst, other.to(dst).contiguous())
    one = torch.arange(rows * cols + 1, device="cuda", dtype=torch.float32)
    _copy(step, one[1:].view(rows, cols), one[1:].view(rows, cols))   # onto itself
    assert torch.equal(one, torch.arange(rows * cols + 1, device="cuda", dtype=torch.float32))


def test_copy_does_what_autograd_and_views_ask_of_copy_():
    """Where copy_ refuses, counts a version, resolves a view or carries a tangent, so does the copy."""
    import torch.autograd.forward_ad as fwAD
    B, step = _step(1, 1)
    src = torch.randn(5, 7, device="cuda")
    leaf = torch.zeros(5, 7, device="cuda", requires_grad=True)
    with pytest.raises(RuntimeError, match="leaf"):
        _copy(step, leaf, src)
    assert not leaf.any()
    base = torch.zeros(9, 7, device="cuda", requires_grad=True)
    saved = torch.zeros(9, 7, device="cuda")
    out = (base * saved).sum()
    _copy(step, saved[2:7], src)   # what the backward pass would read is no longer what it was
    with pytest.raises(RuntimeError, match="modified by an inplace operation"):
        out.backward()
    with torch.inference_mode():
        frozen = torch.zeros(5, 7, device="cuda")
    with pytest.raises(RuntimeError, match="[Ii]nference"):
        _copy(step, frozen, src)
    z = torch.randn(5, 7, device="cuda", dtype=torch.complex64)
    for dst, other in ((torch.ones(5, 7, device="cuda"), torch._efficientzerotensor((5, 7), device="cuda")),
                       (torch.zeros_like(z), z.conj()), (torch.zeros_like(z).conj(), z), (torch.zeros(5, 7, device="cuda"), torch._neg_view(src)),
                       (torch._neg_view(torch.zeros(5, 7, device="cuda")), src)):
        _copy(step, dst, other)
        assert torch.equal(dst.resolve_conj().resolve_neg(), (other * 1).resolve_conj().resolve_neg())
    with fwAD.dual_level():
        dst = torch.zeros(5, 7, device="cuda")
        _copy(step, dst, fwAD.make_dual(src, torch.full_like(src, 2)))
        assert torch.equal(fwAD.unpack_dual(dst).tangent, torch.full_like(src, 2))

    def doubled(x):
        dst = torch.zeros_like(x)
        _copy(step, dst, x)
        return 2 * dst
    assert torch.equal(torch.func.vmap(doubled)(src), 2 * src)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.uint8, torch.int64])
@pytest.mark.parametrize("count,lead", [(1, 0), (1, 1), (7, 3), (255, 1), (4097, 2), (300001, 5)])
def test_copies_of_types_that_are_no_multiple_of_four_bytes(dtype, count, lead):
    B, step = _step(1, 1)
    src = torch.randint(0, 100, (lead + count,), device="cuda").to(dtype)[lead:]
    for d in (0, 1, 2):
        buf = torch.zeros(d + count + 8, device="cuda", dtype=dtype)
        _copy(step, buf[d:d + count], src)
        assert torch.equal(buf[d:d + count], src) and not buf[:d].any() and not buf[d + count:].any()


def test_a_copier_fills_the_rows_it_was_made_for():
    B, step = _step(4, 16)
    step.logits.zero_()
    fill = step.copier(step.logits, [0, 5, 5, 33, 64])
    want = torch.zeros_like(step.logits)
    for i, (a, b) in enumerate(((0, 5), (5, 5), (5, 33), (33, 64))):
        src = torch.full((b - a, step.E), float(i + 1), device="cuda")
        fill[i](src)
        want[a:b] = src
        assert torch.equal(step.logits, want)
    with pytest.raises(RuntimeError):   # as copy_ does: neither the shape nor broadcast to it
        fill[0](torch.zeros(4, step.E, device="cuda"))
    fill[3](torch.arange(step.E, device="cuda", dtype=torch.float64))
    want[33:] = torch.arange(step.E, device="cuda")
    assert torch.equal(step.logits, want)


def _record(step, ticket, n_mb):
    """What eb_schedule_wait gives when the device's buffers that it may fall back on hold something else: the record that the
    kernels left in host memory, or -7 everywhere."""
    from paper_2608_07964_b200 import binding as B
    poison = torch.full((1024,), -7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    h, ld, code = B.EbSchedResult(), (C.c_int32 * (16 * step.D))(), []
    stream = B._stream()
    t = threading.Thread(daemon=True, target=lambda: code.append(step.lib.eb_schedule_wait(
        step.ctx, stream, ticket, n_mb, poison.data_ptr(), poison.data_ptr(), C.addressof(h), C.addressof(ld))))
    t.start()
    t.join(20)
    assert code == [0], "the mark never came"
    return B._sched_dict(h, step.D), [list(ld[j * step.D:(j + 1) * step.D]) for j in range(n_mb)]


@pytest.mark.parametrize("how", ["step", "schedule", "graph"])
@pytest.mark.parametrize("n_mb,tokens,m,policy", [(1, 1, 1, 0), (4, 37, 3, 0), (11, 8, 8, 0), (16, 5, 12, 0), (16, 5, 1, 0), (14, 9, 2, 0), (9, 33, 2, 1),
                                                  (5, 70, 1, 3), (3, 0, 2, 0), (16, 400, 6, 0)])   # one block, several, no tokens, large grids
def test_the_record_is_what_the_kernels_left_in_host_memory(how, n_mb, tokens, m, policy):
    B, step = _step(n_mb, max(tokens, 1))
    batch = B.Batch([tokens * j for j in range(n_mb + 1)], [j % 3 for j in range(n_mb)])
    everything = (1 << n_mb) - 1
    graph = torch.cuda.CUDAGraph()
    step.eb_step(batch, m, policy)
    torch.cuda.synchronize()
    if how == "graph":
        step.watch_schedule(40)
        with torch.cuda.graph(graph):
            step.eb_step(batch, m, policy)
        step.watch_schedule(0)
    for trial in range(3):
        step.logits.normal_(generator=torch.Generator(device="cuda").manual_seed(trial))
        ticket = 40 if how == "graph" else 41 + trial
        step.watch_schedule(ticket)
        route = everything if trial != 1 else everything >> 1   # the last micro-batch keeps its routing
        if how == "graph":
            step.watch_schedule(0)
            graph.replay()
        elif how == "step":
            step.eb_step(batch, m, policy, route)
        else:
            if tokens:
                step.eb_route(batch, route)
            step.eb_schedule(batch, m, policy)
        got, loads = _record(step, ticket, n_mb)
        assert got == step.sched_result() and loads == step.mb_load[:n_mb].cpu().tolist(), trial
        assert min(min(x) for x in loads) >= 0
    # nothing is watched: the device's buffers answer, and these hold -7
    step.watch_schedule(90)
    step.watch_schedule(0)
    step.eb_step(batch, m, policy)
    got, loads = _record(step, 90, n_mb)
    assert got["n_run"] == -7 and loads == [[-7] * step.D] * n_mb


@pytest.mark.parametrize("watched", [True, False])
def test_the_loads_are_those_the_schedule_was_made_from(watched):
    B, step = _step(4, 16)
    batch = B.Batch([0, 16, 32, 48, 64], [0, 1, 2, 0])
    step.eb_step(batch, 3)
    other = torch.arange(16 * step.D, dtype=torch.int32, device="cuda").view(16, step.D) % 11
    step.watch_schedule(70)
    if not watched:
        step.watch_schedule(0)
    step.eb_schedule(batch, 3, mb_load=other)
    got = step.schedule_wait(70, 4, mb_load=other)
    assert got.pop("loads") == other[:4].cpu().tolist() and got == step.sched_result()
