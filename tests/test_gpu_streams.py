"""Calls that read liveness results wait for a run that is still in flight, whatever stream it is ordered on.  The run is
held back by a kernel that sleeps for half a second in front of it; the results go to pinned host memory, which the test
looks at meanwhile: nothing may have been written."""
import threading
import time

import numpy as np
import pytest

from paper_2506_17506_b200 import synth
from tests import helpers as H
from tests.test_gpu_parity import _garbage_rows, _to_dev

pytestmark = pytest.mark.gpu

SLEEP_CYCLES = 1_000_000_000   # about half a second


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_17506_b200 import binding
    return binding


def _program(kind):
    if kind == "short":
        wl = synth.workload(1)
        return synth.build_program(wl.shapes[0], wl.seeds[0])
    wl = synth.workload(2)                                   # 8,000 instructions: its liveness takes an internal stream
    return synth.build_program(wl.shapes[0], wl.seeds[0])


def _call(B, gp, p, call, dev, stream):
    """Buffers for the call (allocating them may wait for the device), and a function that makes it."""
    import torch
    n = {"verify": dev.shape[0] * 16, "diagnose": p.n_instrs, "occupied": p.n_instrs * ((p.P + 31) // 32) * 4}[call]
    host = torch.full((n,), 0xA5, dtype=torch.uint8, pin_memory=True)
    scratch = torch.zeros(1 << 20, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()

    def go():
        s = B._stream_ptr(stream)
        if call == "verify":
            return B._lib.vl_verify(gp.handle, dev.data_ptr(), dev.shape[0], dev.shape[1], host.data_ptr(), s)
        if call == "diagnose":
            return B._lib.vl_diagnose(gp.handle, dev.data_ptr(), 1000, scratch.data_ptr() + 64, scratch.data_ptr(), host.data_ptr(), None, s)
        return B._lib.vl_occupied_masks(gp.handle, dev.data_ptr(), host.data_ptr(), s)

    go()                                     # the working sets of the handle are made now
    torch.cuda.synchronize()
    host.fill_(0xA5)
    return go, host.numpy(), (host, scratch)


def _check(B, oracle_mod, p, call, made, rows, held, what):
    """Makes the call in a thread of its own (it may wait on the host) while `held` sleeps."""
    import torch
    go, host, keep = made
    rc = []
    t = threading.Thread(target=lambda: rc.append(go()))
    t.start()
    time.sleep(0.15)
    early = bool((host != 0xA5).any())
    assert not held.query(), f"{what}: the sleep ended too soon"
    t.join()
    torch.cuda.synchronize()
    assert rc == [B.VL_OK], what
    assert not early, f"{what}: results were written before the liveness run had finished"
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    if call == "verify":
        assert host.tobytes() == op.verify(lv, rows).tobytes(), what
    elif call == "diagnose":
        assert np.array_equal(host, op.violations(lv, rows[0])), what
    else:
        bits = np.unpackbits(host.reshape(p.n_instrs, -1), axis=1, bitorder="little")[:, : p.P]
        assert np.array_equal(bits, op.occupied(lv, rows[0])), what


@pytest.mark.parametrize("call", ["verify", "diagnose", "occupied"])
@pytest.mark.parametrize("n", [1, 2])
def test_batch_in_flight_on_another_stream(B, oracle_mod, call, n):
    import torch
    p = _program("short")
    gps = [B.Program(p) for _ in range(n)]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    rows = _garbage_rows(p, 20, 4)
    dev = _to_dev(rows)
    for _ in range(2):                       # (from the second run on the lengths are known and the call returns at once)
        B.vl_liveness_batch(gps, s1)
        torch.cuda.synchronize()
    made = _call(B, gps[-1], p, call, dev, s2)
    with torch.cuda.stream(s1):
        torch.cuda._sleep(SLEEP_CYCLES)
    B.vl_liveness_batch(gps, s1)
    _check(B, oracle_mod, p, call, made, rows, s1, f"{call} after a batch of {n}")
    for gp in gps:
        gp.close()


@pytest.mark.parametrize("call", ["verify", "diagnose", "occupied"])
@pytest.mark.parametrize("kind", ["short", "long"])
def test_run_in_flight_on_the_per_thread_stream_of_another_thread(B, oracle_mod, call, kind):
    """The per-thread default stream has the same handle in every thread and is another stream in each."""
    import torch
    p = _program(kind)
    gp = B.Program(p)
    per_thread = torch.cuda.ExternalStream(2)
    rows = _garbage_rows(p, 20, 5)
    dev = _to_dev(rows)
    for _ in range(2):
        gp.vl_liveness(per_thread)
        torch.cuda.synchronize()
    made = _call(B, gp, p, call, dev, per_thread)
    with torch.cuda.stream(per_thread):
        torch.cuda._sleep(SLEEP_CYCLES)
    gp.vl_liveness(per_thread)
    _check(B, oracle_mod, p, call, made, rows, per_thread, f"{call}, {kind}")
    gp.close()


def test_run_and_call_on_one_stream(B, oracle_mod):
    """Liveness and verify of a short program on one stream, over and over, no synchronisation by the caller in between."""
    import torch
    p = _program("short")
    gp = B.Program(p)
    s = torch.cuda.Stream()
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    outs = []
    for step in range(5):
        rows = _garbage_rows(p, 60, 40 + step)
        dev = _to_dev(rows)
        torch.cuda.synchronize()
        gp.vl_liveness(s)
        outs.append((gp.vl_verify(dev, None, s), dev, rows))
    torch.cuda.synchronize()
    for out, _, rows in outs:
        assert B.verdicts_to_numpy(out).tobytes() == op.verify(lv, rows).tobytes()
    gp.close()


def test_a_later_batch_of_other_handles_is_not_waited_for(B, oracle_mod):
    """Verdicts of a program whose liveness batch has finished do not wait for a later batch of other programs that is held
    back on its caller's stream."""
    import torch
    p = _program("short")
    mine, theirs = [B.Program(p) for _ in range(3)], [B.Program(p) for _ in range(3)]
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    rows = _garbage_rows(p, 20, 6)
    dev = _to_dev(rows)
    out = torch.zeros((len(rows), 4), dtype=torch.int32, device="cuda")
    for _ in range(2):
        B.vl_liveness_batch(mine, s1)
        B.vl_liveness_batch(theirs, s2)
        mine[2].vl_verify(dev, out, s1)
        torch.cuda.synchronize()
    out.zero_()
    torch.cuda.synchronize()
    B.vl_liveness_batch(mine, s1)
    with torch.cuda.stream(s2):
        torch.cuda._sleep(SLEEP_CYCLES)
    B.vl_liveness_batch(theirs, s2)
    mine[2].vl_verify(dev, out, s1)
    s1.synchronize()
    assert not s2.query(), "the call waited for a batch of other programs"
    torch.cuda.synchronize()
    op = oracle_mod.OracleProgram(p)
    assert B.verdicts_to_numpy(out).tobytes() == op.verify(op.liveness(), rows).tobytes()
    # the handles of a batch do not depend on the one whose event they share
    B.vl_liveness_batch(mine, s1)
    mine[0].close()
    mine[1].vl_liveness(s2)
    for gp in mine[1:] + theirs:
        assert B.verdicts_to_numpy(gp.vl_verify(dev)).tobytes() == op.verify(op.liveness(), rows).tobytes()
        gp.close()


@pytest.mark.parametrize("kind", ["short", "long"])
@pytest.mark.parametrize("same_stream", [False, True])
def test_capture_behind_a_run_in_flight(B, oracle_mod, kind, same_stream):
    """A call that is captured while a liveness run is in flight: the host waits for the run, the graph can be launched."""
    import torch
    p = _program(kind)
    gp = B.Program(p)
    rows = _garbage_rows(p, 30, 8)
    dev = _to_dev(rows)
    out = torch.zeros((len(rows), 4), dtype=torch.int32, device="cuda")
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    gp.vl_liveness(s1)
    gp.vl_verify(dev, out, s1)
    torch.cuda.synchronize()
    out.zero_()
    torch.cuda.synchronize()
    s = s1 if same_stream else s2
    gp.vl_liveness(s1)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s, capture_error_mode="relaxed"):
        gp.vl_verify(dev, out, s)
    op = oracle_mod.OracleProgram(p)
    want = op.verify(op.liveness(), rows)
    for _ in range(2):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert B.verdicts_to_numpy(out).tobytes() == want.tobytes()
    gp.close()


def test_many_rows_on_two_streams(B, oracle_mod):
    """Calls of more rows than a pass holds, on two streams, without anything between them: they do not meet in the handle's
    working set."""
    import torch
    shape = synth.Shape("line", [3100], [], [], [], n_vregs=1000, widths={1: 0.7, 2: 0.2, 4: 0.1}, P=128)
    p = synth.build_program(shape, 3)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    K = 6000
    some = [_garbage_rows(p, 60, 70 + j) for j in range(2)]
    for s in some:
        s[:30] = synth.candidate_rows(p, 30, 0.3, 4)[0]
    picks = [np.random.default_rng(j).integers(0, 60, K) for j in range(2)]
    devs = [_to_dev(s[pick]) for s, pick in zip(some, picks)]
    wants = [op.verify(lv, s)[pick] for s, pick in zip(some, picks)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    outs = [torch.zeros((K, 4), dtype=torch.int32, device="cuda") for _ in range(8)]
    gp.vl_verify(devs[0], outs[0])
    torch.cuda.synchronize()
    for j in range(8):
        gp.vl_verify(devs[j % 2], outs[j], streams[j % 2])
    torch.cuda.synchronize()
    for j in range(8):
        assert B.verdicts_to_numpy(outs[j]).tobytes() == wants[j % 2].tobytes(), f"call {j}"
    gp.close()
