"""The one-kernel path of short jobs: at the edges of what it takes (rows, short chunks, register file sizes) against
the CPU oracle, every verdict field, bit-exact."""
import numpy as np
import pytest

from paper_2506_17506_b200 import synth
from tests import helpers as H
from tests.test_gpu_parity import _assert_same, _garbage_rows, _gpu_verify, _to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_17506_b200 import binding
    return binding


@pytest.mark.parametrize("P,chunk", [(31, 160), (64, 8), (4000, 16), (8000, 160)])
def test_random_programs(B, oracle_mod, P, chunk):
    """Register files whose masks take 512 threads, 256 threads and no block at all (the batched kernels); several
    definitions per instruction, wide and misaligned tuples, rows that collide everywhere."""
    for seed in range(6):
        p = H.random_program(9100 + seed, max_instrs=400, max_vregs=60, max_blocks=9, P=P, widths=(1, 2, 3, 8, 33), B=[4, 3][seed % 2])
        gp = B.Program(p)
        gp.set_option(B.VL_OPT_CHUNK_INSTRS, chunk)
        gp.vl_liveness()
        op = oracle_mod.OracleProgram(p)
        rows = _garbage_rows(p, 40, seed)
        _assert_same(_gpu_verify(B, gp, rows), op.verify(op.liveness(), rows), f"P {P} chunk {chunk} seed {seed}")
        gp.close()


@pytest.mark.parametrize("chunk", [160, 8])
@pytest.mark.parametrize("shape", ["gemm", "attention"])
@pytest.mark.parametrize("per_sm,more", [(0, 1), (1, 0), (1, 1), (2, 0), (2, 1), (3, 0), (3, 1), (5, 0)])
def test_row_counts_and_many_short_chunks(B, oracle_mod, per_sm, more, shape, chunk):
    """One, two and three rows per multiprocessor and one row more, for a program of 2,000 instructions (whose rows count their
    own collisions, in several rounds beyond three) and one of 8,000 (which hands them over from the second row per
    multiprocessor on, and takes the batched kernels beyond three); and with more short chunks (1,000) than a thread block
    has threads."""
    K = per_sm * _sm_count() + more
    wl = synth.workload({"gemm": 1, "attention": 2}[shape])
    p = synth.build_program(wl.shapes[0], wl.seeds[0])
    rows, _ = synth.candidate_rows(p, K, 0.5, 77)
    rows[: K // 10] = _garbage_rows(p, K, 3)[: K // 10]
    gp = B.Program(p)
    gp.set_option(B.VL_OPT_CHUNK_INSTRS, chunk)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    _assert_same(_gpu_verify(B, gp, rows), op.verify(op.liveness(), rows), f"K {K} chunk {chunk}")
    gp.close()


def test_exact_counts_in_global_memory(B, oracle_mod):
    """52,000 vregs and 20,000 registers: the block arrays of the exact counts do not fit a multiprocessor."""
    V = 52000
    blocks = [[([i], [i - 1, i - 2, i - 40] if i >= 40 else []) for i in range(V)]]
    p = synth.program_from_lists(blocks, [], V, [1 + (v % 3 == 0) for v in range(V)], 20000)
    gp = B.Program(p)
    gp.set_option(B.VL_OPT_GROUP, 1)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    rng = np.random.default_rng(5)
    good = (np.arange(V) * 2) % 20000
    tables = [good, np.where(rng.random(V) < 1e-3, 20005, good), np.where(rng.random(V) < 1e-2, 7, good), rng.integers(0, 20000, V)]
    rows = np.stack([H.row_from_table(p, t) for t in tables])
    _assert_same(_gpu_verify(B, gp, rows), op.verify(lv, rows), "global")
    gp.close()


@pytest.mark.parametrize("failing", [1, 12, 60])
def test_exact_count_items(B, oracle_mod, failing):
    """Failing rows of the batched kernels few enough that each fine share of their counts gets a thread block, about
    that many, and more."""
    wl = synth.workload(2)
    p = synth.build_program(wl.shapes[0], wl.seeds[0])
    rows, _ = synth.candidate_rows(p, 70, 0.0, 78)
    bad = (np.arange(failing) * 7) % 70
    rows[bad] = _garbage_rows(p, failing, 5)
    rows[bad[::2]] = synth.candidate_rows(p, failing, 1.0, 79)[0][: len(bad[::2])]
    gp = B.Program(p)
    gp.set_option(B.VL_OPT_GROUP, 8)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    _assert_same(_gpu_verify(B, gp, rows), op.verify(op.liveness(), rows), f"{failing} failing")
    gp.close()


@pytest.mark.parametrize("P,n_banks,K", [(64, 4, 149), (500, 3, 300), (250, 2, 444)])
def test_counts_handed_over(B, oracle_mod, P, n_banks, K):
    """Programs large enough that the rows of a short job leave their counts to the kernel for those: general and
    fast bank tally, rows that collide everywhere and hardly, two calls in a row."""
    V = 7200
    blocks = [[([i], [i - 1, i - 2, i - 17] if i >= 17 else []) for i in range(b * 1800, (b + 1) * 1800)] for b in range(4)]
    p = synth.program_from_lists(blocks, [(0, 1), (1, 1), (1, 2), (2, 3)], V, [1 + (v % 5 == 0) for v in range(V)], P, n_banks)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    rng = np.random.default_rng(K)
    good = (np.arange(V) * 2) % (P - P % 2)
    for call in range(2):
        rows = np.stack([H.row_from_table(p, np.where(rng.random(V) < [0, 0, 3e-4, 0.05, 1][k % 5], rng.integers(0, P, V), good))
                         for k in range(K)])
        _assert_same(_gpu_verify(B, gp, rows), op.verify(lv, rows), f"P {P} call {call}")
    gp.close()


def test_counts_handed_over_after_a_call_that_was_cut_short(B, oracle_mod):
    """A call whose rows were listed for the exact counts, which then never ran (as if their launch had failed: a captured
    call with that kernel switched off), leaves nothing behind for the next one."""
    import torch
    rt = pytest.importorskip("cuda.bindings.runtime")
    P, V, K = 250, 7200, 300
    blocks = [[([i], [i - 1, i - 2, i - 17] if i >= 17 else []) for i in range(b * 1800, (b + 1) * 1800)] for b in range(4)]
    p = synth.program_from_lists(blocks, [(0, 1), (1, 1), (1, 2), (2, 3)], V, [1 + (v % 5 == 0) for v in range(V)], P)
    gp = B.Program(p)
    B.vl_liveness_batch([gp])
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    rng = np.random.default_rng(9)
    good = (np.arange(V) * 2) % P
    def rows_of(share):
        return np.stack([H.row_from_table(p, np.where(rng.random(V) < share[k % len(share)], rng.integers(0, P, V), good)) for k in range(K)])
    rows = rows_of([0, 3e-4, 0.05, 1])
    _assert_same(_gpu_verify(B, gp, rows), op.verify(lv, rows), "before")
    dev, s = _to_dev(rows), torch.cuda.Stream()
    out = torch.full((K, 4), -9, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()

    def ok(r):
        assert int(r[0]) == 0, r
        return r[1] if len(r) == 2 else r[1:]

    ok(rt.cudaStreamBeginCapture(s.cuda_stream, rt.cudaStreamCaptureMode.cudaStreamCaptureModeRelaxed))
    gp.vl_verify(dev, out, s)
    graph = ok(rt.cudaStreamEndCapture(s.cuda_stream))
    nodes, n = ok(rt.cudaGraphGetNodes(graph, 16))
    nodes = nodes[:n]
    kernels = [n for n in nodes if ok(rt.cudaGraphNodeGetType(n)) == rt.cudaGraphNodeType.cudaGraphNodeTypeKernel]
    assert len(kernels) == 2
    whole = ok(rt.cudaGraphInstantiate(graph, 0))
    cut = ok(rt.cudaGraphInstantiate(graph, 0))
    ok(rt.cudaGraphNodeSetEnabled(cut, kernels[1], 0))
    ok(rt.cudaGraphLaunch(cut, s.cuda_stream))
    s.synchronize()
    got, want = B.verdicts_to_numpy(out), op.verify(lv, rows)
    unfinished = got["conflict_pairs"] == np.uint32(2**32 - 9)
    assert (want["conflict_pairs"][unfinished] > 0).any()     # rows that collided were not counted
    rows2 = rows_of([1, 0.05, 0, 3e-4])
    _assert_same(_gpu_verify(B, gp, rows2), op.verify(lv, rows2), "after")
    ok(rt.cudaGraphLaunch(cut, s.cuda_stream))
    for _ in range(2):                                        # and a captured call can be replayed
        ok(rt.cudaGraphLaunch(whole, s.cuda_stream))
        s.synchronize()
        _assert_same(B.verdicts_to_numpy(out), want, "replay")
    for g in (whole, cut):
        rt.cudaGraphExecDestroy(g)
    rt.cudaGraphDestroy(graph)
    gp.close()


@pytest.mark.parametrize("V,takes", [(57000, True), (60000, False)])
def test_a_refused_program_is_refused_for_every_number_of_rows(B, oracle_mod, V, takes):
    """The table of one candidate with its bank nibbles does not fit a multiprocessor, whatever the short jobs' kernel needs."""
    import torch
    blocks = [[([i], [i - 1] if i else []) for i in range(V)]]
    p = synth.program_from_lists(blocks, [], V, [1] * V, 64)
    gp = B.Program(p)
    gp.vl_liveness()
    rows = np.stack([H.row_from_table(p, (np.arange(V) * (k + 1)) % 64) for k in range(3)])
    dev = _to_dev(rows)
    n, off, vreg = 600, *gp.vl_dict_layout()
    many = torch.zeros((n, gp.pitch), dtype=torch.int16, device="cuda").view(torch.uint16)
    calls = [lambda: gp.vl_verify(dev), lambda: gp.vl_verify_dict(torch.zeros((1, (len(vreg) + 7) // 8 * 8), dtype=torch.int16, device="cuda").view(torch.uint16)),
             lambda: gp.vl_verify_host(rows), lambda: gp.vl_verify_until_pass(dev, 1), lambda: B.vl_verify_batch([gp, gp], [dev, dev]),
             lambda: gp.vl_verify(many)]
    for j, call in enumerate(calls):
        if takes:
            call()
            continue
        with pytest.raises(B.VlError) as e:
            call()
        assert e.value.code == B.VL_ERR_UNSUPPORTED, j
    if takes:
        op = oracle_mod.OracleProgram(p)
        _assert_same(_gpu_verify(B, gp, rows), op.verify(op.liveness(), rows))
    gp.close()


def _crowded(n_blocks, per_block, V, P, seed):
    """Every vreg is read again and again in every block: nearly all of them are live everywhere."""
    rng = np.random.default_rng(seed)
    blocks = [[([v], []) for v in range(V)] if b == 0 else [] for b in range(n_blocks)]
    for b in range(n_blocks):
        for _ in range(per_block):
            blocks[b].append(([int(rng.integers(V))], [int(x) for x in rng.integers(0, V, 2)]))
    edges = sorted({(b, b + 1) for b in range(n_blocks - 1)} | {(int(b), int(b) // 2) for b in rng.integers(1, n_blocks, n_blocks)})
    return synth.program_from_lists(blocks, edges, V, [1 + int(x) for x in rng.integers(0, 3, V)], P)


def _sm_count():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("per_block,V,K", [(10, 200, 127), (60, 300, 1), (60, 300, 127), (60, 300, 128), (60, 300, "sms"), (60, 300, "sms+1")])
def test_programs_that_occupy_many_vregs(B, oracle_mod, per_block, V, K):
    """Fewer and more entries of the short chunks than the line between the kernels, at the edges of its row counts."""
    K = {"sms": _sm_count(), "sms+1": _sm_count() + 1}.get(K, K)
    p = _crowded(35, per_block, V, 700, per_block)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    rows = _garbage_rows(p, K, 3)
    rows[::2] = np.stack([H.row_from_table(p, (np.arange(V) * 3 + 7 * (k % 4 == 0) * (np.arange(V) == 5)) % 690) for k in range(len(rows[::2]))])
    _assert_same(_gpu_verify(B, gp, rows), op.verify(op.liveness(), rows), f"K {K}")
    gp.close()


@pytest.mark.parametrize("with_through", [False, True])
@pytest.mark.parametrize("n_banks", [4, 3])
def test_long_lists(B, oracle_mod, with_through, n_banks):
    """More than 1,024 entries per list on average (a warp counts an instruction), with and without a through-set;
    instructions with many definitions and many reads, sources on one register."""
    rng = np.random.default_rng(3)
    A, N = 300, 1300
    body = []
    for i in range(900):
        nd, nr = [(1, 2), (1, 4), (2, 3), (0, 2), (5, 9), (1, 0)][i % 6]
        defs = [A + int(x) for x in rng.choice(N, nd, replace=False)]
        body.append((defs, [int(x) for x in rng.integers(0, A + N, nr)]))
    ends = [([], [A + v for v in range(j, min(j + 4, N))]) for j in range(0, N, 4)]
    if with_through:   # vregs 0 .. A-1 are live through the loop; most of them are not touched in it
        body = [(d, [v for v in r if v >= A or v < 20]) for d, r in body]
    blocks = [[([v], []) for v in range(A)], [([A + v], []) for v in range(N)] + body + ends, [([], list(range(j, j + 4))) for j in range(0, A, 4)]]
    p = synth.program_from_lists(blocks, [(0, 1), (1, 1), (1, 2)], A + N, [1 + (v % 7 == 0) + 2 * (v % 50 == 0) for v in range(A + N)], 3000, n_banks)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    good = np.cumsum(np.concatenate([[0], p.vreg_width[:-1]]))
    assert good[-1] < 2900
    tables = [good, good, np.where(np.arange(A + N) == 700, good[701], good), np.where(rng.random(A + N) < 0.01, good[::-1], good),
              np.where(np.arange(A + N) < 2, 2999, good), np.where(np.arange(A + N) == 40, 3100, good), rng.integers(0, 3000, A + N)]
    rows = np.stack([H.row_from_table(p, t) for t in tables] + list(_garbage_rows(p, 12, 4)))
    rows[1, p.n_operands // 2] += 1
    _assert_same(_gpu_verify(B, gp, rows), op.verify(op.liveness(), rows))
    gp.close()


@pytest.mark.parametrize("K", [20, 300, 700])
def test_kernel_times_of_short_jobs(B, K):
    """Every call records a pass of every handle that asks for it: alone, handed over, in a launch that programs share, on
    lanes, by the batched kernels."""
    import torch
    wl = synth.workload(2)
    big = synth.build_program(wl.shapes[0], wl.seeds[0])
    small = synth.build_program(synth.shape_gemm(), 1)
    progs = [big, small, small]
    gps = [B.Program(p) for p in progs]
    B.vl_liveness_batch(gps)
    rows = [_to_dev(synth.candidate_rows(p, K, 0.3, 5)[0]) for p in progs]
    for gp in gps[:2]:
        gp.set_option(B.VL_OPT_KERNEL_TIMING, 1)
    for call in range(2):
        B.vl_verify_batch(gps, rows)
        torch.cuda.synchronize()
        for gp, n in zip(gps, (1, 1, 0)):
            ms, passes = gp.vl_kernel_times()
            assert passes == n and all(x >= 0 for x in ms) and (ms[0] > 0) == (n > 0)
    B.vl_verify_batch([gps[1], gps[1]], [rows[1], rows[1]])     # a handle given twice in one launch, or in two
    torch.cuda.synchronize()
    ms, passes = gps[1].vl_kernel_times()
    assert passes in (1, 2) and 0 < sum(ms) < 100
    gps[0].vl_verify(rows[0])
    torch.cuda.synchronize()
    ms, passes = gps[0].vl_kernel_times()
    assert passes == 1 and ms[0] > 0
    if K == 300:                                                # 8,000 instructions: k_fused, then k_exact
        assert ms[1] < ms[0] and ms[2] < ms[0] and ms[3] > 0.004
    for gp in gps:
        gp.close()


@pytest.mark.parametrize("shape,n,K", [("gemm", 9, 20), ("attention", 2, 50), ("nested", 8, "sms"), ("mixed", 12, 60)])
def test_short_jobs_of_several_programs(B, oracle_mod, shape, n, K):
    """Jobs that share a launch (many of small programs), take one each (few of larger ones), or go to the batched kernels
    (many rows of large programs); small and large ones together, some without rows."""
    K = _sm_count() if K == "sms" else K
    shapes = {"gemm": [synth.shape_gemm()], "attention": [synth.shape_attention()], "nested": [synth.shape_stress(20000, 6000)],
              "mixed": [synth.shape_tiny(), synth.shape_gemm(), synth.shape_attention()]}[shape]
    cases = []
    for j, s in enumerate(shapes):
        p = synth.build_program(s, j)
        rows = synth.candidate_rows(p, K, 0.3, 60 + j)[0]
        op = oracle_mod.OracleProgram(p)
        cases.append((p, rows, op.verify(op.liveness(), rows)))
    use = [cases[j % len(cases)] for j in range(n)]
    gps = [B.Program(p) for p, _, _ in use]
    devs = [_to_dev(rows[: 0 if j == n // 2 and n > 2 else K]) for j, (_, rows, _) in enumerate(use)]
    for call in range(2):
        B.vl_liveness_batch(gps)
        outs = B.vl_verify_batch(gps, devs)
        for j, (o, (_, _, want)) in enumerate(zip(outs, use)):
            _assert_same(B.verdicts_to_numpy(o), want[: o.shape[0]], f"call {call} program {j}")
    for gp in gps:
        gp.close()
