"""The verify path with eight candidates per thread block: at the edges of what it takes (rows, tiles, widths, register files)
and on both sides of its rules, against the CPU oracle, every verdict field, exact."""
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


def _member(n_instrs, seed):
    shape = synth.Shape("loop", [n_instrs // 4, n_instrs - n_instrs // 4], [(0, 1), (1, 1)], [(1, 1)], [],
                        n_vregs=n_instrs * 2 // 5, widths={1: 0.7, 2: 0.2, 4: 0.1}, P=200)
    return synth.build_program(shape, seed)


def _rows(p, K, seed):
    """Valid rows, rows with one fault, and garbage: many collisions, registers outside the file."""
    rows, _ = synth.candidate_rows(p, K, 0.4, seed)
    rows[5: K: 29] = _garbage_rows(p, K, seed)[5: K: 29]
    return rows


def _launches(B, call):
    before = B.vl_kernel_launches()
    call()
    return B.vl_kernel_launches() - before


# rows: 512 threads, 256 threads, counts handed over or made by the block itself (one launch less), a block with a single row;
# columns: whole tiles, one more, few
@pytest.mark.parametrize("n_instrs,K,launches", [(2000, 889, 2), (2000, 1500, 2), (2000, 2001, 1), (2001, 1184, 2), (2003, 1185, 2), (1500, 3001, 1),
                                                 (4000, 800, 2)])
def test_row_counts(B, oracle_mod, n_instrs, K, launches):
    p = _member(n_instrs, n_instrs + K)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    lv = op.liveness()
    rows = _rows(p, K, K)
    want = op.verify(lv, rows)
    for _ in range(2):
        _assert_same(_gpu_verify(B, gp, rows), want, f"{n_instrs} instructions, {K} rows")
    drows = synth.dict_rows(p, rows)
    got = B.verdicts_to_numpy(gp.vl_verify_dict(_to_dev(drows)))
    _assert_same(got, op.verify_dict(lv, drows), "dictionary rows")
    dev, ddev = _to_dev(rows), _to_dev(drows)
    assert _launches(B, lambda: gp.vl_verify(dev)) == launches, "another path has checked the rows"
    assert _launches(B, lambda: gp.vl_verify_dict(ddev)) == launches, "another path has checked the dictionary rows"
    gp.close()


# the largest tables: a multiprocessor each, 512 threads and 256; one that does not fit
@pytest.mark.parametrize("V,launches", [(10200, 2), (11400, 2), (12500, 3)])
def test_many_vregs(B, oracle_mod, V, launches):
    """A chain: every instruction defines a vreg of its own and reads some of the last ones."""
    rng = np.random.default_rng(V)
    ins = [([v], [int(u) for u in v - rng.integers(1, 9, int(rng.integers(0, 4))) if u >= 0]) for v in range(V)]
    cut = V // 3
    p = synth.program_from_lists([ins[:cut], ins[cut:]], [(0, 1)], V, [1, 2] * (V // 2), 64)
    table = np.arange(V) * 2 % 64
    some = np.stack([H.row_from_table(p, (table + 2 * k) % 64) for k in range(20)])
    for k in range(8):                       # an overlap, a vreg outside the file, an occurrence that differs
        t = (table + 2 * k) % 64
        v = int(rng.integers(20, V))
        t[v] = (t[v - 3], 64 + k)[k % 2]
        some[k] = H.row_from_table(p, t)
    some[8, p.n_operands - 1] += 2
    some[9:11, : p.n_operands] = rng.integers(0, 70, (2, p.n_operands))
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    verdicts = op.verify(op.liveness(), some)
    assert (verdicts["flags"] == B.VL_PASS).any()
    pick = np.arange(500) % 20
    dev = _to_dev(some[pick])
    _assert_same(B.verdicts_to_numpy(gp.vl_verify(dev)), verdicts[pick])
    assert _launches(B, lambda: gp.vl_verify(dev)) == launches, "another path has checked the rows"
    gp.close()


# register files that end inside and at a mask word, widths at 8 (taken) and 9 (not), banks, more blocks than through-sets serve
@pytest.mark.parametrize("P,widths,banks,max_blocks", [(32, (1, 2, 4), 4, 4), (33, (1, 3, 8), 2, 6), (64, (1, 9), 4, 4),
                                                       (500, (1, 2, 4, 8), 1, 8), (2000, (8,), 4, 40), (64, (1, 2), 3, 4)])
def test_random_programs(B, oracle_mod, P, widths, banks, max_blocks):
    for seed in range(3):
        p = H.random_program(8800 + seed, max_instrs=1800, max_vregs=300, max_blocks=max_blocks, P=P, widths=widths, B=banks)
        gp = B.Program(p)
        gp.vl_liveness()
        op = oracle_mod.OracleProgram(p)
        if seed == 1:
            rules = dict(vreg_align=np.where(p.vreg_width > 1, 2, 1), reserved=[p.P - 1])
            op.set_constraints(**rules)
            gp.set_constraints(P=p.P, **rules)
        K = 3000
        rows = np.tile(_garbage_rows(p, 300, seed), (10, 1))
        want = np.tile(op.verify(op.liveness(), rows[:300]), 10)
        _assert_same(_gpu_verify(B, gp, rows[:K]), want, f"P {P} seed {seed}")
        gp.close()


@pytest.mark.parametrize("n,n_instrs,K,launches", [(4, 2000, 900, 1), (9, 4000, 600, 1), (4, 300, 3000, 1), (8, 4000, 800, 32)])
def test_programs_of_many_rows(B, oracle_mod, n, n_instrs, K, launches):
    """Jobs that k_eight would take alone and that k_fused could: they share a launch of one or the other, or run batched (the last)."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines lie elsewhere")
    progs = [_member(n_instrs, 60 + j) for j in range(n)]
    gps = [B.Program(p) for p in progs]
    B.vl_liveness_batch(gps)
    pick = np.arange(K) % 50
    devs, wants = [], []
    for j, p in enumerate(progs):
        op = oracle_mod.OracleProgram(p)
        some = _rows(p, 50, j)
        wants.append(op.verify(op.liveness(), some)[pick])
        devs.append(_to_dev(some[pick]))
    B.vl_verify_batch(gps, devs)
    before = B.vl_kernel_launches()
    outs = B.vl_verify_batch(gps, devs)
    torch.cuda.synchronize()
    assert B.vl_kernel_launches() - before == launches
    for o, w in zip(outs, wants):
        _assert_same(B.verdicts_to_numpy(o), w)
    for gp in gps:
        gp.close()


def test_several_programs(B, oracle_mod):
    """Jobs of several programs in one call, enough of them for the kernel to take them together; one that it does not take."""
    import torch
    progs = [_member(900 + 331 * j, j) for j in range(9)]
    progs.append(H.random_program(8900, max_instrs=900, max_vregs=200, P=64, widths=(1, 9)))
    Ks = [100, 131, 8, 1, 97, 200, 148, 120, 90, 110]
    gps = [B.Program(p) for p in progs]
    B.vl_liveness_batch(gps)
    rows = [_rows(p, K, K) if p.gen else _garbage_rows(p, K, K) for p, K in zip(progs, Ks)]
    wants = []
    for p, r in zip(progs, rows):
        op = oracle_mod.OracleProgram(p)
        wants.append(op.verify(op.liveness(), r))
    for reps in (1, 4):
        outs = B.vl_verify_batch(gps * reps, [_to_dev(r) for r in rows] * reps)
        torch.cuda.synchronize()
        for o, w in zip(outs, wants * reps):
            _assert_same(B.verdicts_to_numpy(o), w)
    for gp in gps:
        gp.close()


# counts handed over (512 and 256 threads), made by the block itself
@pytest.mark.parametrize("K", [40, 1500, 2500])
def test_bounded_wait_runs_out(B, oracle_mod, K):
    """The wait of the consumers for their first tile runs out (test hook): the call returns, no verdict passes, the status says so,
    and the next call is exact again."""
    import torch
    p = _member(2000, K)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    rows = _rows(p, K, K)
    want = op.verify(op.liveness(), rows)
    _assert_same(_gpu_verify(B, gp, rows), want, "before")
    gp.set_option(B.VL_OPT_TEST_WAIT, 1)
    out = gp.vl_verify(_to_dev(rows))
    torch.cuda.synchronize()
    with pytest.raises(B.VlError) as e:
        gp.vl_verify_status()
    assert e.value.code == B.VL_ERR_DEVICE_WAIT
    got = B.verdicts_to_numpy(out)
    assert np.all(got["flags"] == 0) and np.all(got["first_violation_instr"] == -1), "a row of a block that gave up has a verdict"
    gp.set_option(B.VL_OPT_TEST_WAIT, 0)
    for _ in range(2):
        _assert_same(_gpu_verify(B, gp, rows), want, "after the wait ran out")
    gp.close()


# counts handed over (few rows; many rows of a long program, up to the most), made by the block itself; candidates in fine items, in
# coarse ones, one item each
@pytest.mark.parametrize("n_instrs,K,launches", [(2399, 2000, 2), (2399, 2001, 1), (2400, 2001, 2), (2400, 4800, 2), (2400, 4801, 1), (3500, 6800, 2), (4100, 700, 2)])
@pytest.mark.parametrize("noise", [0.004, 0.2, 1.0])
def test_rows_that_collide_everywhere(B, oracle_mod, n_instrs, K, launches, noise):
    """Rows of random registers (every chunk collides, vregs outside the file, tuples across mask words) among valid ones."""
    p = _member(n_instrs, 7)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    some = _rows(p, 100, 3)
    some[50:] = _garbage_rows(p, 50, 4)
    verdicts = op.verify(op.liveness(), some)
    rng = np.random.default_rng(K)
    pick = np.where(rng.random(K) < noise, rng.integers(50, 100, K), rng.integers(0, 50, K))
    dev = _to_dev(some[pick])
    out = gp.vl_verify(dev)
    before = B.vl_kernel_launches()
    gp.vl_verify(dev, out)
    assert B.vl_kernel_launches() - before == launches, "another path has checked the rows"
    _assert_same(B.verdicts_to_numpy(out), verdicts[pick], f"{K} rows")
    gp.close()


@pytest.mark.parametrize("K", [600, 1500])
def test_tuples_across_mask_words(B, oracle_mod, K):
    """Valid rows whose tuples sit anywhere: ranges that reach into the next word of the occupancy masks, in every block."""
    import copy
    p = copy.copy(_member(3000, 5))
    rows, _ = synth.candidate_rows(p, K, 0.2, 9)
    rows += 3
    p.P += 8
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    want = op.verify(op.liveness(), rows)
    assert (want["flags"] == B.VL_PASS).mean() > 0.7
    _assert_same(_gpu_verify(B, gp, rows), want)
    gp.close()


@pytest.mark.parametrize("n_instrs,K,launches", [(11200, 1184, 2), (11200, 1190, 4), (11200, 1381, 4), (11200, 1382, 2), (10900, 1190, 2), (16100, 1430, 4), (16100, 1184, 2)])
def test_route(B, oracle_mod, n_instrs, K, launches):
    """On both sides of the lines beyond one block per multiprocessor (148 of them)."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the lines lie elsewhere")
    p = _member(n_instrs, 7)
    gp = B.Program(p)
    gp.vl_liveness()
    op = oracle_mod.OracleProgram(p)
    some = _rows(p, 60, 3)
    verdicts = op.verify(op.liveness(), some)
    pick = np.arange(K) % 60
    dev = _to_dev(some[pick])
    out = gp.vl_verify(dev)
    before = B.vl_kernel_launches()
    gp.vl_verify(dev, out)
    assert B.vl_kernel_launches() - before == launches, "another path has checked the rows"
    _assert_same(B.verdicts_to_numpy(out), verdicts[pick], f"{K} rows")
    gp.close()
