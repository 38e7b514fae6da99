"""Liveness of short programs (one cluster of thread blocks, or one block): at the edges of the pieces, of the shares and of
what it takes, against the CPU oracle, every result and every verdict field, exact."""
import numpy as np
import pytest

from paper_2506_17506_b200 import synth
from tests import helpers as H
from tests.test_gpu_parity import _assert_same, _check_liveness_result, _garbage_rows, _gpu_verify

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2506_17506_b200 import binding
    return binding


def _program(n_instrs, n_blocks, n_vregs, max_reads, seed):
    """A loop nest over n_blocks blocks; instructions of 0 to 3 definitions and up to max_reads reads, repeats among them."""
    rng = np.random.default_rng(seed)
    blocks = [[] for _ in range(n_blocks)]
    for v in range(0, n_vregs, 3):  # strict: the entry block defines everything
        blocks[0].append((list(range(v, min(v + 3, n_vregs))), []))
    for i in range(n_instrs - len(blocks[0])):
        nd = min(int(rng.choice([0, 1, 1, 1, 2, 3])), n_vregs)
        defs = rng.choice(n_vregs, nd, replace=False).tolist()
        reads = rng.integers(0, n_vregs, int(rng.integers(0, max_reads + 1))).tolist()
        blocks[i * n_blocks // max(1, n_instrs)].append((defs, reads))
    edges = sorted({(b, b + 1) for b in range(n_blocks - 1)} | {(b, b) for b in range(1, n_blocks)} | {(n_blocks - 1, n_blocks // 2)})
    return synth.program_from_lists(blocks, edges, n_vregs, [int(w) for w in rng.choice([1, 1, 2, 4], n_vregs)], 64, 4)


# instructions around 32 pieces (one block or a cluster) and around 4,096 (a cluster or the separate kernels); instructions of so
# many operands that a piece holds one, or is one; more than 32 and more than 1,024 vregs; many blocks, few chunks, long chunks;
# long programs whose instructions of many operands share pieces, with bitsets that fit shared memory and ones that do not
CASES = [(256, 1, 5, 3, 160), (257, 2, 40, 3, 160), (250, 3, 70, 40, 160), (1000, 7, 1100, 6, 160), (4096, 5, 300, 3, 160),
         (4097, 5, 300, 3, 160), (2000, 40, 200, 4, 160), (2000, 3, 200, 4, 8), (3000, 2, 100, 3, 65536), (300, 2, 2100, 100, 24),
         (4200, 5, 300, 40, 160), (4300, 2, 40, 90, 24), (6000, 3, 9000, 60, 160)]


@pytest.mark.parametrize("n_instrs,n_blocks,n_vregs,max_reads,chunk", CASES)
def test_results(B, oracle_mod, n_instrs, n_blocks, n_vregs, max_reads, chunk):
    p = _program(n_instrs, n_blocks, n_vregs, max_reads, n_instrs + n_vregs)
    gp = B.Program(p)
    gp.set_option(B.VL_OPT_CHUNK_INSTRS, chunk)
    rows = _garbage_rows(p, 6, 3)
    want = None
    for run in range(3):
        gp.vl_liveness()
        _, lv = _check_liveness_result(B, oracle_mod, gp, p)
        if want is None:
            want = oracle_mod.OracleProgram(p).verify(lv, rows)
        _assert_same(_gpu_verify(B, gp, rows), want, f"run {run}")
    gp.close()


def test_batch_of_short_and_long_programs(B, oracle_mod):
    """Programs of both kinds in one call."""
    progs = [_program(n, 3, 90, 4, n) for n in (64, 4500, 700, 257, 5000, 4096)]
    gps = [B.Program(p) for p in progs]
    for _ in range(3):
        B.vl_liveness_batch(gps)
    for gp, p in zip(gps, progs):
        _check_liveness_result(B, oracle_mod, gp, p)
        gp.close()
