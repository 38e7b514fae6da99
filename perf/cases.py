"""Timing cases of the candidate verifier: what its users have it do, over the range of sizes they have.

A case names a program (a shape of ``synth`` and its seed), a number of candidate rows with the share of
faulted ones, and the entry points one pass goes through (``path``):

* ``verify``    ``vl_verify`` of rows resident in device memory on a handle whose liveness is known (the
                resampling loop: more candidates of a kernel in hand)
* ``step``      ``vl_liveness`` then ``vl_verify`` (a kernel that has just come in, or has just changed)
* ``dict``      ``vl_verify_dict``: rows as one dictionary per basic block, the form the model emits
* ``host``      ``vl_verify_host``: rows in pinned host memory, verdicts back on the host
* ``until``     ``vl_verify_until_pass``: resampling with early exit, batch by batch
* ``batch``     many programs at once: ``vl_liveness_batch``, ``vl_verify_batch``, ``vl_resample_stats``
* ``feedback``  ``vl_liveness``, ``vl_diagnose`` and ``vl_occupied_masks`` of one failing row

Every output is an integer, so every result has to be equal.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2506_17506_b200 import binding as vl
from paper_2506_17506_b200 import synth

_W2 = {1: 0.70, 2: 0.20, 4: 0.10}
MAX_BYTES = 1_950_000_000       # candidate bytes of a drawn case: no more than the largest listed one
STRESS_MIN = 8000               # instructions from which the nested-loop shape has room for its accumulators


def listed():
    return [
        # the smallest call: a straight-line kernel of 64 instructions, pass@100; launches and host work count
        dict(name="tiny_step_100", path="step", shape="tiny", seed=0, K=100, faults=0.30, rules=False),
        # one more sample of a GEMM-shaped kernel in the regeneration loop
        dict(name="gemm_verify_1", path="verify", shape="gemm", seed=1, K=1, faults=0.0, rules=False),
        # pass@100 of a GEMM-shaped kernel that has just come in
        dict(name="gemm_step_100", path="step", shape="gemm", seed=1, K=100, faults=0.20, rules=False),
        # a thousand samples of an attention-shaped kernel
        dict(name="attention_verify_1000", path="verify", shape="attention", seed=2, K=1000, faults=0.10, rules=False),
        # the same kernel with its candidates as the model emits them, one dictionary per basic block
        dict(name="attention_dict_1000", path="dict", shape="attention", seed=2, K=1000, faults=0.10, rules=False),
        # odd sizes, alignment + register classes + reserved registers, and a poor model (a third of the rows fail)
        dict(name="nested_rules_777", path="verify", shape="nested", n_instrs=11317, n_vregs=3301, seed=7, K=777,
             faults=0.33, rules=True),
        # a test set: 64 kernels of 1,000 to 4,000 instructions, 100 samples each, with the pass@k statistics
        dict(name="batch_64x100", path="batch", shape="members", n_programs=64, seed=0, K=100, faults=0.15, rules=False),
        # offline filtering: 10,000 samples of the largest kernel of the test configurations
        dict(name="stress_step_10000", path="step", shape="nested", n_instrs=32000, n_vregs=10000, seed=4, K=10000,
             faults=0.05, rules=False),
        # a kernel with more vregs than a table of eight candidates can hold on one multiprocessor
        dict(name="large_verify_1000", path="verify", shape="nested", n_instrs=64000, n_vregs=20000, seed=4, K=1000,
             faults=0.05, rules=False),
        # samples that arrive on the host: copies in and out are part of the call
        dict(name="attention_host_1000", path="host", shape="attention", seed=2, K=1000, faults=0.10, rules=False),
        # resampling with early exit, in batches of 25, under a model that rarely gets it right
        dict(name="gemm_until_25", path="until", shape="gemm", seed=1, K=200, batch_rows=25, faults=0.97, rules=False),
        # what the sampler gets back for one failing candidate: conflicts, violation kinds, occupied registers
        dict(name="attention_feedback", path="feedback", shape="attention", seed=2, K=1, faults=1.0, rules=False),
    ]


def draw(rng):
    path = rng.choice(["step", "step", "verify", "verify", "verify", "dict", "host", "until", "batch", "feedback"])
    if path == "batch":
        return dict(path=path, shape="members", n_programs=int(round(_log_uniform(rng, 2, 96))), seed=rng.randrange(1000),
                    K=int(round(_log_uniform(rng, 1, 128))), faults=round(rng.uniform(0.0, 0.4), 3), rules=False)
    n_instrs = int(round(_log_uniform(rng, 40, 64000 if path in ("step", "verify", "dict") else 20000)))
    case = dict(path=path, n_instrs=n_instrs, seed=rng.randrange(1000), faults=round(rng.uniform(0.0, 0.4), 3),
                rules=path in ("verify", "dict", "host") and rng.random() < 0.25)
    if n_instrs >= STRESS_MIN and (n_instrs > 16000 or rng.random() < 0.7):
        case.update(shape="nested", n_vregs=int(n_instrs * rng.uniform(0.22, 0.34)))
    elif n_instrs >= 700:
        loops = rng.randint(1, 4)
        case.update(shape="loops", loops=loops, n_vregs=int(n_instrs * rng.uniform(0.28, 0.45)) + 32 * loops // 4)
    else:
        case.update(shape="line", n_vregs=max(8, int(n_instrs * rng.uniform(0.3, 0.45))))
    top = {"until": 400, "feedback": 1, "host": 2000}.get(path, 10000)
    top = max(1, min(top, MAX_BYTES // (8 * n_instrs)))
    case["K"] = int(round(_log_uniform(rng, 1, top)))
    if path == "until":
        case["batch_rows"] = rng.choice([8, 10, 25, 50, 100])
        case["faults"] = round(rng.uniform(0.85, 1.0), 3)
    if path == "feedback":
        case["faults"] = 1.0
    return case


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# ------------------------------------------------------------------------------------------- programs
def _loops_shape(n_instrs, n_vregs, loops):
    """Prologue, `loops` self-looping bodies with 32 accumulators each, epilogue."""
    pro = max(80, n_instrs // 10)
    body = (n_instrs - 2 * pro) // loops
    sizes = [pro] + [body] * loops + [n_instrs - pro - body * loops]
    edges = []
    for j in range(loops + 1):
        edges.append((j, j + 1))
        if 1 <= j <= loops:
            edges.append((j, j))
    return synth.Shape("loops", sizes, edges, [(j, j) for j in range(1, loops + 1)],
                       [synth.AccGroup(32, j - 1, (j,), j + 1) for j in range(1, loops + 1)],
                       n_vregs=n_vregs, widths=_W2, P=256)


@functools.lru_cache(maxsize=128)
def _program(shape, seed, n_instrs, n_vregs, loops):
    if shape == "tiny":
        s = synth.shape_tiny()
    elif shape == "gemm":
        s = synth.shape_gemm()
    elif shape == "attention":
        s = synth.shape_attention()
    elif shape == "nested":
        s = synth.shape_stress(n_instrs, n_vregs)
    elif shape == "loops":
        s = _loops_shape(n_instrs, n_vregs, loops)
    elif shape == "member":
        s = synth.shape_batch_member(n_instrs)
    else:
        s = synth.Shape("line", [n_instrs], [], [], [], n_vregs=n_vregs, widths=_W2, P=64)
    return synth.build_program(s, seed)


def _programs(case):
    if case["shape"] == "members":
        first = case["seed"] * 256
        return [_program("member", first + j, first + j, 0, 0) for j in range(case["n_programs"])]
    return [_program(case["shape"], case["seed"], case.get("n_instrs", 0), case.get("n_vregs", 0), case.get("loops", 0))]


@functools.lru_cache(maxsize=16)
def _dict_first_op(shape, seed, n_instrs, n_vregs, loops):
    return synth.dict_layout(_program(shape, seed, n_instrs, n_vregs, loops))[2]


# ----------------------------------------------------------------------------------------- candidates
def _overlap_pairs(prog):
    """(v, u) vreg pairs: v defined by an instruction, u another vreg that the next instruction of the block
    reads, so that u is live where v is written."""
    first = prog.instr_op_off.astype(np.int64)[:-1]
    n_ops = np.diff(prog.instr_op_off.astype(np.int64))
    last_of_block = np.zeros(prog.n_instrs, dtype=bool)
    last_of_block[prog.block_instr_off[1:].astype(np.int64) - 1] = True
    i = np.nonzero(~last_of_block[:-1] & (n_ops[1:] > 1))[0]
    v, u = prog.op_vreg[first[i]].astype(np.int64), prog.op_vreg[first[i + 1] + n_ops[i + 1] - 1].astype(np.int64)
    return v[v != u], u[v != u]


def _classes(prog):
    """Register class of every vreg: the half of the register file that its base allocation lies in."""
    return (prog.gen["base"] >= prog.P // 2).astype(np.int64)


def _rows(prog, K, faults, rules, seed, columns=None):
    """K candidate rows on the GPU (uint16, one column per operand, or the given operand columns).  Valid rows
    are random renamings of the program's base allocation: registers permuted in aligned groups of the widest
    tuple, inside each half of the file and with the last group in its place if there are rules to keep.  A
    share of the rows, at random places, carries one fault: an occurrence that differs, a vreg on the
    registers of one that is live where it is written, or a vreg outside the register file."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)

    def ints(hi, n):
        return torch.randint(0, hi, (n,), device="cuda", generator=gen)

    width = torch.from_numpy(prog.vreg_width.astype(np.int32)).cuda()
    P, W = prog.P, int(prog.vreg_width.max())
    ng = P // W
    base = torch.from_numpy(prog.gen["base"].astype(np.int32)).cuda()
    grp, off = (base // W).long(), base % W
    col_vreg = (prog.op_vreg if columns is None else prog.op_vreg[columns]).astype(np.int64)
    cols = torch.from_numpy(col_vreg).cuda()
    n_cols = len(col_vreg)
    repeats = np.setdiff1d(np.arange(n_cols), np.unique(col_vreg, return_index=True)[1])
    repeats = torch.from_numpy(repeats).cuda()
    v_of, u_of = (torch.from_numpy(x).cuda() for x in _overlap_pairs(prog))
    out = torch.zeros((K, max(8, (n_cols + 7) // 8 * 8)), dtype=torch.int16, device="cuda")
    # 0: valid, 1: an occurrence differs, 2: overlap, 3: outside the file
    kind = torch.where(torch.rand(K, device="cuda", generator=gen) < faults, 1 + ints(3, K), 0)
    for k0 in range(0, K, 1024):
        n = min(1024, K - k0)
        kd, r = kind[k0:k0 + n], torch.arange(n, device="cuda")
        key = torch.rand((n, ng), device="cuda", generator=gen)
        if rules:
            key += (torch.arange(ng, device="cuda") >= ng // 2).float()
            key[:, -1] = 3.0
        flip = torch.randint(0, W, (n, ng), device="cuda", generator=gen, dtype=torch.int32)
        table = key.argsort(dim=1).int()[:, grp] * W + ((off ^ flip[:, grp]) & ~(width - 1))
        pick = ints(v_of.numel(), n) if v_of.numel() else None
        if pick is not None:
            v, u = v_of[pick], u_of[pick]
            hit = kd == 2
            table[r[hit], v[hit]] = torch.minimum(table[r, u], P - width[v])[hit]
        v, far = ints(prog.n_vregs, n), (P + ints(64, n)).int()
        hit = kd == 3
        table[r[hit], v[hit]] = far[hit]
        rows = table.short().index_select(1, cols)
        if repeats.numel():
            c, step = repeats[ints(repeats.numel(), n)], 1 + ints(P - 1, n)
            hit = kd == 1
            rows[r[hit], c[hit]] = ((rows[r, c].long() + step) % P).short()[hit]
        out[k0:k0 + n, :n_cols] = rows
    return out.view(torch.uint16)


def _rules(prog):
    """Tuples on multiples of their width, vregs in two classes (the halves of the register file), the last two
    registers reserved."""
    P = prog.P
    return dict(vreg_align=prog.vreg_width, vreg_class=_classes(prog), class_ranges=[(0, P // 2), (P // 2, P)],
                reserved=[P - 2, P - 1], P=P)


def prepare(case, seed):
    progs = _programs(case)
    handles = [vl.Program(p) for p in progs]
    path = case["path"]
    state = dict(path=path, handles=handles, P=progs[0].P, n_banks=progs[0].B)
    columns = None
    if path == "dict":
        columns = _dict_first_op(case["shape"], case["seed"], case.get("n_instrs", 0), case.get("n_vregs", 0), case.get("loops", 0))
    rows = [_rows(p, case["K"], case["faults"], case["rules"], seed * 1009 + j, columns) for j, p in enumerate(progs)]
    if case["rules"]:
        handles[0].set_constraints(**_rules(progs[0]))
    if path in ("verify", "dict", "host", "until"):
        for h in handles:
            h.vl_liveness()
            h.vl_liveness_wait()
    if path == "host":
        host = torch.empty(rows[0].shape, dtype=torch.int16, pin_memory=True)
        host.copy_(rows[0].view(torch.int16))
        state.update(rows=host, out=np.zeros(case["K"], dtype=vl.VERDICT_DTYPE))
    else:
        state["rows"] = rows
        # one buffer for the verdicts of all programs, a part of it for each
        state["verdicts"] = torch.empty((len(progs), case["K"], 4), dtype=torch.int32, device="cuda")
        state["outs"] = list(state["verdicts"])
    if path == "until":
        state["batch_rows"] = case["batch_rows"]
    torch.cuda.synchronize()
    return state


def run(state):
    path, h = state["path"], state["handles"][0]
    if path == "verify":
        return h.vl_verify(state["rows"][0], state["outs"][0])
    if path == "step":
        h.vl_liveness()
        return h.vl_verify(state["rows"][0], state["outs"][0])
    if path == "dict":
        return h.vl_verify_dict(state["rows"][0], state["outs"][0])
    if path == "host":
        v = h.vl_verify_host(state["rows"], state["out"])
        return [v[f] for f in v.dtype.names]
    if path == "until":
        out, done, first = h.vl_verify_until_pass(state["rows"][0], state["batch_rows"])
        return [out, done, first]
    if path == "batch":
        vl.vl_liveness_batch(state["handles"])
        outs = vl.vl_verify_batch(state["handles"], state["rows"], state["outs"])
        rec, summary = vl.vl_resample_stats(outs, (1, 10, 100))
        return [state["verdicts"], rec["first_pass"].astype(np.int64), rec["n_pass"].astype(np.int64),
                [summary["n_cases"], summary["n_solved"], summary["sum_tries"], summary["max_tries"], *summary["pass_at"]]]
    # feedback; the conflict records come in no particular order: a reader sorts them by instruction
    h.vl_liveness()
    row = state["rows"][0][0]
    records, n, kinds, hist = h.vl_diagnose(row, n_banks=state["n_banks"])
    records = records[np.lexsort(records.T[::-1])].astype(np.int64)
    return [records, n, kinds, hist.astype(np.int64), h.vl_occupied_masks(row, state["P"])]


def work(case):
    """Candidate columns read once (2 bytes each), verdicts written once (16 bytes each), the program's operands
    read once where liveness is part of the pass; one comparison per column."""
    total_bytes = total_ops = 0
    for p in _programs(case):
        cols = p.n_operands
        if case["path"] == "dict":
            cols = len(_dict_first_op(case["shape"], case["seed"], case.get("n_instrs", 0), case.get("n_vregs", 0), case.get("loops", 0)))
        K = case["K"]
        if case["path"] == "until":     # rows up to the batch that is expected to hold a passing one
            K = min(K, max(case["batch_rows"], int(1.0 / max(1e-3, 1.0 - case["faults"]))))
        total_bytes += K * (2 * cols + 16)
        total_ops += K * cols
        if case["path"] in ("step", "batch", "feedback"):
            total_bytes += 4 * (p.n_operands + p.n_instrs)
        if case["path"] == "feedback":  # the masks: one byte per instruction and register, and the violation kinds
            total_bytes += p.n_instrs * (p.P + 1)
    return {"bytes": total_bytes, "flops": total_ops}


def tolerance(case):
    return "exact"
