"""Host side of the library against the oracle: registry, trace, classification and schedule must be
bit-exact (compared as exported blobs); error paths return codes, never crash.  No GPU needed."""
import ctypes
import os
import re
import struct
import subprocess
import sys
from dataclasses import replace

import numpy as np
import pytest

import seeded_inputs as si
from conftest import MACHINE
from oracle import policy, trace, validate
from paper_2609_06172_b200 import binding as tb
from paper_2609_06172_b200 import build as tbuild
from paper_2609_06172_b200.session import Session


@pytest.fixture(scope="module", autouse=True)
def _built():
    tbuild.build()


def pack_trace(ops):
    out = []
    for o in ops:
        out.append(struct.pack("<IQiIQQI", o.step, o.site, o.layer, o.kind, o.flops, o.hbm, len(o.acc)))
        out += [struct.pack("<IIQ", *a) for a in o.acc]
    return b"".join(out)


def oracle_blobs(lay, bits=15, expert_counts=None, budget=None):
    ops, steps = trace.run_trace(lay, expert_counts=expert_counts)
    pl = policy.plan(lay.tensors, ops, steps, policy.Machine(**MACHINE), budget or lay.budget, bits)
    return ops, steps, pl.blobs()


def test_library_exports_every_declared_symbol():
    hdr = open(os.path.join(os.path.dirname(tbuild.INCLUDE), "include", "tgp.h")).read()
    declared = set(re.findall(r"\b(tgp_[a-z_0-9]+)\s*\(", hdr))
    lib = ctypes.CDLL(tbuild.LIB)
    for name in declared:
        assert hasattr(lib, name), name
    assert declared == set(tb.exported_symbols())


@pytest.mark.parametrize("c", [1, 2, 3, 4])
def test_plan_bit_exact_dense_configs(c):
    lay = si.build_layout(si.CONFIGS[c])
    s = Session(lay, MACHINE)
    got = s.plan()
    ops, steps, want = oracle_blobs(lay)
    assert s.ctx.trace_export() == pack_trace(ops)
    for k in want:
        assert got[k] == want[k], k
    s.close()


def synthetic_expert_counts(cfg, rng):
    """Top-2 routing counts with a Zipf-like popularity (counts only; no forward pass involved)."""
    p = np.array([r ** -1.2 for r in range(1, cfg.E + 1)])
    p /= p.sum()
    out = np.zeros((1 + cfg.T, cfg.L, cfg.E), dtype=np.uint32)
    for k in range(1 + cfg.T):
        M = cfg.B * (cfg.S if k == 0 else 1)
        for l in range(cfg.L):
            for _ in range(M):
                e = rng.choice(cfg.E, size=2, replace=False, p=p)
                out[k, l, e] += 1
    return out


def test_plan_bit_exact_moe_reduced_and_full_shape():
    rng = np.random.default_rng(5)
    small = replace(si.CONFIGS[5], L=3, B=4, S=8, T=6, TK=4)
    lay = si.build_layout(small, budget=3 << 30)
    ec = synthetic_expert_counts(small, rng)
    s = Session(lay, MACHINE, router_bias=si.router_bias(small))
    got = s.plan(expert_counts=ec)
    ops, steps, want = oracle_blobs(lay, expert_counts=ec)
    assert s.ctx.trace_export() == pack_trace(ops)
    for k in want:
        assert got[k] == want[k], k
    validate.check(lay.tensors, ops, steps, lay.budget, got)
    s.close()
    # full config-5 shape and budget, every expert hit in every step (the worst case for the link)
    cfg = si.CONFIGS[5]
    lay = si.build_layout(cfg)
    ec = np.zeros((1 + cfg.T, cfg.L, cfg.E), dtype=np.uint32)
    ec[0] = cfg.B * cfg.S * 2 // cfg.E
    ec[1:] = cfg.B * 2 // cfg.E
    s = Session(lay, MACHINE, router_bias=si.router_bias(cfg))
    got = s.plan(expert_counts=ec)
    ops, steps, want = oracle_blobs(lay, expert_counts=ec)
    for k in want:
        assert got[k] == want[k], k
    s.close()


@pytest.mark.parametrize("bits", [0, tb.BIT_A, tb.BIT_P, tb.BIT_A | tb.BIT_P, tb.BIT_ZC, 7, tb.BIT_W, 15])
def test_plan_bit_exact_under_ablation_bits(bits):
    lay = si.build_layout(si.CONFIGS[1])
    s = Session(lay, MACHINE)
    try:
        got = s.plan(bits=bits)
    except tb.TgpError as e:
        assert e.code == tb.E_BUDGET_TOO_SMALL
        with pytest.raises(policy.PlanError):
            oracle_blobs(lay, bits)
        return
    ops, steps, want = oracle_blobs(lay, bits)
    for k in want:
        assert got[k] == want[k], (bits, k)
    validate.check(lay.tensors, ops, steps, lay.budget, got)
    s.close()


@pytest.mark.parametrize("first_step", [0, 2, 20])
def test_windowed_pin_reservation_is_bit_exact_and_moves_fewer_bytes(first_step):
    """A long decode on a small model whose KV tiles (32 KiB) hold two 16 KiB weight blocks: the slots of the tiles born
    in later decode steps house unpinned weight blocks until then.  Library and oracle agree bit for bit, with the bit
    on and off, for the whole run and for a tail plan; the windowed plan passes the validator and moves fewer bytes."""
    cfg = replace(si.CONFIGS[1], B=4, S=30, T=40, TK=16)
    lay = si.build_layout(cfg, cap=16 << 10)
    ops, steps = trace.run_trace(lay)
    mach = policy.Machine(**MACHINE)
    totals = {}
    for bits in (7, 15):
        s = Session(lay, MACHINE)
        got = s.plan(bits=bits)
        if first_step:
            s.ctx.replan_begin(first_step)
            s.ctx.replan_wait()
            got = s.ctx.plan_blobs(tail=True)
            want = policy.plan_tail(lay.tensors, ops, steps, mach, lay.budget, first_step, bits=bits).blobs()
        else:
            want = policy.plan(lay.tensors, ops, steps, mach, lay.budget, bits=bits).blobs()
        for k in want:
            assert got[k] == want[k], (bits, k)
        validate.check(lay.tensors, ops, steps, lay.budget, got, first_step=first_step)
        totals[bits] = int(np.frombuffer(got["totals"], dtype="<u8").reshape(-1, 4)[:, 0].sum())
        s.close()
    if first_step == 0:
        assert totals[15] < totals[7]
    else:
        assert totals[15] <= totals[7]


def test_library_plan_passes_the_validator_config_2():
    lay = si.build_layout(si.CONFIGS[2])
    s = Session(lay, MACHINE)
    got = s.plan(T=8)
    ops, steps = trace.run_trace(lay, n_decode=8)
    validate.check(lay.tensors, ops, steps, lay.budget, got)
    s.close()


def test_schedule_is_independent_of_the_pool_address():
    lay = si.build_layout(si.CONFIGS[1])
    a = Session(lay, MACHINE, pool_base=1 << 30)
    b = Session(lay, MACHINE, pool_base=(7 << 40) + 512 * 12345)
    assert a.plan() == b.plan()
    assert a.ctx.tensor_identity(17) == b.ctx.tensor_identity(17)
    a.close(), b.close()


def test_trace_recorded_through_the_c_calls_equals_model_trace():
    lay = si.build_layout(si.CONFIGS[1])
    ops, steps = trace.run_trace(lay, n_decode=2)
    s = Session(lay, MACHINE)
    s.ctx.trace_begin()
    for (kind, first, count) in steps:
        s.ctx.trace_step(kind)
        for o in ops[first:first + count]:
            s.ctx.trace_op(o.site, o.layer, o.kind, o.flops, o.hbm, o.acc)
    s.ctx.trace_end()
    s.ctx.plan()
    manual = s.ctx.plan_blobs()
    assert s.plan(T=2) == manual
    s.close()


def test_registry_lookup_identity_and_errors():
    ctx = tb.Ctx(**MACHINE)
    buf = np.zeros(1 << 16, dtype=np.uint8)
    base = (buf.ctypes.data + 511) // 512 * 512
    pool = ctx.pool_register(base, 32768, tb.POOL_PLAIN)
    a = ctx.tensor_register(pool, 0, 1000, 0xABC, 0, 2, tb.T_READONLY)
    b = ctx.tensor_register(pool, 4096, 2048, 0xABC, 0, 3, tb.T_READONLY)
    c = ctx.tensor_register(pool, 1024, 512, 0xDEF, 1, 13, tb.T_MUTABLE)       # out of address order
    assert ctx.tensor_lookup(base + 999) == (a, 999)
    assert ctx.tensor_lookup(base + 4096 + 7) == (b, 7)
    assert ctx.tensor_lookup(base + 1024) == (c, 0)
    assert ctx.tensor_identity(a) == (0xABC, 0) and ctx.tensor_identity(b) == (0xABC, 1) and ctx.tensor_identity(c) == (0xDEF, 0)
    for args, code in [((pool, 512, 1024, 1, 0, 2, tb.T_READONLY), tb.E_OVERLAP),        # into a and c
                       ((pool, 3584, 1024, 1, 0, 2, tb.T_READONLY), tb.E_OVERLAP),       # into b
                       ((pool, 32768 - 512, 1024, 1, 0, 2, tb.T_READONLY), tb.E_RANGE),
                       ((pool, 100, 8, 1, 0, 2, tb.T_READONLY), tb.E_INVAL),             # unaligned
                       ((pool + 5, 0, 8, 1, 0, 2, tb.T_READONLY), tb.E_INVAL),
                       ((pool, 8192, 8, 1, 0, 2, 3), tb.E_INVAL)]:
        with pytest.raises(tb.TgpError) as ei:
            ctx.tensor_register(*args)
        assert ei.value.code == code
    for addr in (base + 1000, base + 3000, base - 1, base + 40000):
        with pytest.raises(tb.TgpError) as ei:
            ctx.tensor_lookup(addr)
        assert ei.value.code == tb.E_RANGE
    with pytest.raises(tb.TgpError) as ei:
        ctx.pool_register(base + 512, 1024, tb.POOL_PLAIN)
    assert ei.value.code == tb.E_OVERLAP
    # trace errors
    with pytest.raises(tb.TgpError):
        ctx.plan()                                               # nothing traced
    ctx.trace_begin()
    ctx.trace_step(tb.PREFILL)
    for acc, code in [([(99, tb.R, 8)], tb.E_UNKNOWN_TENSOR), ([(a, tb.W, 8)], tb.E_INVAL), ([(a, tb.R, 8), (a, tb.R, 8)], tb.E_INVAL)]:
        with pytest.raises(tb.TgpError) as ei:
            ctx.trace_op(1, 0, 2, 10, 10, acc)
        assert ei.value.code == code
    ctx.trace_op(1, 0, 2, 10, 10, [(a, tb.R, 1000)])
    ctx.trace_end()
    with pytest.raises(tb.TgpError) as ei:
        ctx.plan()                                               # no budget
    assert ei.value.code == tb.E_STATE
    ctx.set_budget(1024)
    with pytest.raises(tb.TgpError) as ei:
        ctx.plan()
    assert ei.value.code == tb.E_BUDGET_TOO_SMALL
    with pytest.raises(tb.TgpError) as ei:
        ctx.plan_export(tb.X_COMMANDS)
    assert ei.value.code == tb.E_NO_PLAN
    ctx.set_budget(4096)
    ctx.plan()
    assert len(ctx.plan_export(tb.X_COMMANDS)) == 45
    with pytest.raises(tb.TgpError):
        ctx.tensor_register(pool, 16384, 512, 1, 0, 2, tb.T_READONLY)     # registry frozen after tracing
    # stepping without a device binding is a state error, not a crash
    with pytest.raises(tb.TgpError) as ei:
        ctx.step(tb.PREFILL, np.zeros(4, np.int32), 1, 4, 1 << 20, None, None, None)
    assert ei.value.code == tb.E_STATE
    ctx.close()


def test_model_bind_rejects_bad_shapes_and_roles():
    lay = si.build_layout(si.CONFIGS[1])
    s = Session(lay, MACHINE)
    bad = tb.ModelCfg(4, 256, 4, 3, 64, 1024, 4096, 0, 0, 1, 48, 16, 10000.0, 1e-5)          # Hq % Hkv != 0
    with pytest.raises(tb.TgpError):
        s.ctx.model_bind(bad, s.roles)
    long_ctx = tb.ModelCfg(4, 256, 4, 4, 64, 1024, 4096, 0, 0, 1, 65 * 16, 16, 10000.0, 1e-5)   # 65 tiles > 64
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.model_bind(long_ctx, s.roles)
    assert ei.value.code == tb.E_TOO_LARGE
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.model_bind(s.cfg, s.roles + [s.roles[0]])
    assert ei.value.code == tb.E_INVAL
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.model_trace(40, 16)                                # S + T beyond max_len
    assert ei.value.code == tb.E_INVAL
    s.close()


def test_step_refuses_host_tokens_outside_the_vocabulary_before_touching_a_device():
    """A host token id outside [0, V) would send the embedding gather past its table; tgp_step() must refuse it at the
    boundary (no GPU involved: the check comes before the engine is looked at), and an op whose tensor has no model role
    must be a mismatch code, not a crash."""
    lay = si.build_layout(si.CONFIGS[1])
    s = Session(lay, MACHINE)
    s.plan(T=1)
    cfg = lay.cfg
    dummy = np.zeros(16, dtype=np.float32)                      # stands for the logits pointer; never written without a workspace
    for bad in (-1, cfg.V, 2 ** 31 - 1):
        tok = np.zeros((cfg.B, cfg.S), dtype=np.int32)
        tok[0, 5] = bad
        with pytest.raises(tb.TgpError) as ei:
            s.ctx.step(tb.PREFILL, tok, cfg.B, cfg.S, dummy, None, None, None)
        assert ei.value.code == tb.E_INVAL and "vocabulary" in str(ei.value)
    ok = np.full((cfg.B, cfg.S), cfg.V - 1, dtype=np.int32)
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.step(tb.PREFILL, ok, cfg.B, cfg.S, dummy, None, None, None)
    assert ei.value.code == tb.E_STATE                          # legal tokens get as far as "no workspace bound"
    s.close()


def test_replan_from_a_timing_log_is_bit_exact_and_changes_classes():
    """Runtime monitor: the same integer log of kernel times fed to both planners gives the same schedule; an op whose
    kernel ran longer than its bytes take on the link stops being link-bound, and its tensors lose their pin score."""
    lay = si.build_layout(si.CONFIGS[1])
    ops, steps = trace.run_trace(lay)
    rng = np.random.default_rng(11)
    # synthetic log: most ops fast (1 us), a third not measured (0), norm ops slow (20 us >> 512 B over the link)
    ns = np.where(rng.random(len(ops)) < 0.33, 0, 1000).astype(np.uint64)
    for i, o in enumerate(ops):
        if o.kind == trace.OP_RMSNORM:
            ns[i] = 20000
    s = Session(lay, MACHINE)
    base = s.plan()
    s.ctx.set_measured_times(ns)
    s.ctx.plan()
    got = s.ctx.plan_blobs()
    want = policy.plan(lay.tensors, ops, steps, policy.Machine(**MACHINE), lay.budget, measured_ns=ns.tolist()).blobs()
    assert got == want
    validate.check(lay.tensors, ops, steps, lay.budget, got)
    assert got["classes"] != base["classes"]
    norm_ops = [i for i, o in enumerate(ops) if o.kind == trace.OP_RMSNORM]
    assert all(base["classes"][i] == policy.CLS_LINK for i in norm_ops) and all(got["classes"][i] != policy.CLS_LINK for i in norm_ops)
    gain = lay.blocks(si.K_G1, 0)[0].tid
    crit = lambda blobs, t: blobs["tensors"][t * 10]
    assert crit(base, gain) == 1 and crit(got, gain) == 0
    # clearing the log restores the analytic plan; a log of the wrong length is refused
    s.ctx.set_measured_times(None)
    s.ctx.plan()
    assert s.ctx.plan_blobs() == base
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.set_measured_times(ns[:-1])
    assert ei.value.code == tb.E_STATE
    s.close()


@pytest.mark.parametrize("c,first_step", [(1, 1), (1, 9), (2, 3)])
def test_tail_replan_in_the_middle_of_a_run_is_bit_exact(c, first_step):
    """Runtime monitor, second half: the steps from a boundary on are planned again, as a trace of their own, from the
    timing log so far, on a helper thread.  The same integer log fed to the oracle's tail planner gives the same blobs;
    the tail plan passes the validator started from an empty arena with the earlier steps' writes in the pool."""
    cfg = si.CONFIGS[c] if c == 1 else replace(si.CONFIGS[c], T=6)
    lay = si.build_layout(cfg)
    ops, steps = trace.run_trace(lay)
    first_op = steps[first_step][1]
    rng = np.random.default_rng(first_step)
    ns = np.zeros(len(ops), dtype=np.uint64)
    ns[:first_op] = rng.integers(500, 40000, first_op)                    # measured so far
    # ops still to come: the time of the same op in the last measured step of the same kind, where there is one
    if first_step >= 2:
        o0, n = steps[first_step - 1][1], steps[first_step - 1][2]
        for k in range(first_step, len(steps)):
            if steps[k][2] == n:
                ns[steps[k][1]: steps[k][1] + n] = ns[o0: o0 + n]
    s = Session(lay, MACHINE)
    base = s.plan(T=cfg.T)
    s.ctx.replan_begin(first_step, ns)
    s.ctx.replan_wait()
    got = s.ctx.plan_blobs(tail=True)
    assert s.ctx.plan_blobs() == base                                     # the plan in use is untouched until the commit
    want = policy.plan_tail(lay.tensors, ops, steps, policy.Machine(**MACHINE), lay.budget, first_step, measured_ns=ns.tolist()).blobs()
    assert got == want
    validate.check(lay.tensors, ops, steps, lay.budget, got, first_step=first_step)
    assert len(got["classes"]) == len(ops) - first_op and len(got["totals"]) == 32 * (len(steps) - first_step)
    # without a log the tail plan is the analytic one
    s.ctx.set_measured_times(None)
    s.ctx.plan()
    s.ctx.replan_begin(first_step)
    s.ctx.replan_wait()
    assert s.ctx.plan_blobs(tail=True) == policy.plan_tail(lay.tensors, ops, steps, policy.Machine(**MACHINE), lay.budget, first_step).blobs()
    # call-order and argument errors are codes
    for bad in (0, len(steps)):
        with pytest.raises(tb.TgpError) as ei:
            s.ctx.replan_begin(bad)
        assert ei.value.code == tb.E_INVAL
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.replan_begin(first_step, ns[:-1])
    assert ei.value.code == tb.E_INVAL
    with pytest.raises(tb.TgpError) as ei:
        s.ctx.replan_commit()                                             # no engine without a device
    assert ei.value.code == tb.E_STATE
    s.close()


def _resident_of(blobs, n_tensors, first_op):
    """tensor -> arena offset of the pins of a plan that are on the device when op first_op starts: placed before it, or
    never placed at all (kept by that plan itself)."""
    P = validate.parse(blobs, n_tensors)
    placed = {}
    for (seq, kind, t, nb, po, ao, w, f, r) in P["cmds"]:
        if kind != validate.CMD_D2H:
            placed.setdefault((t, ao), f)
    return {t: o for t, o in P["pins"] if placed.get((t, o), -1) < first_op}


@pytest.mark.parametrize("c,first_step", [(1, 2), (1, 9), (2, 3)])
def test_tail_replan_that_keeps_the_resident_pins_is_bit_exact(c, first_step):
    """With tgp_set_replan_keep the tail plan keeps the pinned tensors that are on the device at the boundary: same blobs as
    the oracle's tail planner given that resident set, valid for a replay that starts with them resident, nothing of
    them placed again, fewer bytes in the first tail step than a tail that starts cold; with the switch off again the
    planner returns the cold tail."""
    cfg = si.CONFIGS[c] if c == 1 else replace(si.CONFIGS[c], T=8)
    lay = si.build_layout(cfg)
    ops, steps = trace.run_trace(lay)
    mach = policy.Machine(**MACHINE)
    rng = np.random.default_rng(10 + first_step)
    ns = np.zeros(len(ops), dtype=np.uint64)
    ns[:steps[first_step][1]] = rng.integers(500, 40000, steps[first_step][1])
    s = Session(lay, MACHINE)
    base = s.plan(T=cfg.T)
    s.ctx.replan_begin(first_step, ns)
    s.ctx.replan_wait()
    cold = s.ctx.plan_blobs(tail=True)
    s.ctx.set_replan_keep(True)
    s.ctx.replan_begin(first_step, ns)
    s.ctx.replan_wait()
    got = s.ctx.plan_blobs(tail=True)
    res = _resident_of(base, len(lay.tensors), steps[first_step][1])
    assert res
    want = policy.plan_tail(lay.tensors, ops, steps, mach, lay.budget, first_step, measured_ns=ns.tolist(), resident=res).blobs()
    assert got == want
    validate.check(lay.tensors, ops, steps, lay.budget, got, first_step=first_step, resident=res)
    P = validate.parse(got, len(lay.tensors))
    off = dict(P["pins"])
    kept = {t for t, o in res.items() if off.get(t) == o}
    assert kept and not ({c[2] for c in P["cmds"] if c[1] != validate.CMD_D2H} & kept)
    assert validate.parse(got, len(lay.tensors))["totals"][0][0] < validate.parse(cold, len(lay.tensors))["totals"][0][0]
    s.ctx.set_replan_keep(False)
    s.ctx.replan_begin(first_step, ns)
    s.ctx.replan_wait()
    assert s.ctx.plan_blobs(tail=True) == cold                              # the switch is per plan: off again, the cold tail again
    s.close()


def test_measured_time_link_test_by_hand():
    toy = policy.Machine(1000, 100, 10, 10)            # link 10 B/s
    # 100 bytes over the link take 10 s: a 9 s kernel is link-bound, a 10 s or 11 s kernel is not
    assert policy.classify(5000, 300, 100, toy, measured_ns=9_000_000_000) == policy.CLS_LINK
    assert policy.classify(5000, 300, 100, toy, measured_ns=10_000_000_000) == policy.CLS_COMPUTE
    assert policy.classify(100, 600, 100, toy, measured_ns=11_000_000_000) == policy.CLS_HBM
    assert policy.classify(5000, 300, 100, toy, measured_ns=0) == policy.CLS_LINK          # no measurement: analytic


def test_aliased_host_pool_shares_pages_between_layer_groups_only():
    """The fallback for pools larger than the host can page-lock: layers l and l + phys share physical pages, everything
    else (embedding, head, KV tiles) stays private, and the virtual layout is the ordinary one."""
    from paper_2609_06172_b200.runner import AliasedPool
    cfg = replace(si.CONFIGS[1], L=6, d=1024, F=4096, Hq=16, Hkv=16)   # layer regions are multiples of the page size here
    lay = si.build_layout(cfg)
    try:
        p = AliasedPool(lay, 2)
    except ValueError as ex:
        pytest.skip(f"layout not page-aligned on this machine: {ex}")
    a = p.numpy()
    assert a.size == lay.pool_bytes and p.phys_bytes - lay.pool_bytes + 4 * p.layer_bytes in range(0, 4096)      # fresh pages read as zero
    w = [t for t in lay.tensors if t.kind == si.K_WQ]
    by_layer = {t.layer: t for t in w}
    a[by_layer[1].pool_off] = 7                                     # layer 1 ...
    assert a[by_layer[3].pool_off] == 7 and a[by_layer[5].pool_off] == 7        # ... is layers 3 and 5
    assert a[by_layer[0].pool_off] == 0 and a[by_layer[2].pool_off] == 0
    kv = [t for t in lay.tensors if t.kind == si.K_KT]
    a[kv[0].pool_off] = 9
    assert sum(int(a[t.pool_off] == 9) for t in kv) == 1            # KV tiles are private
    emb = next(t for t in lay.tensors if t.kind == si.K_EMBED)
    a[emb.pool_off + 5] = 3
    assert int((a[:emb.size] == 3).sum()) == 1 and all(int(a[t.pool_off + 5]) != 3 for t in w)
    p.close()


@pytest.mark.parametrize("M,n,K,family", [(12, 12000, 1000, 0), (16, 8065, 2056, 0), (9, 32000, 4104, 0), (12, 12000, 2048, 2), (16, 8065, 2048, 2), (16, 8064, 4096, 1), (17, 64, 1000, 2),
                                          (12, 12000, 1024, 0), (9, 18944, 1504, 0), (9, 8065, 1536, 2), (9, 18945, 64, 2)])
def test_products_of_9_to_16_rows_take_the_tcgen05_kernel_only_where_it_is_ahead_and_as_exact(M, n, K, family):
    """K not a multiple of 32 stays with the CUDA cores (key 0, launched alone), whose sums are closer to 64 bits; K below 1536 on fewer
    tiles of 128 rows than SMs (148) with the split-K kernel, which is faster."""
    assert tb.k_gemm_group_key(M, n, K) >> 24 == family


def test_addresses_of_every_kind_of_argument_alone_and_in_arrays():
    import torch

    class Stream:
        cuda_stream = 77

    class Holder:
        def __init__(self, **kw):
            self.__dict__.update(kw)

    a, t = np.arange(12, dtype=np.float32), torch.zeros(5)
    cases = [(None, None), (4096, 4096), (True, True), (a, a.ctypes.data), (a[3:], a.ctypes.data + 12), (t, t.data_ptr()), (t[2:], t.data_ptr() + 8),
             (torch.nn.Parameter(t), t.data_ptr()), (Stream(), 77), (Holder(cuda_stream=5), 5), (Holder(data_ptr=lambda: 9, cuda_stream=5), 9), (Holder(cuda_stream=6), 6)]
    for _ in range(2):                                     # the first use of a type and the next
        for x, want in cases:
            assert tb._ptr(x) == want
    for bad in ("x", 1.5, Holder(), [1]):
        for _ in range(2):
            with pytest.raises(TypeError):
                tb._ptr(bad)
    assert [v for v in tb._pointers([x for x, _ in cases])] == [w if w is None else int(w) for _, w in cases]
    assert list(tb._pointers([t[1:], t])) == [t.data_ptr() + 4, t.data_ptr()] and len(tb._pointers([])) == 1
    assert list(tb._pointers((Holder(cuda_stream=3), Holder(data_ptr=lambda: 4)))) == [3, 4]


def test_the_address_of_an_object_is_its_own_not_that_of_its_type():
    class Arg:                                             # a stream, and a buffer where it has one
        cuda_stream = 7

    buffer = Arg()
    buffer.data_ptr = lambda: 9
    for x, want in ((Arg(), 7), (buffer, 9), (Arg(), 7)):
        assert tb._ptr(x) == want
    assert list(tb._pointers([Arg(), buffer])) == [7, 9]


def test_what_is_kept_for_addresses_and_arrays_is_bounded():
    for i in range(200):
        assert tb._ptr(type("Number", (int,), {})(i)) == i
        assert len(tb._pointers([8] * i)) == max(1, i) and tb._pointers([8] * i)[0] == (8 if i else None)
    assert len(tb._ACCESSORS) <= 64 and len(tb._POINTER_ARRAYS) <= 64


def test_pointer_lists_have_the_length_the_library_is_told():
    """Lists of another length than the first of a call: NULL for what is missing, which the library refuses where it would use it, an
    IndexError for more; any iterable will do."""
    for ka, va, n in (tb._tile_arrays([16, 32, 48], [64, 80]), tb._tile_arrays((16, 32, 48), (v for v in (64, 80)))):
        assert n == 3 and list(ka) == [16, 32, 48] and list(va) == [64, 80, None]
    with pytest.raises(IndexError):
        tb._tile_arrays([16], [64, 80])
    # (no rows, or a call that is refused: nothing is launched)
    group = lambda outs: tb.k_gemm_group(16, [16, 32, 48], outs, 0, [8, 8, 8], 64, [8, 8, 8])
    group([64, 80, 96])
    group(v for v in (64, 80, 96))
    with pytest.raises(tb.TgpError) as e:
        group([64, 80])
    assert e.value.code == tb.E_INVAL
    with pytest.raises(IndexError):
        group([64, 80, 96, 112])


def test_null_tiles_are_refused_where_the_call_uses_them():
    mc = tb.ModelCfg()
    mc.B, mc.Hq, mc.Hkv, mc.Dh, mc.TK, mc.max_len = 1, 2, 1, 64, 16, 48
    calls = [lambda k, v, B, q, p: tb.k_rope_kv(16, 16, 16, 16, k, v, 16, 16, mc, B, q, p), lambda k, v, B, q, p: tb.k_attn(16, k, v, 16, mc, B, q, p)]
    for call in calls:
        for k, v, q, p in (([16, None, 48], [16, 32, 48], 32, 10), ([16, 32, 48], [16, 32], 1, 47), ([16, 32, 48], [16, None, 48], 1, 16), ([16, 32, 48], [], 48, 0)):
            with pytest.raises(tb.TgpError) as e:
                call(k, v, 1, q, p)
            assert e.value.code == tb.E_INVAL
        call([None, 32], [None, None], 0, 1, 16)            # (no sequence: nothing is used, nothing launched)
    for k, v, p in (([16], [None], 0), ([16, 32], [16], 16), ([None, 32], [16, 32], 20)):
        with pytest.raises(tb.TgpError) as e:
            tb.k_attn_decode_static(16, k, v, 16, mc, 1, p)
        assert e.value.code == tb.E_INVAL


def test_calls_without_ctypes_take_and_refuse_what_the_general_path_does(monkeypatch):
    """The extension's functions leave what they do not know to the general path, having done nothing, and return the library's code for the rest: the same
    outcome with and without them, for arguments of every kind (no rows, or refused: nothing is launched)."""
    import torch
    t, a = torch.zeros(64), np.zeros(64, dtype=np.float32)
    mc = tb.ModelCfg()
    mc.B, mc.Hq, mc.Hkv, mc.Dh, mc.TK, mc.max_len = 1, 2, 1, 64, 16, 48

    class Holder:
        cuda_stream = 0

    def outcome(f):
        try:
            return f()
        except tb.TgpError as e:
            return "TgpError", e.code, str(e)
        except Exception as e:
            return type(e), str(e)

    calls = []
    for p in (None, 16, True, t, torch.nn.Parameter(t), t[3:], a, "x", 1.5, Holder(), [1]):
        calls += [lambda p=p: tb.k_embed(p, 16, p, 0, 8, 8), lambda p=p: tb.k_rmsnorm(p, 8, p, 16, 0, 8, 1e-5, 0), lambda p=p: tb.k_gemm(p, 16, p, 0, 8, 8, 8, 0, False),
                  lambda p=p: tb.k_gemm(16, p, 16, 1, 8, 12, 8, 0, 0), lambda p=p: tb.k_swiglu(p, p, 16, 0), lambda p=p: tb.k_argmax(p, 16, 0, 8), lambda p=p: tb.k_rmsnorm(16, 8, 16, 16, 0, 8, 1e-5, p),
                  lambda p=p: tb.k_gemm_group(p, [16, p], [16, 16], 0, [8, 8], 64, [8, 8]), lambda p=p: tb.k_attn(16, [p], [16], 16, mc, 0, 1, 0, p)]
    for n in (0, np.uint32(0), 0.0, True, None, "0", -1 << 32, 1 << 32):
        calls += [lambda n=n: tb.k_embed(16, 16, 16, n, 8, 8) if n is not True else None, lambda n=n: tb.k_rmsnorm(16, 8, 16, 16, n, 8, 1e-5) if n is not True else None, lambda n=n: tb.k_gemm(16, 16, 16, 0, 8, 8, 8, 0, n),
                  lambda n=n: tb.k_gemm_group(16, [16], [16], 0, [n], 64, [8]), lambda n=n: tb.k_rope_kv(16, 16, 16, 16, [16], [16], 16, 16, mc, 0, 1, n), lambda n=n: tb.k_rmsnorm(16, 8, 16, 16, 0, 8, n)]
    for k, v in (([], []), ([16], (32,)), ((16, 32), [16]), ([16], [16, 32]), (range(2), [16, 32]), ([16] * 300, [16] * 300), (t.tolist()[:1], [16]), (16, 16)):
        calls += [lambda k=k, v=v: tb.k_attn(16, k, v, 16, mc, 0, 1, 0), lambda k=k, v=v: tb.k_rope_kv(16, 16, 16, 16, k, v, 16, 16, mc, 0, 1, 0),
                  lambda k=k, v=v: tb.k_gemm_group(16, k, v, 0, [8] * 2, 64, [8] * 2), lambda k=k, v=v: tb.k_gemm_group(16, [16, 16], [16, 16], 0, k, 64, v)]
    for c in (None, 16, tb.Machine(), a):
        calls += [lambda c=c: tb.k_attn(16, [16], [16], 16, c, 0, 1, 0), lambda c=c: tb.k_rope_kv(16, 16, 16, 16, [16], [16], 16, 16, c, 0, 1, 0)]
    calls.append(lambda: tb.k_gemm(A=16, W=16, Cout=16, M=0, n=8, K=8, ldc=8, col0=0, accumulate=False, stream=None))
    calls.append(lambda: tb.k_gemm(16, 16))
    tb.lib()
    assert tb._fast.__name__.endswith("_fastcall")
    assert tb._fast.gemm(t, 16, 16, 0, 8, 8, 8, 0, False, None) == 0 and tb._fast.gemm(a, 16, 16, 0, 8, 8, 8, 0, False, None) is None
    fast = [outcome(f) for f in calls]
    monkeypatch.setattr(tb, "_fast", tb._General())
    monkeypatch.setattr(tb._General, "__getattr__", lambda self, name: lambda *args: None)
    assert fast == [outcome(f) for f in calls]
    assert sum(o is None for o in fast) > 40 and sum(isinstance(o, tuple) for o in fast) > 40


def test_lists_that_change_while_their_addresses_are_read_are_left_to_the_general_path():
    """An active function mode (torch.device() installs one) makes a tensor's data_ptr() run Python, which may do anything to the list at hand, give the call an
    exception, or call the library again: nothing that is gone is read.  In a process of its own, whose end says so."""
    code = """
import torch
from torch.overrides import TorchFunctionMode
from paper_2609_06172_b200 import binding as tb
tb.lib()
assert tb._fast.__name__.endswith("_fastcall")
mc = tb.ModelCfg()
mc.B, mc.Hq, mc.Hkv, mc.Dh, mc.TK, mc.max_len = 1, 2, 1, 64, 16, 256

class Mode(TorchFunctionMode):
    def __init__(self, at, act):
        super().__init__()
        self.n, self.at, self.act = 0, at, act
    def __torch_function__(self, f, types, args=(), kwargs=None):
        self.n += 1
        if self.n == self.at:
            self.act()
        return f(*args, **(kwargs or {}))

def swap(x):
    x[:] = [torch.zeros(8) for _ in range(4)] + [16] * 4

def nested():
    assert tb._fast.gemm_group(16, [torch.zeros(8)] * 2, [16] * 2, 0, [8] * 2, 64, [8] * 2, 0, None) == 0
    for i in range(20):                                       # types that fill the table of known ones while one is being looked at
        tb._fast.swiglu(type("T%d" % i, (torch.Tensor,), {})(), 16, 16, 0, None)

for act in (list.clear, list.pop, swap, lambda x: x.extend(x), lambda x: nested()):
    for at in range(1, 8):
        for call in (lambda x: tb._fast.gemm_group(16, x, [16] * 8, 0, [8] * 8, 64, [8] * 8, 0, None), lambda x: tb._fast.gemm_group(16, [16] * 8, x, 0, [8] * 8, 64, [8] * 8, 0, None),
                     lambda x: tb._fast.attn(16, x, [16] * 8, 16, mc, 0, 1, 0, None, None), lambda x: tb._fast.rope_kv(16, 16, 16, 16, [16] * 8, x, 16, 16, mc, 0, 1, 0, None)):
            x = [torch.zeros(8) for _ in range(8)]
            with Mode(at, lambda: act(x)):
                rc = call(x)
            assert rc in ((0,) if len(x) == 8 else (None,)), (act, at, rc)

def interrupt():
    raise KeyboardInterrupt
for act, out in ((lambda: 1 / 0, ZeroDivisionError), (interrupt, KeyboardInterrupt)):
    x = [torch.zeros(8) for _ in range(8)]
    try:
        with Mode(2, act):
            rc = tb.k_gemm_group(16, x, [16] * 8, 0, [8] * 8, 64, [8] * 8)
    except KeyboardInterrupt as e:
        assert out is KeyboardInterrupt
    else:
        assert out is ZeroDivisionError and rc is None        # raised once: the general path has taken the call
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(tb.__file__)))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=root)
    assert r.returncode == 0, (r.returncode, r.stderr)


@pytest.mark.parametrize("cc", ["false", "/nonexistent/cc"])
def test_a_machine_that_cannot_build_the_extension_still_builds_the_library(cc, monkeypatch, tmp_path):
    """ctypes serves every call, so a missing C compiler is a warning; an extension of an earlier build does not stay beside a newer library."""
    old = tmp_path / "_fastcall.so"
    old.write_bytes(b"")
    os.utime(old, (0, 0))
    monkeypatch.setattr(tbuild, "FASTCALL", str(old))
    monkeypatch.setenv("CC", cc)
    assert tbuild.needs_build()
    with pytest.warns(RuntimeWarning, match="ctypes"):
        assert tbuild.build() == tbuild.LIB
    assert not old.exists() and os.path.exists(tbuild.LIB)
    monkeypatch.setenv("CC", "gcc")
    tbuild.build()
    assert old.stat().st_size and not tbuild.needs_build()
