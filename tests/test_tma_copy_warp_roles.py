"""The discrete model of the TMA kernel's hand-offs with its present roles: one copy warp, the compute
warps and two halo warps that both read the stage and write the ring, for a step and for the read-out, which
stores nothing: its compute warps arrive on OUT_FULL right after a pull and read the ring after that, while
the copy warp refills the stage.  Broken variants must be caught."""
import inspect

import pytest

import tests.test_tma_copy_warp_protocol as copy_warp
import tests.test_tma_protocol as model


def _runner():
    """model.run with a second halo warp: one more arrival on RING, one more reader of a stage"""
    src = inspect.getsource(model.run)
    for old, new in (('counts["R%d" % s] = C + 2', 'counts["R%d" % s] = C + 3'), ("nreaders = C + 1", "nreaders = C + 2")):
        assert src.count(old) == 1, old
        src = src.replace(old, new)
    return src


def _step(items, S, R, C, stall, mutation=None):
    prog = copy_warp.programs(items, S, R, C, stall, mutation if mutation in ("refill_before_store", "out_before_ring") else None)
    halo = prog.pop("halo")
    prog["halo0"], prog["halo1"] = halo, copy_warp.programs(items, S, R, C, stall)["halo"]
    return prog


def _readout(items, S, R, C, stall, mutation=None):
    prog = _step(items, S, R, C, stall)
    for c in range(C):
        P, k = [], 0
        for z0, z1 in items:
            for n in range(z1 - z0 + 2):
                s = k % S
                P += [("waitfull", s, k), ("read", s, k), ("ring_write", k % R, k)]
                if mutation == "out_before_read":
                    P.insert(-2, ("arrive", "OF%d" % s))
                P.append(("sync", "R%d" % s))
                if mutation != "out_before_read":
                    P.append(("arrive", "OF%d" % s))
                k += 1
                if n >= 2:
                    P += [("ring_read", (k - d) % R, k - d) for d in (3, 2, 1)]
        prog["compute%d" % c] = P
    prog["producer"] = [op for op in prog["producer"] if op[0] != "storeread"]
    if mutation == "refill_unasked":
        prog["producer"] = [op for op in prog["producer"] if not (op[0] == "sync" and op[1].startswith("OF"))]
        for c in range(C):
            prog["compute%d" % c] = [op for op in prog["compute%d" % c] if not (op[0] == "arrive" and op[1].startswith("OF"))]
    return prog


def _run(programs, seed, mutation=None, ring=None, **over):
    scope = dict(vars(model), programs=programs)
    exec(_runner(), scope)
    case = dict(model._random_case(seed), **over)
    if ring:
        case["R"] = ring
    scope["run"](seed=seed, mutation=mutation, **case)


@pytest.mark.parametrize("programs", [_step, _readout])
def test_two_halo_warps_random_interleavings(programs):
    for seed in range(300):
        _run(programs, seed)


@pytest.mark.parametrize("programs,mutation,ring", [(_step, "refill_before_store", None), (_step, "out_before_ring", None),
                                                    (_step, None, 3),
                                                    (_readout, "refill_unasked", None), (_readout, "out_before_read", None),
                                                    (_readout, None, 3)])
def test_broken_variants_are_caught(programs, mutation, ring):
    for seed in range(300):
        try:
            _run(programs, seed, mutation, ring, stall=False, timeout_prob=0)
        except (AssertionError, model.Deadlock):
            return
    pytest.fail("not caught")
