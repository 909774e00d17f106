"""Discrete model of the TMA kernel's hand-offs with one copy warp for loads and stores: the copy warp
arrives on RING(s) after a use's loads, syncs OUT_FULL(s) with the compute warps, stores the stage and
refills it.  Run over random interleavings, stalls and timeouts with the checks of the two-warp model
(no deadlock, no barrier lapped, no stage, output or ring race); broken variants must be caught."""
import pytest

import tests.test_tma_protocol as model


def programs(items, S, R, C, stall, mutation=None):
    prog = model_programs(items, S, R, C, stall, mutation if mutation in ("halo_arrives_ring", "out_before_ring") else None)
    uses = [(p, z0) for z0, z1 in items for p in range(z0 - 1, z1 + 1)]

    def load(k):
        return [("issue", k % S, k, stall and k == 0), ("arrive", "R%d" % (k % S))]

    P = [op for k in range(min(S, len(uses))) for op in load(k)]
    for k, (p, z0) in enumerate(uses):
        s = k % S
        refill = load(k + S) if k + S < len(uses) else []
        P.append(("sync", "OF%d" % s))
        if mutation == "refill_before_store":
            P += refill
        if p > z0:
            P.append(("storeread", s, k))
        if mutation != "refill_before_store":
            P += refill
    P += [("drainfull", q % S, q) for q in range(max(len(uses) - S, 0), len(uses))]
    prog["producer"] = P
    del prog["storer"]
    return prog


model_programs = model.programs


def test_copy_warp_protocol_random_interleavings(monkeypatch):
    monkeypatch.setattr(model, "programs", programs)
    for seed in range(1500):
        model.run(seed=seed, **model._random_case(seed))


@pytest.mark.parametrize("mutation", ["halo_arrives_ring", "out_before_ring", "refill_before_store"])
def test_broken_copy_warp_protocols_are_caught(monkeypatch, mutation):
    monkeypatch.setattr(model, "programs", programs)
    caught = 0
    for seed in range(400):
        case = dict(model._random_case(seed), stall=False, timeout_prob=0)
        try:
            model.run(seed=seed, mutation=mutation, **case)
        except (AssertionError, model.Deadlock):
            caught += 1
    assert caught > 0, mutation
