"""Waits of the fused training kernel (k_train_chain in rt_mlp.cu) on the CPU.

An mbarrier wait by parity is right only while its barrier is at most one
phase past the one awaited. The kernel's roles are written down here as their
waits and arrivals, in program order. For each role in turn every other role
runs as far as it can while that one is held at each of its waits (no role
chooses, so nothing can run further), and the awaited barrier must not have
completed a second phase by then; and all roles must end."""
import pytest


def roles(L, nc, nc0, tiles, ring):
    """{role: [("wait" | "sync" | "arrive", barrier, phase)]}, {barrier: arrivals of a phase}; arrivals count
    warps for what warps 0-7 arrive on, else threads."""
    passes = 2 * L - 1
    need = {"feat": 8, "done": 1, "stored": 1, "named": 8}
    for c in range(nc):
        need["chunk", c] = need["only", c] = 8 if nc == 1 else 4
    for s in range(ring):
        need["full", s] = need["empty", s] = 1
    ops = {}

    def w(role, bar, phase):
        ops.setdefault(role, []).append(("wait", bar, phase))

    def a(role, bar):
        ops.setdefault(role, []).append(("arrive", bar, 0))

    it = 0
    for _ in range(tiles):
        for p in range(passes):
            for _ in range(nc0 if p == 0 else nc):
                if it >= ring:
                    w("weights", ("empty", it % ring), it // ring - 1)
                a("weights", ("full", it % ring))
                it += 1
    it = stage = 0
    for t in range(tiles):
        for p in range(passes):
            if p == 0:
                w("mma", "feat", t)
            for kc in range(nc0 if p == 0 else nc):
                if p > 0:
                    w("mma", ("chunk", kc), stage)
                w("mma", ("full", it % ring), it // ring)
                a("mma", ("empty", it % ring))
                it += 1
            a("mma", "done")
            stage += p > 0
    stage = only = 0
    for t in range(tiles):
        for q in range(2 * L + 1):
            last = q in (L, 2 * L)
            if q == 0:
                w("store", "feat", t)
            for c in range(nc if q else 0):
                w("store", ("only" if last else "chunk", c), only if last else stage)
            only += last
            stage += q > 0 and not last
            a("store", "stored")
    for warp in range(8):
        r, g = f"epilogue {warp}", warp // 4
        chunks = range(0 if nc == 1 else g, nc, 2)
        nst = done = named = 0
        for t in range(tiles):
            if nst > 0:
                w(r, "stored", nst - 1)
            a(r, "feat")
            nst += 1
            for p in range(passes):
                w(r, "done", done)
                done += 1
                w(r, "stored", nst - 1)
                nst += 1
                for c in chunks:
                    a(r, ("only" if p in (L - 1, passes - 1) else "chunk", c))
                if p != L - 1:
                    continue
                for _ in range(2):   # around the head's gradients
                    a(r, "named")
                    ops[r].append(("sync", "named", named))
                    named += 1
                w(r, "stored", nst - 1)
                nst += 1
                for c in chunks:
                    a(r, ("only" if L == 1 else "chunk", c))
    return ops, need


def overtaken(ops, need):
    """Waits whose barrier can be two phases on: (role, barrier, phase, phases completed)."""
    bad = set()
    for held in ops:
        got = dict.fromkeys(need, 0)   # arrivals
        at = dict.fromkeys(ops, 0)

        def complete(bar):
            return got[bar] // need[bar]

        def run(role):
            moved = False
            while at[role] < len(ops[role]):
                kind, bar, phase = ops[role][at[role]]
                if kind == "arrive":
                    got[bar] += 1
                elif complete(bar) <= phase:
                    break
                at[role] += 1
                moved = True
                if role == held:
                    break
            return moved

        while True:
            while any([run(r) for r in ops if r != held]):
                pass
            if at[held] < len(ops[held]):
                kind, bar, phase = ops[held][at[held]]
                if kind == "wait" and complete(bar) > phase + 1:
                    bad.add((held, bar, phase, complete(bar)))
            if not run(held):
                break
        for r in ops:
            assert at[r] == len(ops[r]), f"{r} waits for ever at {ops[r][at[r]]}"
    return bad


@pytest.mark.parametrize("L", [1, 2, 3, 8])
@pytest.mark.parametrize("nc", [1, 2, 3, 4])
@pytest.mark.parametrize("tiles,nc0,ring", [(1, 1, 4), (3, 1, 2), (2, 4, 3)])
def test_no_wait_is_overtaken(L, nc, tiles, nc0, ring):
    assert not overtaken(*roles(L, nc, nc0, tiles, ring))
