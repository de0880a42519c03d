"""Randomised model of the prefill kernel's mbarrier protocol (csrc/pad_prefill_tc.cu).

The kernel runs a K producer, a V producer, an S issuer, a P.V issuer and two slots of four
softmax warps that hand 128-key tiles to each other through mbarriers waited on by phase
parity.  In pairs both slots use every tile (S_g = Q_g K^T, O_g += P_g V); shared out (split)
slot 0 takes the even tiles and slot 1 the odd ones, both on Q_0.  K tiles live in 3 stages and
V tiles in 2 (4 and 4 at head_dim 64); each slot has one TMEM S buffer, over which P goes, and
P of a tile is released in two parts, each with its own P.V.  The V producer clears the last tile's
rows past the last visible key where there are any (part), and the softmax of that tile waits for
it.  At the end a slot's rows leave through its own Q stage; shared out, the slots first
exchange (m, l) through the second Q stage, which holds nothing, and half of each other's O
rows through the K stages.

The model runs that schedule with loads and MMAs that complete after random delays, and checks
under many random interleavings that no stage or buffer is overwritten while a load lands in it or
something still reads it, that O is rescaled only when no P.V into it is in flight, that no
P.V reads a tile that is not yet cleared, and that nothing deadlocks.  Each of MISTAKES, a slip
planted in the schedule, fails it.
"""
import random

import pytest

N_WARPS = 4  # per slot


class Bar:
    def __init__(s, count):
        s.count = count
        s.pending = 0
        s.done = 0

    def arrive(s):
        s.pending += 1
        if s.pending == s.count:
            s.pending = 0
            s.done += 1

    def ready(s, parity):
        return (s.done % 2) != parity


MISTAKES = {
    # name: the forms (pairs or split) in which it matters
    "rescale_skips_pvlo": (False, True),        # second part rescaled without the first part's P.V
    "s_skips_pvdone": (False, True),            # S over a P that its P.V still reads
    "kfree_after_slot_0": (False,),             # a K stage released before slot 1's S
    "vfree_after_slot_0": (False,),             # a V stage released before slot 1's P.V
    "parts_share_a_barrier": (False, True),     # one P-written barrier for both parts
    "no_wait_for_clear": (False, True),         # the last tile's P released before its V is cleared
    "merge_skips_the_other_slot": (True,),      # O rows into the K stages before both slots are done
    "output_skips_the_other_slot": (True,),     # the other slot's O rows taken before they are there
    "dealloc_without_tdone": (False, True),
}


def run(n, split, stages, seed, part=False, lazy_prob=0.3, mistake=None):
    assert mistake is None or mistake in MISTAKES
    rnd = random.Random(seed)
    KS, VS = stages
    mine = [(n + 1) // 2, n // 2] if split else [n, n]
    kfull, kfree = ([Bar(1) for _ in range(KS)] for _ in range(2))
    vfull, vfree = ([Bar(1) for _ in range(VS)] for _ in range(2))
    qfull = [Bar(1) for _ in range(2)]
    sfull = [Bar(1) for _ in range(2)]
    plo = [Bar(N_WARPS) for _ in range(2)]
    phi = [Bar(N_WARPS) for _ in range(2)]
    if mistake == "parts_share_a_barrier":
        phi = plo
    pvlo = [Bar(1) for _ in range(2)]
    pvdone = [Bar(1) for _ in range(2)]
    vclear, drain_s, drain_pv = Bar(1), Bar(1), Bar(1)
    tdone = Bar(2 * N_WARPS)

    kst, vst = [-1] * KS, [-1] * VS  # tile in each stage (-1: never loaded, None: a load is landing)
    clear = set()                    # V tiles whose unseen rows are cleared
    qst = [None, None]
    s_buf = [None, None]             # tile whose S (or P) the slot's buffer holds
    written = [[0, 0], [0, 0]]       # warps that wrote each part of P of the slot's current tile
    into_o = [0, 0]                  # P.V MMAs into O_g in flight
    reading, inflight, commits = [], [], []
    issued = {"S": [], "PV": []}     # per issuer (a commit tracks only its own MMAs)
    tmem_users = set((g, w) for g in range(2) for w in range(N_WARPS))
    now = [0]

    def async_op(fn):
        inflight.append([now[0] + rnd.randint(1, 30), fn])

    def commit(who, bar):
        pend = [op for op in issued[who] if not op["done"]]
        if pend:
            commits.append({"wait": pend, "bar": bar})
        else:
            bar.arrive()

    def mma(who, regions, done):
        op = {"done": False, "regions": regions}
        issued[who].append(op)
        reading.append(op)

        def fin():
            op["done"] = True
            reading.remove(op)
            done()
        async_op(fin)

    def busy(region):
        return any(region in op["regions"] for op in reading)

    def idle(kind):
        st = {"K": kst, "V": vst, "Q": qst}[kind]
        for s in range(len(st)):
            assert not busy((kind, s)), f"{kind} stage {s} reused while an MMA reads it"
            assert st[s] is not None or (kind, split, s) == ("Q", True, 1), f"{kind} stage {s} reused while loading"

    def slots(t):
        return [(t & 1, t >> 1)] if split else [(0, t), (1, t)]

    def load(kind, t):
        st, ns, full = (kst, KS, kfull) if kind == "K" else (vst, VS, vfull)
        s = t % ns
        assert not busy((kind, s)), f"{kind} stage {s} reloaded while an MMA reads it"
        st[s] = None

        def landed():
            st[s] = t
            full[s].arrive()
        async_op(landed)

    def prologue():
        for g in range(1 if split else 2):
            def landed(g=g):
                qst[g] = "Q"
                qfull[g].arrive()
            async_op(landed)
        load("K", 0)
        load("V", 0)

    def producer(kind):
        ns, freed = (KS, kfree) if kind == "K" else (VS, vfree)
        s, ph = 1, 0
        for t in range(1, n):
            if s == ns:
                s, ph = 0, ph + 1
            if ph > 0:
                yield (freed[s], (ph - 1) & 1)
            load(kind, t)
            s += 1
        if kind == "V" and part:
            t = n - 1
            yield (vfull[t % VS], (t // VS) & 1)
            assert vst[t % VS] == t, "cleared before the tile has landed"
            for _ in range(rnd.choice([0, 5, 80])):
                yield None
            clear.add(t)
            vclear.arrive()

    def s_issuer():
        s, ph = 0, 0
        for t in range(n):
            yield (kfull[s], ph)
            for g, j in slots(t):
                if j == 0:
                    yield (qfull[0 if split else g], 0)
                elif mistake != "s_skips_pvdone":
                    yield (pvdone[g], (j - 1) & 1)
                assert kst[s] == t, f"S({t}) reads a K stage that does not hold it"
                assert qst[0 if split else g] == "Q", f"S({t}) of slot {g} before its Q"
                assert not into_o[g] and not busy(("P", g)), f"S({t}) over a P that is still read"
                if j:
                    assert written[g] == [N_WARPS, N_WARPS], f"S({t}) over scores still in use"
                s_buf[g] = None

                def done(g=g, t=t):
                    s_buf[g] = t
                    written[g] = [0, 0]
                mma("S", [("K", s), ("Q", 0 if split else g)], done)
                commit("S", sfull[g])
                if split or g == (0 if mistake == "kfree_after_slot_0" else 1):
                    commit("S", kfree[s])
            s += 1
            if s == KS:
                s, ph = 0, ph ^ 1
        commit("S", drain_s)
        yield (drain_s, 0)

    def pv_issuer():
        s, ph = 0, 0
        for t in range(n):
            yield (vfull[s], ph)
            for g, j in slots(t):
                for h in range(2):
                    yield ((phi if h else plo)[g], j & 1)
                    assert s_buf[g] == t and written[g][h] == N_WARPS, f"P.V({t}) of slot {g} before part {h} of its P"
                    assert vst[s] == t, f"P.V({t}) reads a V stage that does not hold it"
                    assert not part or t < n - 1 or t in clear, "P.V reads the last V tile before it is cleared"
                    into_o[g] += 1

                    def done(g=g):
                        into_o[g] -= 1
                    mma("PV", [("V", s), ("P", g)], done)
                    if h == 0:
                        commit("PV", pvlo[g])
                commit("PV", pvdone[g])
                if split or g == (0 if mistake == "vfree_after_slot_0" else 1):
                    commit("PV", vfree[s])
            s += 1
            if s == VS:
                s, ph = 0, ph ^ 1
        commit("PV", drain_pv)
        yield (drain_pv, 0)

    met = [0, 0]                      # arrivals at the two block barriers of the shared-out form

    def meet(k):
        met[k] += 1
        while met[k] < 2 * N_WARPS:
            yield None

    staged = set()

    def softmax(g, w):
        for j in range(mine[g]):
            t = 2 * j + g if split else j
            yield (sfull[g], j & 1)
            assert s_buf[g] == t, f"softmax of slot {g} reads S({t}) before it is done"
            for h in range(2):
                for _ in range(rnd.randint(0, 3)):
                    yield None
                if rnd.random() < lazy_prob and (j > 0 or h == 1):
                    if h == 1:
                        if mistake != "rescale_skips_pvlo":
                            yield (pvlo[g], j & 1)
                    else:             # (S of this tile was issued after it: never a real wait)
                        yield (pvdone[g], (j - 1) & 1)
                    assert not into_o[g], "O rescaled while a P.V into it is in flight"
                if h == 0 and part and t == n - 1 and mistake != "no_wait_for_clear":
                    yield (vclear, 0)
                written[g][h] += 1
                (phi if h else plo)[g].arrive()
        if mine[g]:
            yield (pvdone[g], (mine[g] - 1) & 1)
            assert not into_o[g], "O read before its last P.V"
        if split:
            assert not busy(("Q", 1)) and qst[1] is None    # (m, l): nothing else uses the second Q stage
            if mistake != "merge_skips_the_other_slot":
                yield from meet(0)
            idle("K")                 # the O rows go there
            for _ in range(rnd.randint(0, 3)):
                yield None
            staged.add((g, w))
            if mistake != "output_skips_the_other_slot":
                yield from meet(1)
            assert (1 - g, w) in staged, "the other slot's rows read before they are there"
        assert not busy(("Q", g)), f"slot {g} writes its rows over a Q that an S still reads"
        for _ in range(rnd.randint(0, 3)):
            yield None
        tmem_users.discard((g, w))
        tdone.arrive()

    def dealloc():
        if mistake != "dealloc_without_tdone":
            yield (tdone, 0)
        else:
            yield (drain_pv, 0)
        assert not tmem_users, "TMEM freed while a softmax warp still reads it"

    prologue()
    actors = [producer("K"), producer("V"), s_issuer(), pv_issuer(), dealloc()]
    actors += [softmax(g, w) for g in range(2) for w in range(N_WARPS)]
    waiting, alive = [None] * len(actors), [True] * len(actors)
    for step in range(400000):
        if not any(alive):
            return True
        now[0] += 1
        rnd.shuffle(inflight)
        for op in list(inflight):
            if op[0] <= now[0] and rnd.random() < 0.7:
                inflight.remove(op)
                op[1]()
        for c in list(commits):
            if all(o["done"] for o in c["wait"]):
                commits.remove(c)
                c["bar"].arrive()
        progressed = False
        for i in rnd.sample(range(len(actors)), len(actors)):
            if not alive[i]:
                continue
            if waiting[i] is not None:
                bar, parity = waiting[i]
                if not bar.ready(parity):
                    continue
                waiting[i] = None
            progressed = True
            if rnd.random() < 0.5:
                continue
            try:
                waiting[i] = next(actors[i])
            except StopIteration:
                alive[i] = False
        if any(alive) and not progressed and not inflight and not commits:
            raise AssertionError(f"deadlock: {n} tiles, split {split}, stages {stages}")
    raise AssertionError("no progress")


STAGES = [(3, 2), (4, 4)]  # K and V stages at head_dim 128 and 64


@pytest.mark.parametrize("split", [False, True])
@pytest.mark.parametrize("stages", STAGES)
@pytest.mark.parametrize("n", range(1, 12))
def test_prefill_barrier_protocol(n, stages, split):
    """One tile, odd and even counts, a slot without a tile, rings that wrap; the last tile cleared or not."""
    for seed in range(30):
        for part in (False, True):
            assert run(n, split, stages, seed * 131 + n, part=part)


@pytest.mark.parametrize("mistake", sorted(MISTAKES))
def test_prefill_model_detects_planted_mistakes(mistake):
    for split in MISTAKES[mistake]:
        fails = 0
        for n in range(2, 9):
            for seed in range(30):
                try:
                    run(n, split, STAGES[seed & 1], seed * 11 + n, part=True, lazy_prob=0.6, mistake=mistake)
                except AssertionError:
                    fails += 1
        assert fails > 0, (mistake, split)
