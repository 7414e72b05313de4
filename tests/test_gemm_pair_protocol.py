"""A model of the barrier schedule of the W8A8 GEMM's pairs of CTAs (csrc/w8a8.cu, cta_group::2), checked over every
interleaving, with and without a wait that runs out.

Both producers wait for their own empty barriers (one commit of rank 0's UMMA thread arrives at both) and load their
half of a k-block; both halves count on rank 0's full barrier of the stage, which rank 0's producer arms for both. The
UMMA thread of rank 0 waits for the full barriers and for the accumulator set (an arrival from either CTA's read-back
warps), and commits the set to both. A role whose wait runs out, or whose CTA has aborted, stops there. At the end the
CTAs exchange how many k-blocks their producers have loaded and whether they have aborted; if either has, rank 0 goes
through the last round of every stage: it arms what it has not armed, takes back what rank 1 has not loaded, and waits
for the rest.

Checked: a stage is loaded again only after the UMMAs that read it, an accumulator set is written only after both CTAs
have read it, every run ends, and no load is in flight when the CTAs leave."""
import pytest

HALF = 1   # bytes of one rank's half of a k-block, in halves


class Violation(AssertionError):
    pass


def explore(tiles, n_kb, st, abort, drain="handshake"):
    """tiles of n_kb k-blocks each, st stages, two accumulator sets. abort: waits may run out at any time.
    drain: what happens before the CTAs leave ("handshake", or "rank 0": only what rank 0 has armed is waited for).
    Returns the number of states."""
    total = tiles * n_kb
    # full[s]: (phase, armed, bytes expected minus landed); counts of completed phases of the other barriers are
    # derived from the work done.  State: producers' k-blocks issued (2), UMMAs issued, commits landed, sets
    # committed and landed, tiles read back by each CTA (2), loads in flight, full barriers, aborted (2), stopped roles
    start = (0, 0, 0, 0, 0, 0, frozenset(), ((0, 0, 0),) * st, (False, False), frozenset())
    seen, stack = set(), [start]
    ends = 0

    def settle(bar):
        phase, armed, left = bar
        return (phase + 1, 0, 0) if armed and left == 0 else bar

    while stack:
        s = stack.pop()
        if s in seen:
            continue
        seen.add(s)
        g0, g1, u, landed, r0, r1, flight, full, aborted, stopped = s
        nxt = []

        def go(**k):
            d = dict(g0=g0, g1=g1, u=u, landed=landed, r0=r0, r1=r1, flight=flight, full=full, aborted=aborted,
                     stopped=stopped)
            d.update(k)
            nxt.append(tuple(d[x] for x in ("g0", "g1", "u", "landed", "r0", "r1", "flight", "full", "aborted",
                                            "stopped")))

        def may_stop(role, cta):
            if abort and role not in stopped:
                a = list(aborted)
                a[cta] = True
                go(stopped=stopped | {role}, aborted=tuple(a))

        for rank, g in ((0, g0), (1, g1)):
            role = "tma%d" % rank
            if role in stopped or g == total:
                continue
            if landed >= g - st + 1:            # the empty barrier's phase: the UMMAs of k-block g - st are done
                i, bar = g % st, list(full[g % st])
                if rank == 0:
                    if bar[1]:
                        raise Violation(f"full barrier {i} armed twice")
                    bar[1], bar[2] = 1, bar[2] + 2 * HALF
                nf = full[:i] + (tuple(bar),) + full[i + 1:]
                go(**{"g%d" % rank: g + 1, "flight": flight | {(rank, g)}, "full": nf})
            else:
                may_stop(role, rank)
        for rank, g in flight:                  # a load lands
            i = g % st
            if landed < g - st + 1:
                raise Violation(f"k-block {g} overwrites a stage whose UMMAs have not completed")
            bar = list(full[i])
            bar[2] -= HALF
            go(flight=flight - {(rank, g)}, full=full[:i] + (settle(tuple(bar)),) + full[i + 1:])
        if "mma" not in stopped and u < total:
            t = u // n_kb
            if u % n_kb == 0 and min(r0, r1) < t - 1:
                may_stop("mma", 0)
            elif full[u % st][0] < u // st + 1:
                may_stop("mma", 0)
            else:
                if any((k, u) in flight for k in (0, 1)) or min(g0, g1) <= u:
                    raise Violation(f"UMMA {u} reads a half that has not landed")
                go(u=u + 1)
        if landed < u:
            go(landed=landed + 1)
        for rank, r in ((0, r0), (1, r1)):
            role = "epi%d" % rank
            if role in stopped or r == tiles:
                continue
            if landed >= (r + 1) * n_kb:        # the set's commit follows its last k-block's
                if u > (r + 2) * n_kb:
                    raise Violation(f"tile {r} is read after its set was written again")
                go(**{"r%d" % rank: r + 1})
            else:
                may_stop(role, rank)
        done = all(("tma%d" % k) in stopped or g == total for k, g in ((0, g0), (1, g1))) and \
            ("mma" in stopped or u == total) and landed == u and \
            all(("epi%d" % k) in stopped or r == tiles for k, r in ((0, r0), (1, r1)))
        if done:
            ends += 1
            _leave(g0, g1, st, flight, full, any(aborted), drain, settle)
        elif not nxt:
            raise Violation(f"deadlock at {s}")
        stack.extend(nxt)
    assert ends > 0
    return len(seen)


def _leave(g0, g1, st, flight, full, aborted, drain, settle):
    """Every order in which the loads in flight can land: the drain's waits all end, and none is left after it."""
    full = [list(b) for b in full]
    g = max(g0, g1) if drain == "handshake" else g0
    waits = []
    if aborted:
        for i in range(max(g - st, 0), g):
            b = full[i % st]
            if drain == "handshake":
                if i >= g0:
                    if b[1]:
                        raise Violation(f"full barrier {i % st} armed twice by the drain")
                    b[1], b[2] = 1, b[2] + HALF
                if i >= g1:
                    b[2] -= HALF
                full[i % st] = list(settle(tuple(b)))
            waits.append(i)
    for rank, k in flight:   # all land sooner or later; what is waited for has to include each of them
        if k not in waits:
            raise Violation(f"rank {rank}'s load of k-block {k} is in flight when the CTAs leave")
        b = full[k % st]
        b[2] -= HALF
        full[k % st] = list(settle(tuple(b)))
    for i in waits:
        if full[i % st][0] < i // st + 1:
            raise Violation(f"the drain's wait for k-block {i} never ends")


@pytest.mark.parametrize("tiles,n_kb,st", [(1, 3, 2), (2, 2, 2), (3, 1, 2), (2, 3, 3)])
def test_a_pair_runs_to_its_end(tiles, n_kb, st):
    assert explore(tiles, n_kb, st, abort=False) > 0


@pytest.mark.parametrize("tiles,n_kb,st", [(1, 3, 2), (2, 2, 2), (3, 1, 2), (1, 4, 3)])
def test_no_load_is_in_flight_when_an_aborted_pair_leaves(tiles, n_kb, st):
    assert explore(tiles, n_kb, st, abort=True) > 0


def test_the_model_sees_a_drain_of_rank_0s_loads_alone():
    with pytest.raises(Violation, match="in flight when the CTAs leave|never ends"):
        explore(1, 3, 2, abort=True, drain="rank 0")
