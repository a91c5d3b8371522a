"""The rings of key and value stages of the chunk attention's warp-specialised kernel, as a model of its roles whose every interleaving is
searched: two issuing warps (one per query tile, of which one may have fewer key tiles or none), two copying warps, the staging threads, and
the tensor pipe, which finishes late.  Barriers count phases and are tested by parity, as in the kernel (prefill_attn_ws_kernel in
csrc/prefill.cu); a state that nothing can leave before all tiles are through is a wait that runs out."""
import pytest

KS, VS = 2, 3                                           # depths of the key and the value ring


def _stuck(nt, staged, mine, looks_at_all):
    """Number of stuck states with nt key tiles, the first `staged` of them written by the staging threads, and mine[t] tiles of query
    tile t.  looks_at_all: an issuing warp tests the arrival of every key tile, also of those that it does not read."""
    def landed(count, g, depth):                        # mbarrier.test_wait.parity on a barrier with `count` complete phases
        return (count & 1) != ((g // depth) & 1)

    def phases(tiles, stage, depth):                    # complete phases of a stage's "landed" barrier after the first `tiles` tiles
        return (tiles - stage + depth - 1) // depth

    def left(t, g, issued, done):                       # query tile t no longer needs the stage of key tile g
        return done[t] > g if g < mine[t] else issued[t] > g

    def steps(s):
        # per query tile: score tiles issued / done, products issued / done; key and value tiles that have landed
        sc, sd, pv, pd, k, v = s
        out = []
        put = lambda x, t, n: x[:t] + (n,) + x[t + 1:]  # noqa: E731
        for t in range(2):
            g = pv[t]
            if g < sc[t] and landed(phases(v, g % VS, VS), g, VS):
                assert v > g                            # the parity was not mistaken for another phase's
                if g >= mine[t] or sd[t] > g:           # a tile of the other query tile is only released; probabilities follow the scores
                    out.append((sc, sd, put(pv, t, g + 1), pd, k, v))
            g = sc[t]
            if g < nt and g < pv[t] + 2:
                if (g >= mine[t] and g + KS >= staged and not looks_at_all) or landed(phases(k, g % KS, KS), g, KS):
                    assert k > g or g >= mine[t]
                    out.append((put(sc, t, g + 1), sd, pv, pd, k, v))
            if sd[t] < min(sc[t], mine[t]):             # the tensor pipe finishes scores, in order
                out.append((sc, put(sd, t, sd[t] + 1), pv, pd, k, v))
            if pd[t] < min(pv[t], mine[t]):
                out.append((sc, sd, pv, put(pd, t, pd[t] + 1), k, v))
        free_v = v < VS or all(left(t, v - VS, pv, pd) for t in range(2))
        if k == v and k < staged and free_v and (k < KS or all(left(t, k - KS, sc, sd) for t in range(2))):
            out.append((sc, sd, pv, pd, k + 1, v + 1))
        if k >= staged and v >= staged:                 # the chunk's own tiles: keys and values advance on their own
            if k < nt and (k < KS or all(k - KS >= mine[t] or sd[t] > k - KS for t in range(2))):
                out.append((sc, sd, pv, pd, k + 1, v))
            if v < nt and free_v:
                out.append((sc, sd, pv, pd, k, v + 1))
        return out

    first = ((0, 0), (0, 0), (0, 0), (0, 0), 0, 0)
    seen, todo, stuck = {first}, [first], 0
    while todo:
        s = todo.pop()
        nxt = steps(s)
        if not nxt and min(s[2]) < nt:
            stuck += 1
        for n in nxt:
            if n not in seen:
                seen.add(n)
                todo.append(n)
    return stuck


CASES = [(nt, staged, other) for nt in range(1, 8) for staged in sorted({0, 1, 2, 3, nt // 2, nt - 1, nt}) if staged <= nt
         for other in sorted({0, 1, nt - 2, nt - 1, nt}) if 0 <= other <= nt]


@pytest.mark.parametrize("swapped", [False, True])
def test_no_wait_runs_out(swapped):
    for nt, staged, other in CASES:
        assert _stuck(nt, staged, (other, nt) if swapped else (nt, other), looks_at_all=False) == 0, (nt, staged, other)


def test_testing_every_key_tile_would_stick():
    """Why an issuing warp does not look for copied key tiles that it does not read: from three tiles on the copies can refill a stage before it has
    looked, and its parity then reads "not landed" for good."""
    assert [nt for nt in range(1, 8) if _stuck(nt, 0, (nt, 0), looks_at_all=True)] == [3, 4, 5, 6, 7]
