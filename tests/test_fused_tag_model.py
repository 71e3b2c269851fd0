"""Model check, on CPU, of the slot tags in the single-kernel batch: lookups
that read a tag and later the word, claims that own a slot by its tag, and
chains and erases that change the word first and the tag in a second step.

Every step below is one access at the GPU's point of coherence, in the order
the kernel issues it (an access whose operands depend on a returned value
comes after it; a fence orders what lies around it).  All interleavings of the
actors are run.  test_fused_protocol.py and test_fused_claims.py check the same
protocol one level up, with a probe of a bucket and a free slot as single
steps."""
import itertools

import pytest

EMPTY = None
MOVE = 1 << 16
TRANSIT = MOVE - 1


def explore(state, actors):
    """All final states: depth-first over every interleaving.  An actor is a
    list of steps; a step is f(state, regs) -> True (done), False (blocked, try
    later) or "end" (the actor stops).  state and regs are dicts of plain
    values."""
    finals, seen = [], set()

    def freeze(st, pcs, regs):
        return (tuple(sorted(st.items(), key=str)), pcs,
                tuple(tuple(sorted(r.items())) for r in regs))

    def go(st, pcs, regs):
        key = freeze(st, pcs, regs)
        if key in seen:
            return
        seen.add(key)
        moved = False
        for a, steps in enumerate(actors):
            if pcs[a] >= len(steps):
                continue
            s2, r2 = dict(st), [dict(r) for r in regs]
            ok = steps[pcs[a]](s2, r2[a])
            if ok is False:
                continue
            moved = True
            pc = len(steps) if ok == "end" else pcs[a] + 1
            go(s2, pcs[:a] + (pc,) + pcs[a + 1:], r2)
        if not moved:
            finals.append((st, pcs, regs))

    go(state, (0,) * len(actors), [{} for _ in actors])
    return finals


# ---- lookups beside chains ---------------------------------------------------
# One slot in each candidate bucket of K (bucket 0 is its BitHash1 bucket, whose
# version its moves mark) and a stash.

def mark(st, r):
    st["ver"] += 1
    return True


def unmark(st, r):
    st["ver"] += MOVE - 1
    return True


def set_word(b, w):
    def f(st, r):
        st["word", b] = w
        return True
    return f


def xor(b, d):
    def f(st, r):
        st["tag", b] ^= d
        return True
    return f


def move(src, dst, tags, swap_in, early=False):
    """A chain swaps K out of `src` for Y and puts it into `dst`: a claim (tag,
    then word) or a swap with Z (word, then tag), or the stash.  `early`: the
    version says that the move is over before its last access."""
    out = [mark, set_word(src, "Y"), xor(src, tags["K"] ^ tags["Y"])]
    if dst == "stash":
        put = [set_word("stash", "K")]
    elif swap_in:
        put = [set_word(dst, "K"), xor(dst, tags["Z"] ^ tags["K"])]
    else:
        put = [xor(dst, tags["K"]), set_word(dst, "K")]  # the tag was 0
    return out + (put[:-1] + [unmark, put[-1]] if early else put + [unmark])


def lookup(order, tags, extra):
    """version, tags (in `order`), the words whose tag matches (or that the
    approximate match adds, `extra`), stash, version"""
    def v0(st, r):
        r["v0"] = st["ver"]
        return True

    def tag(b):
        def f(st, r):
            r[f"look{b}"] = st["tag", b] == tags["K"] or b in extra
            return True
        return f

    def word(b):
        def f(st, r):
            r["hit"] = r.get("hit", False) or (r[f"look{b}"] and st["word", b] == "K")
            return True
        return f

    def stash(st, r):
        r["hit"] = r.get("hit", False) or st["word", "stash"] == "K"
        return True

    def v1(st, r):
        quiet = (r["v0"] & TRANSIT) == 0 and r["v0"] == st["ver"]
        r["verdict"] = "hit" if r["hit"] else "miss" if quiet else "retry"
        return True
    return [v0] + [tag(b) for b in order] + [word(0), word(1), stash, v1]


TAGS = [{"K": 1, "Y": 2, "Z": 3}, {"K": 1, "Y": 1, "Z": 2}, {"K": 1, "Y": 2, "Z": 1},
        {"K": 5, "Y": 5, "Z": 5}]


def verdicts(start, moves, tags, swap_in, extra=(), early=False):
    state = {"ver": 0, ("word", "stash"): EMPTY}
    for b in (0, 1):
        w = "K" if b == start else ("Z" if swap_in else EMPTY)
        state["word", b] = w
        state["tag", b] = tags[w] if w else 0
    chain = []
    for i, (src, dst) in enumerate(moves):
        if i:  # what the first move left in K's way moves on or is erased first
            if dst != "stash" and not swap_in:
                chain += [set_word(dst, EMPTY), xor(dst, tags["Y"])]
            elif dst != "stash":
                chain += [set_word(dst, "Z"), xor(dst, tags["Y"] ^ tags["Z"])]
        chain += move(src, dst, tags, swap_in, early)
    out = set()
    for order in ((0, 1), (1, 0)):
        for st, pcs, regs in explore(state, [chain, lookup(order, tags, extra)]):
            out.add(regs[1]["verdict"])
    return out


ROUTES = [(0, [(0, 1)]), (1, [(1, 0)]), (0, [(0, 1), (1, 0)]), (1, [(1, 0), (0, 1)]),
          (0, [(0, "stash")]), (1, [(1, 0), (0, "stash")])]


@pytest.mark.parametrize("start,moves", ROUTES)
@pytest.mark.parametrize("swap_in", [False, True])
def test_no_lookup_loses_the_key(start, moves, swap_in):
    for tags in TAGS:
        for extra in ((), (0,), (1,), (0, 1)):
            assert "miss" not in verdicts(start, moves, tags, swap_in, extra), (tags, extra)


@pytest.mark.parametrize("swap_in", [False, True])
def test_a_move_that_ends_before_its_last_access_loses_it(swap_in):
    # without the fence between a swap's tag change (or a claim's word) and the
    # version
    assert "miss" in verdicts(0, [(0, 1)], TAGS[0], swap_in, early=True)


# ---- who owns a slot -----------------------------------------------------------
# One slot that holds X, in a bucket with a lock.

def eraser(word, tags):
    """An erase of `word`: swaps it for EMPTY, then frees the tag.  It comes here
    whatever the tag (the approximate match may bring it by another one)."""
    def cas(st, r):
        if st["word"] != word:
            return "end"
        st["word"] = EMPTY
        st["erased", word] = True
        return True

    def free(st, r):
        st["tag"] ^= tags[word]
        return True
    return [cas, free]


def claimer(word, tags):
    def see(st, r):
        return True if st["tag"] == 0 else "end"

    def cas(st, r):
        if st["tag"] != 0:
            return "end"
        st["tag"] = tags[word]
        st["claimed", word] = True
        return True

    def store(st, r):
        if st["word"] is not EMPTY:
            st["overwrote"] = st["word"]
        st["word"] = word
        return True
    return [see, cas, store]


def swapper(word, tags, unlock_early=False, exchange=False):
    """A chain with `word` in hand swaps it in under the bucket lock."""
    def lock(st, r):
        if st["lock"]:
            return False
        st["lock"] = True
        return True

    def read(st, r):
        r["w"] = st["word"]
        if r["w"] is EMPTY:
            st["lock"] = False
            return "end"
        return True

    def cas(st, r):
        if st["word"] != r["w"] and not exchange:
            st["lock"] = False
            return "end"
        r["w"] = st["word"]
        st["word"] = word
        st["hand", word] = r["w"]
        return True

    def retag(st, r):
        st["tag"] ^= tags.get(r["w"], 0) ^ tags[word]
        return True

    def unlock(st, r):
        st["lock"] = False
        return True
    tail = [unlock, retag] if unlock_early else [retag, unlock]
    return [lock, read, cas] + tail


def faults(tags, actors):
    """What is wrong in any final state."""
    state = {"word": "X", "tag": tags["X"], "lock": False, "overwrote": EMPTY}
    bad = set()
    for st, pcs, regs in explore(state, actors):
        assert not st["lock"]
        have = [st["word"]] + [v for k, v in st.items() if isinstance(k, tuple) and k[0] == "hand"]
        gone = [k[1] for k in st if isinstance(k, tuple) and k[0] == "erased"]
        placed = ["X"] + [k[1] for k in st if isinstance(k, tuple) and k[0] in ("claimed", "hand")]
        if st["overwrote"] is not EMPTY:
            bad.add("overwrote")
        for w in placed:
            if have.count(w) + gone.count(w) != 1:
                bad.add("lost or doubled " + w)
        if any(v is EMPTY for k, v in st.items() if isinstance(k, tuple) and k[0] == "hand"):
            bad.add("EMPTY in hand")
        if st["tag"] != (0 if st["word"] is EMPTY else tags[st["word"]]):
            bad.add("tag")
    return bad


# all tags different; three that cancel (1 ^ 2 ^ 3 = 0); pairs and all alike
OWN_TAGS = [dict(zip("XYZN", t)) for t in
            itertools.chain([(1, 2, 4, 8), (1, 2, 3, 4), (2, 3, 1, 1)],
                        itertools.product((1, 2), repeat=4))]


@pytest.mark.parametrize("tags", OWN_TAGS, ids=str)
def test_slots_keep_one_owner(tags):
    for actors in (
            [eraser("X", tags), claimer("N", tags), swapper("Y", tags)],
            [eraser("Y", tags), claimer("N", tags), swapper("Y", tags)],
            [eraser("X", tags), eraser("Y", tags), claimer("N", tags),
             swapper("Y", tags)],
            [claimer("N", tags), swapper("Y", tags), swapper("Z", tags)],
            [eraser("Y", tags), claimer("N", tags), swapper("Y", tags), swapper("Z", tags)],
            [eraser("X", tags), eraser("Z", tags), claimer("N", tags),
             swapper("Y", tags), swapper("Z", tags)]):
        assert not faults(tags, actors), actors


def test_an_unlock_before_the_tag_change_loses_words():
    # two pending tag changes may sum to 0 while the slot holds a word, and a
    # claim then stores over it
    tags = {"X": 1, "Y": 2, "Z": 3, "N": 4}
    bad = faults(tags, [claimer("N", tags), swapper("Y", tags, unlock_early=True),
                        swapper("Z", tags, unlock_early=True)])
    assert "overwrote" in bad


def test_an_exchange_beside_erases_loses_words():
    tags = {"X": 1, "Y": 2, "Z": 4, "N": 8}
    assert faults(tags, [eraser("X", tags), claimer("N", tags),
                         swapper("Y", tags, exchange=True)])
