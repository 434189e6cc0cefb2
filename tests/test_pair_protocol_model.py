"""A CPU model of decode_pair's synchronisation (csrc/decode_pair.cu): per CTA of the
pair four softmax warps and thirteen dequantising warps, the leader's MMA issuer and the
other CTA's query loader, written as the barrier, buffer and MMA operations each of them
performs per tile, in program order. A scheduler runs them under random interleavings;
MMAs and commits complete in order at random later points, and arrivals and marks that
cross to the other CTA are delivered later still, commits' in order, the threads' in any
order.

Checked at every step, as in the model of decode_main: parity waits neither pass on an
older phase nor miss theirs; nothing is written while an MMA or copy in flight touches
it; an MMA reads only operands that are completely written for its tile, scores and
outputs are read only when they hold the tile expected; the epilogue's staging in the P
tiles meets no weights; every warp sees a raise that any warp of its CTA marked, and the
issuer sees it before PV reads P. Mutations must be caught: each wait taken out, QK not
held behind the PV of two tiles before ("window"), the renewal at a segment's start
without its exchange, which also keeps the next weights out of the epilogue's staging
("renew_sync"), a mark that is not released or not acquired by the arrival it goes with,
and the issuer waiting for a rewritten P in place of passing on to the next QK
("issuer_passes").
"""
import random

import pytest

from test_protocol_model import Bar, Hazard

SOFT, DQ = 4, 13


def tiles(refs, segments, renews, my_ref):
    """The pair's tile list. refs: block counts (1 or 2) of its reference tiles; segments:
    block counts; renews[r][s]: even blocks of segment s at which CTA r renews (the first
    block of every segment but the first always); my_ref[r]: CTA r's reference tile, or -1."""
    out = []
    for i, cnt in enumerate(refs):
        out += [dict(ref=True, tile=i, end=k + 1 == cnt) for k in range(cnt)]
    for s, cnt in enumerate(segments):
        for q in range(cnt):
            out.append(dict(ref=False, seg=s, first=q == 0, last=q + 1 == cnt, even=q % 2 == 0, more=q + 1 < cnt,
                            renew=[q in renews[r][s] if q or not s else True for r in range(2)]))
    for r in range(2):  # without a reference tile the range's first block renews
        if my_ref[r] < 0:
            out[sum(refs)]["renew"][r] = True
    return out


class Pair:
    def __init__(self, tl, my_ref, over, seed, drop=()):
        self.rng = random.Random(seed)
        self.async_weight = self.rng.choice([1.0, 0.3, 0.05])
        self.net_weight = self.rng.choice([1.0, 0.1])
        self.slow = self.rng.choice([None, None, ("s", 0), ("s", 1), ("d", 0), ("d", 1), "i"])  # a slow role
        self.t, self.my_ref, self.over, self.drop = tl, my_ref, over, drop
        self.refs = sum(x["ref"] for x in tl)
        self.bars = {}
        for i in range(2):
            for n, c in (("k_full", 18), ("v_full", 16), ("p_full", 8)):
                self.bars[n, i] = Bar(c)
            self.bars["p_fixed", i] = Bar(4)
            for r in range(2):
                self.bars["k_free", r, i] = Bar(1)
                self.bars["pv_done", r, i] = Bar(1)
        for i in range(4):
            self.bars["s_free", i] = Bar(8)
            for r in range(2):
                self.bars["s_full", r, i] = Bar(1)
        self.bars["o_free",], self.bars["q_peer",] = Bar(8), Bar(1)
        for r in range(2):
            self.bars["q_free", r], self.bars["q_bar", r], self.bars["grp", r] = Bar(1), Bar(1), Bar(4)
        self.parts, self.state = {}, {}
        self.fifo, self.copies, self.net, self.commits = [], [], [], []
        self.marks = {}    # ("over", r, st) of the CTA; ("raised", r, st) as the leader sees it
        self.staging = {}  # (r, P tile, row half) -> warp
        self.actors = {("s", r, w): self.softmax(r, w) for r in range(2) for w in range(SOFT)}
        self.actors.update({("d", r, d): self.dequant(r, d) for r in range(2) for d in range(DQ)})
        self.actors["q"] = self.query()
        self.cur = {a: None for a in self.actors}
        # the issuer's registers
        self.sq = self.sp = self.n = self.v = self.qseg = self.pseg = 0
        self.fixes, self.q_state, self.blocked = [0, 0], 0, False
        while self.sp < len(tl) and tl[self.sp]["ref"]:
            self.sp += 1

    # ---------------------------------------------------------------- programs
    def dequant(self, r, d):
        own, k = d < 9, d if d < 9 else 4 * r + d - 9
        to_v = not own or (k < 8 and k >> 2 == r)
        v = 0
        for n, t in enumerate(self.t):
            if own:
                if n >= 2 and "k_free" not in self.drop:
                    yield ("wait", ("k_free", r, n & 1), (n >> 1) - 1)
                yield ("write", ("K", r, n & 1), n, d)
                yield ("arrive", r, ("k_full", n & 1))
            if not t["ref"]:
                if to_v:
                    if v >= 2 and "v_slot" not in self.drop:
                        yield ("wait", ("pv_done", r, v & 1), (v >> 1) - 1)
                    yield ("write", ("V", r, v & 1), v, d)
                    yield ("arrive", r, ("v_full", v & 1))
                v += 1

    def softmax(self, r, w):
        st = dict(gph=0)
        n = v = seg_v = 0
        due = False

        def exchange(drop=False):
            if drop:
                return
            yield ("arrive", r, ("grp", r))
            yield ("wait", ("grp", r), st["gph"])
            st["gph"] += 1

        def move_ref(i):
            if i == seg_v:
                return
            if "move_pv" not in self.drop:
                yield ("wait", ("pv_done", r, (i - 1) & 1), (i - 1) >> 1)
            yield ("tmem_rw", ("O", r), i - 1)

        def wait_s(i):
            if "s_full" not in self.drop:
                yield ("wait", ("s_full", r, i & 3), i >> 2)
            yield ("read", ("S", r, i & 3), i)

        def settle(odd, nxt):
            if "settle_grp" not in self.drop:
                yield ("wait", ("grp", r), st["gph"])
            st["gph"] += 1
            yield ("vote", r, (v - 1) & 1, v)
            if self.over[r].get(v - 1):
                yield ("read", ("S", r, (n - 1) & 3), n - 1)
                if odd or nxt:
                    i = n - 2 if odd else n
                    yield ("read", ("S", r, i & 3), i)
                yield from exchange()
                yield from move_ref(v - 1)
                yield ("read", ("S", r, (n - 1) & 3), n - 1)
                yield ("weights", r, (v - 1) & 1, (v - 1, "fixed"), w)
                yield ("arrive", r, ("p_fixed", r))
            if odd:
                yield ("arrive", r, ("s_free", (n - 2) & 3))
            if not nxt:
                yield ("arrive", r, ("s_free", (n - 1) & 3))

        for t in self.t:
            if t["ref"]:
                yield from wait_s(n)
                yield ("arrive", r, ("s_free", n & 3))
                if t["end"] and t["tile"] == self.my_ref[r]:
                    yield from exchange()
                n += 1
                continue
            if t["first"]:
                seg_v = v
            yield from wait_s(n)
            if due:
                yield from settle(t["even"], not t["even"])
            if t["renew"][r]:
                if t["more"]:
                    yield from wait_s(n + 1)
                yield from exchange("renew_sync" in self.drop)
                yield from move_ref(v)
            yield ("weights", r, v & 1, (v, "new"), w)
            mark = w in self.over[r].get(v, ())
            if mark:
                yield ("mark", r, v & 1, v + 1)
            yield ("arrive", r, ("p_full", v & 1), ("raised", r, v & 1, v + 1) if mark else None)
            yield ("arrive", r, ("grp", r))
            due = True
            n, v = n + 1, v + 1
            if not t["last"]:
                continue
            yield from settle(not t["even"], False)
            due = False
            yield from exchange()
            if "epi_pv" not in self.drop:
                yield ("wait", ("pv_done", r, (v - 1) & 1), (v - 1) >> 1)
            yield ("stage", r, w)
            yield ("read", ("O", r), v - 1)
            yield ("unstage", r, w)
            yield ("arrive", r, ("o_free",))

    def query(self):
        segs = 1 + max(t["seg"] for t in self.t if not t["ref"])
        for s in range(segs):
            if s and "q_free" not in self.drop:
                yield ("wait", ("q_free", 1), s - 1)
            yield ("copy", ("Q", 1), s, ("q_bar", 1))
            yield ("wait", ("q_bar", 1), s)
            yield ("arrive", 1, ("q_peer",))
        yield ("wait", ("q_free", 1), segs - 1)  # the last commit's arrival at this CTA

    # The issuer: one pass of its loop, PV first. dry: only whether it would do something.
    def issue(self, dry):
        T = self.t
        test = lambda bar, i: self.test(bar, i)  # noqa: E731
        if self.sp < len(T):
            t, st, ph = T[self.sp], self.v & 1, self.v >> 1
            ready = (("p_full" in self.drop or test(("p_full", st), ph)) and
                     ("v_full" in self.drop or test(("v_full", st), ph)) and
                     (not t["first"] or self.pseg == 0 or "o_free" in self.drop or test(("o_free",), self.pseg - 1)))
            fix = [False, False]
            if ready:
                for r in range(2):
                    fix[r] = self.marks.get(("raised", r, st)) == self.v + 1
                    if fix[r] and "p_fixed" not in self.drop:
                        ready = ready and test(("p_fixed", r), self.fixes[r])
                if not ready and "issuer_passes" in self.drop:
                    return False  # (the mistake once made: waits for the rewrite here)
            if ready:
                if dry:
                    return True
                for r in range(2):
                    self.fixes[r] += fix[r]
                reads = [(("V", r, st), self.v, 8) for r in range(2)]
                reads += [(("P", r, st), (self.v, "fixed" if self.over[r].get(self.v) else "new"), 4) for r in range(2)]
                self.mma(reads, [("O", 0), ("O", 1)], self.v)
                self.fifo.append(("commit", ("pv_done", st)))
                self.pseg += t["last"]
                self.v, self.sp = self.v + 1, self.sp + 1
                return True
        if self.sq < len(T):
            t, st = T[self.sq], self.n & 1
            if self.q_state == 0 and (self.qseg == 0 or "q_free" in self.drop or test(("q_free", 0), self.qseg - 1)):
                if dry:
                    return True
                self.copy(("Q", 0), self.qseg, ("q_bar", 0))
                self.q_state = 1
                return True
            if self.q_state == 1 and test(("q_bar", 0), self.qseg) and \
                    ("q_peer" in self.drop or test(("q_peer",), self.qseg)):
                if dry:
                    return True
                self.q_state = 2
                return True
            if (self.q_state == 2 and ("window" in self.drop or self.n < self.v + 2 + self.refs) and
                    ("k_full" in self.drop or test(("k_full", st), self.n >> 1)) and
                    (self.n < 4 or "s_free" in self.drop or test(("s_free", self.n & 3), (self.n >> 2) - 1))):
                if dry:
                    return True
                reads = [(("K", r, st), self.n, 9) for r in range(2)] + [(("Q", r), self.qseg, None) for r in range(2)]
                self.mma(reads, [("S", r, self.n & 3) for r in range(2)], self.n)
                self.fifo += [("commit", ("s_full", self.n & 3)), ("commit", ("k_free", st))]
                if not t["ref"] and t["last"]:
                    self.fifo.append(("commit", ("q_free",)))
                    self.q_state = 0
                    self.qseg += 1
                self.n, self.sq = self.n + 1, self.sq + 1
                return True
        return False

    # ---------------------------------------------------------------- semantics
    def test(self, bar, i):
        done = self.bars[bar].done
        if done < i or done > i + 1:
            raise Hazard(f"{bar}: probe of phase {i} with {done} done")
        return done == i + 1

    def touched(self, buf, writes_only=False):
        for op in self.fifo:
            if op[0] == "mma" and (buf in op[2] or (not writes_only and any(x[0] == buf for x in op[1]))):
                return True
        return any(c[0] == buf for c in self.copies)

    def arrive(self, name):
        b = self.bars[name]
        b.arrived += 1
        if b.arrived == b.count:
            b.arrived = 0
            b.done += 1
            for i in b.waiting:
                if b.done > i + 1:
                    raise Hazard(f"{name}: a waiter for phase {i} missed it")

    def write(self, buf, ver, part):
        if self.touched(buf):
            raise Hazard(f"{buf} {ver} written while an MMA or copy touches it")
        held = self.parts.setdefault(buf, [None, set()])
        if held[0] != ver:
            self.parts[buf] = held = [ver, set()]
        held[1].add(part)

    def mma(self, reads, writes, ver):
        for buf, want, nparts in reads:
            if nparts is None:
                ok = self.state.get(buf) == want
            else:
                held = self.parts.get(buf, (None, ()))
                ok = held[0] == want and len(held[1]) == nparts
            if not ok:
                raise Hazard(f"MMA {ver} reads {buf} before it holds {want}")
        self.fifo.append(("mma", reads, writes, ver))

    def copy(self, buf, ver, bar):
        if self.touched(buf):
            raise Hazard(f"copy into {buf} while an MMA reads it")
        self.copies.append((buf, ver, bar))

    def start(self, actor, op):
        if op[0] == "wait":
            b = self.bars[op[1]]
            if b.done < op[2] or b.done > op[2] + 1:
                raise Hazard(f"{actor} waits for {op[1]} phase {op[2]} with {b.done} done")
            b.waiting.append(op[2])

    def execute(self, actor, op):
        kind = op[0]
        if kind == "wait":
            self.bars[op[1]].waiting.remove(op[2])
        elif kind == "arrive":
            r, name, mark = op[1], op[2], op[3] if len(op) > 3 else None
            leaders = name[0] != "grp"
            if mark is not None:
                visible = "mark_release" not in self.drop and "mark_acquire" not in self.drop
                if visible and r == 0:
                    self.marks[mark[:3]] = mark[3]
                elif not visible:
                    self.net.append(("mark", mark))
                    mark = None
            if leaders and r == 1:
                self.net.append(("arrive", name, mark))
            else:
                self.arrive(name)
        elif kind == "write":
            self.write(*op[1:])
        elif kind == "weights":
            _, r, st, ver, w = op
            if (r, st, w & 1) in self.staging:
                raise Hazard(f"weights {ver} of CTA {r} into the staging of warp {self.staging[r, st, w & 1]}")
            self.write(("P", r, st), ver, w)
        elif kind == "stage":
            _, r, w = op
            if self.touched(("P", r, w >> 1)):
                raise Hazard("staging over weights that PV reads")
            self.parts.pop(("P", r, w >> 1), None)
            self.staging[r, w >> 1, w & 1] = w
        elif kind == "unstage":
            del self.staging[op[1], op[2] >> 1, op[2] & 1]
        elif kind == "mark":
            self.marks["over", op[1], op[2]] = op[3]
        elif kind == "vote":
            _, r, st, v = op
            if bool(self.over[r].get(v - 1)) != (self.marks.get(("over", r, st)) == v):
                raise Hazard(f"a warp of CTA {r} misses the raise of tile {v - 1}")
        elif kind in ("read", "tmem_rw"):
            _, buf, ver = op
            if self.touched(buf, writes_only=kind == "read"):
                raise Hazard(f"{actor} accesses {buf} while an MMA writes it")
            if self.state.get(buf) != ver:
                raise Hazard(f"{actor} expects {buf} of tile {ver}, holds {self.state.get(buf)}")
        elif kind == "copy":
            self.copy(*op[1:])

    def async_step(self, what):
        if what == "copy":
            buf, ver, bar = self.copies.pop(0)
            self.state[buf] = ver
            self.arrive(bar)
        elif what == "net":
            op = self.net.pop(self.rng.randrange(len(self.net)))
            if op[0] == "mark":
                self.marks[op[1][:3]] = op[1][3]
            else:
                if op[2] is not None:
                    self.marks[op[2][:3]] = op[2][3]
                self.arrive(op[1])
        elif what == "commit":
            self.arrive(self.commits.pop(0))
        else:
            op = self.fifo.pop(0)
            if op[0] == "mma":
                for buf in op[2]:
                    self.state[buf] = op[3]
            else:
                name, tail = op[1][0], op[1][1:]
                self.arrive((name, 0) + tail)
                self.commits.append((name, 1) + tail)  # reaches the other CTA later

    def run(self, max_steps=200000):
        for _ in range(max_steps):
            for a, g in self.actors.items():
                if self.cur[a] is None and g is not None:
                    try:
                        self.cur[a] = next(g)
                        self.start(a, self.cur[a])
                    except StopIteration:
                        self.actors[a] = None
            threads = [a for a, op in self.cur.items()
                       if op is not None and (op[0] != "wait" or self.bars[op[1]].done >= op[2] + 1)]
            if self.issue(True):
                threads.append("i")
            quick = [a for a in threads if a != self.slow and (self.slow is None or a[:2] != self.slow)]
            if quick and self.rng.random() < 0.98:
                threads = quick
            engines = [(w, wt) for w, q, wt in (("mma", self.fifo, self.async_weight), ("copy", self.copies, 1.0),
                                                ("net", self.net, self.net_weight),
                                                ("commit", self.commits, self.net_weight)) if q]
            if not threads and not engines:
                if any(op is not None for op in self.cur.values()) or self.sp < len(self.t):
                    raise Hazard(f"deadlock: {[(a, op) for a, op in self.cur.items() if op is not None]}")
                return
            if not any(op is not None for op in self.cur.values()) and not self.fifo and self.commits \
                    and self.sp == len(self.t):
                raise Hazard(f"a CTA leaves before the arrivals {self.commits}")
            if engines and (not threads or self.rng.random() < 0.3):
                what = self.rng.choices([e[0] for e in engines], [e[1] for e in engines])[0]
                if not threads or self.rng.random() < dict(engines)[what]:
                    self.async_step(what)
                    continue
            if threads:
                who = self.rng.choice(threads)
                if who == "i":
                    self.issue(False)
                else:
                    op, self.cur[who] = self.cur[who], None
                    self.execute(who, op)
        raise Hazard("step limit")


def _random_case(seed):
    rng = random.Random(1000 + seed)
    refs = rng.choice([[], [], [2], [1], [2, 2], [2, 1]])
    my_ref = [rng.choice([-1] + list(range(len(refs)))) for _ in range(2)]
    if refs:  # every reference tile is somebody's
        my_ref = rng.choice([[0, -1], [-1, 0], [0, 0]] if len(refs) == 1 else [[0, 1], [1, 0]])
    segments = [rng.choice([1, 2, 3, 4, 7, 8]) for _ in range(rng.randint(1, 3))]
    renews = [[{q for q in range(0, c, 2) if q and rng.random() < 0.3} for c in segments] for _ in range(2)]
    tl = tiles(refs, segments, renews, my_ref)
    p = rng.choice([0.0, 0.2, 0.6, 1.0])
    over = [{}, {}]
    for r in range(2):
        for v in range(sum(segments)):
            if rng.random() < p:
                over[r][v] = set(rng.sample(range(SOFT), rng.randint(1, SOFT)))
    return tl, my_ref, over


def _run(seed, drop=()):
    Pair(*_random_case(seed), seed, drop).run()


@pytest.mark.parametrize("block", range(6))
def test_pair_protocol_has_no_hazard(block):
    for seed in range(25 * block, 25 * block + 25):
        _run(seed)


@pytest.mark.parametrize("drop", ["k_full", "v_full", "p_full", "s_free", "k_free", "v_slot", "s_full", "settle_grp",
                                  "move_pv", "epi_pv", "p_fixed", "q_free", "q_peer", "renew_sync", "window",
                                  "issuer_passes", "mark_release", "mark_acquire"])
def test_model_catches(drop):
    for seed in range(150):
        try:
            _run(seed, (drop,))
        except Hazard:
            return
    raise AssertionError(drop)


def test_o_free_is_implied():
    # the next segment's weights, which its first PV waits for, are written after the
    # epilogue has read O; the wait stays as a guard
    for seed in range(60):
        _run(seed, ("o_free",))
