"""The chunked refresh kernel's roles meet at mbarriers, whose parity cannot tell phase n + 1 from phase n - 1: a wait for phase n has
to come, in every possible timing, before phase n + 1 completes.  Here the roles of refresh_chunked.cu are written down as their
sequences of waits and arrivals (one unit of several chunks), and every wait is checked against the order those impose.  The number of
wait sites per barrier is compared with the source, so that a new wait there has to be entered here."""
import os
import re
from collections import defaultdict

import pytest

import paper_2608_30386_b200

SOURCE = os.path.join(os.path.dirname(paper_2608_30386_b200.__file__), "csrc", "refresh_chunked.cu")
CHUNKS = 7


class Order:
    """Operations of roles, in program order each; barrier phases complete behind all their arrivals and the phase before."""

    def __init__(self, split):
        self.split = split                      # barrier -> how many there are, taken by chunk index in turn
        self.before = defaultdict(set)          # operation or event -> what comes directly before it
        self.last, self.arrivals, self.waits, self.n = {}, defaultdict(list), [], 0
        self.unwaited, self.waited = set(), set()

    def op(self, role):
        self.n += 1
        if role in self.last:
            self.before[self.n].add(self.last[role])
        self.last[role] = self.n
        return self.n

    def phase(self, bar, chunk):
        m = self.split.get(bar, 1)
        return bar, chunk % m, chunk // m

    def arrive(self, role, bar, chunk):
        self.arrivals[self.phase(bar, chunk)].append(self.op(role))

    def later(self, role, bar, chunk):  # an arrival by the tensor core or a copy, some time after the role has asked for it
        self.arrive(role, bar, chunk)
        self.unwaited.add(self.phase(bar, chunk))

    def wait(self, role, bar, chunk):
        w = self.op(role)
        self.before[w].add(self.phase(bar, chunk))
        self.waits.append((w, role, bar, self.phase(bar, chunk)))
        self.waited.add(self.phase(bar, chunk))

    def meet(self, role, name, chunk):  # a named barrier of the block
        event = ("named", name, chunk)
        self.before[event].add(self.op(role))
        self.before[self.op(role)].add(event)

    def overtaken(self):
        for (bar, i, k), ops in self.arrivals.items():
            self.before[bar, i, k].update(ops)
            if k:
                self.before[bar, i, k].add((bar, i, k - 1))
        behind = {}

        def reach(x):  # everything that comes before x
            stack = [x]
            while stack:
                y = stack[-1]
                todo = [z for z in self.before[y] if z not in behind]
                if y in behind or not todo:
                    behind[y] = set(self.before[y]).union(*(behind[z] for z in self.before[y])) if self.before[y] else set()
                    stack.pop()
                else:
                    assert len(stack) < 10 * self.n, "a circular wait"
                    stack.extend(todo)
            return behind[x]

        return {f"{bar} by {role}" for w, role, bar, (b, i, k) in self.waits
                if (b, i, k + 1) in self.arrivals and w not in reach((b, i, k + 1))}


def roles(alone, kda, with_o):
    two = {b: 2 for b in ("rdy_prep", "bar_ap", "bar_ro", "g_full", "kq_full")} if alone else {}
    x = Order({**two, "bar_s": 2, "rdy_fac": 4 if alone else 2})
    chain, producers, out = [f"chain {i}" for i in range(8)], [f"producer {i}" for i in range(8 if alone else 4)], [f"out {i}" for i in range(4)]

    def mma1(role, n):
        x.wait(role, "rdy_prep", n)
        x.later(role, "bar_ap", n)

    def take_a(role, n):
        x.wait(role, "bar_ap", n)
        if alone and n:
            x.wait(role, "rdy_rhs", n - 1)
        x.meet(role, "A", n)

    def take_p(role, n):
        x.wait(role, "bar_ap", n)
        if not alone and n:
            x.wait(role, "tp_free", n - 1)

    for n in range(CHUNKS):  # the issuing warp
        if alone:
            x.wait("issue", "bar_ap", n)
            x.wait("issue", "rdy_half", n)
        else:
            mma1("issue", n)
            take_a("issue", n)
        x.wait("issue", "rdy_state", n)
        x.later("issue", "bar_ro", n)
        if not alone:
            x.wait("issue", "rdy_t", n)
        x.wait("issue", "rdy_rhs", n)
        x.later("issue", "bar_u", n)
        x.wait("issue", "bar_u", n)
        x.wait("issue", "rdy_u", n)
        for bar in ("bar_s", "bar_o")[:2 if with_o else 1] if alone else ("bar_o", "bar_s"):
            x.later("issue", bar, n)

    x.later("triangular", "v_full", 0)
    if kda and not alone:
        x.arrive("triangular", "rdy_prep", 0)
    for n in range(CHUNKS):
        x.wait("triangular", "bar_ap", n)
        x.meet("triangular", "A", n)
        x.arrive("triangular", "a_taken", n)
        if not alone and n:
            x.wait("triangular", "tp_free", n - 1)
        x.arrive("triangular", "rdy_rhs" if alone else "rdy_t", n)
        if n + 1 < CHUNKS:
            if kda and not alone:
                x.arrive("triangular", "rdy_prep", n + 1)
            x.wait("triangular", "rdy_rhs", n)
            x.later("triangular", "v_full", n + 1)

    if alone:
        def copy(n):
            for bar in ("g_full", "kq_full") if kda else ("kq_full",):
                x.later("mma1", bar, n)
        copy(0)
        copy(1)
        for n in range(CHUNKS):
            if n:
                x.wait("mma1", "bar_ro", n - 1)
            mma1("mma1", n)
            take_a("mma1", n)
            if n + 2 < CHUNKS:
                copy(n + 2)

    def next_p(role, n):
        if role in out[2:]:
            take_p(role, n)
        x.arrive(role, "rdy_rhs", n)

    for role in out if alone and with_o else ():
        next_p(role, 0)
        for n in range(CHUNKS):
            x.wait(role, "bar_o", n)
            if n + 1 < CHUNKS:
                next_p(role, n + 1)
            x.meet(role, "O tile free", n)
            x.meet(role, "O tile", n)

    for i, role in enumerate(producers):
        def kq(n):
            if with_o or i & 3 < 2:
                x.later(role, "kq_full", n)
        if not alone:
            if kda:
                x.later(role, "g_full", 0)
            kq(0)
        if not kda and i == 0:
            x.arrive(role, "rdy_fac", 0)
        for n in range(CHUNKS):
            if alone or not kda:
                x.meet(role, "producers", n)
            x.wait(role, "kq_full", n)
            if kda:
                x.wait(role, "g_full", n)
            if alone and n > 1:
                x.wait(role, "bar_ro", n - 2)
            for half in (i >> 2,) if alone else (0, 1):
                if kda:
                    if half == 0:
                        x.arrive(role, "rdy_fac", n)
                    x.meet(role, f"half {half}", n)
                if not alone and n and half == 0:
                    x.wait(role, "bar_ro", n - 1)
            x.arrive(role, "rdy_prep", n)
            if n + 1 < CHUNKS:
                if not kda and i == 0:
                    x.arrive(role, "rdy_fac", n + 1)
                if not alone and kda:
                    if n:
                        x.wait(role, "bar_s", n - 1)
                    kq(n + 1)
                if not alone:
                    x.wait(role, "bar_ap", n)
                    if kda:
                        x.later(role, "g_full", n + 1)
                    else:
                        kq(n + 1)

    for i, role in enumerate(chain):
        for n in range(CHUNKS):
            x.wait(role, "rdy_fac", n)
            if n:
                x.wait(role, "bar_s", n - 1)
            if alone:
                x.arrive(role, "rdy_half", n)
            x.arrive(role, "rdy_state", n)
            if not alone and with_o and i & 3 >= 2:
                take_p(role, n)
            for bar in ("a_taken", "v_full", "bar_ro"):
                x.wait(role, bar, n)
            x.arrive(role, "rdy_rhs", n)
            x.wait(role, "bar_u", n)
            x.arrive(role, "rdy_u", n)
            if not alone:
                x.wait(role, "bar_o", n)
                if with_o:
                    x.meet(role, "O tile", n)
                x.arrive(role, "tp_free", n)
        x.wait(role, "bar_s", CHUNKS - 1)  # the end of the unit
    return x


FORMS = [(alone, kda, with_o) for alone in (True, False) for kda in (True, False) for with_o in (True, False)]


@pytest.mark.parametrize("alone,kda,with_o", FORMS)
def test_no_wait_can_be_overtaken(alone, kda, with_o):
    assert roles(alone, kda, with_o).overtaken() == set()


@pytest.mark.parametrize("alone,kda,with_o", FORMS)
def test_nothing_arrives_after_the_block_has_left(alone, kda, with_o):
    x = roles(alone, kda, with_o)
    assert x.unwaited <= x.waited


def test_named_barriers_hold_every_warp_that_meets_there():
    # after a time-out the mbarriers hold nobody back any more; warps that only arrived would run ahead and complete a later phase alone
    assert "bar.arrive" not in re.sub(r"//.*", "", open(SOURCE).read())


def test_every_wait_of_the_kernel_is_entered_above():
    text = re.sub(r"//.*", "", open(SOURCE).read())
    outputs = text[text.index("auto outputs ="):text.index("if (warp == WARP_MMA) {", text.index("auto outputs ="))]
    assert "wait_bar" not in outputs  # its callers wait, once per chunk
    assert re.findall(r"(?:if \(.*\) )?mma_commit\(&misc->bar_o\)", text) == ["if (WITH_O || !ALONE) mma_commit(&misc->bar_o)"]
    assert "for (int i = 0; i < 2; ++i) mbar_init(&misc->bar_s[i], 1);" in text  # two in both forms
    sites = defaultdict(int)
    for bar in re.findall(r"wait_bar\(&misc->(\w+)", text):
        sites[bar] += 1
    # (kq_full, g_full: in one place; rdy_prep: in mma1; rdy_rhs: the issuing warp's, take_a's and the triangular warp's; bar_ap: also of the
    # ALONE form's issuing warp; bar_ro: MMA1's warp, two for the producers by KDA / GDN, theirs in ALONE, the chain's; bar_o: the output
    # warps' and the chain's)
    assert dict(sites) == {"rdy_prep": 1, "bar_ap": 5, "rdy_rhs": 3, "tp_free": 2, "bar_o": 2, "rdy_half": 1, "rdy_state": 1, "rdy_t": 1,
                           "bar_u": 2, "rdy_u": 1, "bar_ro": 5, "kq_full": 1, "g_full": 1, "bar_s": 3, "rdy_fac": 1, "a_taken": 1,
                           "v_full": 1}
