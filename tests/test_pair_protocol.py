"""The hand-overs of the CTA-pair kernel (csrc/nsp_bwd_pair.cu) as a model on the CPU: its roles, barriers and buffers, run under
random and lopsided delays. Two kinds of fault are looked for. A wait goes by the parity of a phase alone, so a barrier that is
two phases ahead of a waiter holds it for good, and one that is a phase behind lets it through; and every buffer and TMEM region has
to hold the step that its reader means, from the start of the read to its end. A missing wait shows up here without a GPU."""
import heapq
import random
import re
from pathlib import Path

import pytest


class Fault(Exception):
    pass


class Barrier:
    def __init__(self, sim, name, count):
        self.sim, self.name, self.count, self.left, self.phase, self.waiters = sim, name, count, count, 0, []

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.phase = self.count, self.phase + 1
            waiters, self.waiters = self.waiters, []
            for who, look in waiters:  # they wake up some time later
                self.sim.at(0.02 + self.sim.delay(who, "wake"), look)

    def passed(self, k):  # the hardware's test for phase k, by parity, against what is meant
        test = (self.phase & 1) != (k & 1)
        if test != (k < self.phase):
            raise Fault("%s: waits for phase %d, barrier in phase %d" % (self.name, k, self.phase))
        return test


class Cell:
    """A buffer or TMEM region: the step it holds, None while it is being written."""

    def __init__(self, name):
        self.name, self.step, self.readers = name, None, 0

    def check(self, step):
        if self.step != step:
            raise Fault("%s holds step %s, step %d meant" % (self.name, self.step, step))

    def write(self, step):
        if self.readers:
            raise Fault("%s is written for step %d while it is read" % (self.name, step))
        self.step = step


class Sim:
    def __init__(self, items, seed, without=()):
        self.rng, self.now, self.queue, self.n = random.Random(seed), 0.0, [], 0
        self.items, self.without = items, set(without)
        # every run has its own idea of which activities are slow
        self.slow, self.waiting = {}, []
        count = {"qr": 2, "dor": 2, "doc": 2, "qc": 2, "s_read": 16, "p_ready": 16, "ds_ready": 16, "dq_empty": 16, "x_peer": 2}
        self.bar = {n: Barrier(self, n, c) for n, c in count.items()}  # qr ..: one load of each CTA
        for r in (0, 1):
            for n, c in {"s_full": 1, "dp_full": 1, "dq_full": 1, "dv_done": 1, "dk_done": 1, "x_own": 4, "x_full": 4, "ld_full0": 1,
                         "ld_full1": 1, "ld_empty0": 8, "ld_empty1": 8}.items():
                self.bar[n, r] = Barrier(self, "%s of CTA %d" % (n, r), c)
        names = ["q_row", "do_row", "q_col", "do_col", "lse0", "lse1"]
        self.cell = {(n, r): Cell("%s of CTA %d" % (n, r)) for n in names for r in (0, 1)}
        for r in (0, 1):
            for w in range(8):  # a softmax warp's lanes of the regions, its part of dS^T and of P^T
                for n in ("S_lo", "S_hi", "DP_lo", "DP_hi", "P", "DS", "X"):
                    self.cell[n, r, w] = Cell("%s of warp %d of CTA %d" % (n, w, r))
            for w in range(8):
                self.cell["DQ", r, w] = Cell("dQ^T of dQ warp %d of CTA %d" % (w, r))
        self.pipe = {"A": [], "B": []}
        self.busy = {"A": False, "B": False}
        self.meet, self.left = 0, 0

    def delay(self, who, what):
        key = (who, what)
        if key not in self.slow:
            self.slow[key] = self.rng.choice([0.02, 0.1, 0.3, 1.0, 1.0, 4.0, 20.0])
        return self.slow[key] * self.rng.random()

    def at(self, t, f):
        self.n += 1
        heapq.heappush(self.queue, (self.now + t, self.n, f))

    # ---- roles are generators that yield ("wait", [(barrier, phase)..]) or ("work", name)
    def role(self, who, gen):
        def go():
            try:
                kind, arg = next(gen)
            except StopIteration:
                self.left -= 1
                return
            if kind == "work":
                self.at(self.delay(who, arg), go)
            elif kind == "meet":
                self.meet += 1
                if self.meet % self.roles:
                    self.waiting.append(go)
                else:
                    for w in self.waiting + [go]:
                        self.at(0.01, w)
                    self.waiting = []
            else:
                def look():
                    late = [b for b, k in arg if not b.passed(k)]
                    if late:
                        late[0].waiters.append((who, look))
                    else:
                        go()
                look()

        self.left += 1
        self.at(0, go)

    def wait(self, *pairs):
        return "wait", [(self.bar[n], k) for n, k in pairs]

    def skip(self, name):
        return name in self.without

    # ---- asynchronous work
    def load(self, rank, cell, bar, step):
        self.cell[cell, rank].write(None)
        def done():
            self.cell[cell, rank].write(step)
            self.bar[bar].arrive()
        self.at(0.1 + self.delay("load%d" % rank, cell), done)

    def product(self, issuer, name, step, reads, writes, bars, over=()):
        """reads, writes, over (overwritten): cells; bars complete when it and all before it of this issuer have."""
        self.pipe[issuer].append((name, step, reads, writes, bars, over))
        self.pump(issuer)

    def pump(self, issuer):
        if self.busy[issuer] or not self.pipe[issuer]:
            return
        name, step, reads, writes, bars, over = self.pipe[issuer].pop(0)
        self.busy[issuer] = True
        for c in reads:
            c.check(step)
            c.readers += 1
        for c in [*writes, *over]:
            c.write(None)
        def done():
            for c in reads:
                c.check(step)
                c.readers -= 1
            for c in writes:
                c.write(step)
            self.busy[issuer] = False
            for b in bars:
                self.at(0.02, lambda b=b: [self.bar[b, r].arrive() for r in (0, 1)])
            self.pump(issuer)
        self.at(0.2 + self.delay(issuer, name), done)

    def remote(self, rank, bar):
        if rank == 0:
            self.bar[bar].arrive()
        else:
            self.at(0.2, self.bar[bar].arrive)

    def cells(self, name):
        return [self.cell[name, r, w] for r in (0, 1) for w in range(8)]

    # ---- the roles
    def producer(self, r):
        gs = 0
        for steps in self.items:
            yield "meet", 0
            for cell, bar in (("q_row", "qr"), ("do_row", "dor"), ("do_col", "doc"), ("q_col", "qc")):
                self.load(r, cell, bar, gs)
            for vt in range(steps - 1):
                for full, cell, bar in (("s_full", "q_row", "qr"), ("dp_full", "do_row", "dor"), ("dv_done", "do_col", "doc"),
                                        ("dk_done", "q_col", "qc")):
                    yield self.wait(((full, r), gs + vt))
                    self.load(r, cell, bar, gs + vt + 1)
            gs += steps

    def loader(self, r):
        gs = 0
        for steps in self.items:
            yield "meet", 0
            for cs in range(gs, gs + steps):
                yield self.wait((("ld_empty%d" % (cs & 1), r), (cs >> 1) - 1))
                self.cell["lse%d" % (cs & 1), r].write(None)
                yield "work", "lse"
                self.cell["lse%d" % (cs & 1), r].write(cs)
                self.bar["ld_full%d" % (cs & 1), r].arrive()
            gs += steps

    def relay(self, part):
        gs = 0
        for steps in self.items:
            yield "meet", 0
            for cs in range(gs, gs + steps):
                yield self.wait(((part, 1), cs))
                yield "work", "relay"
                self.remote(1, "x_peer")
            gs += steps

    def issuer_a(self):
        gs = 0
        both = lambda n: [self.cell[n, r] for r in (0, 1)]
        for steps in self.items:
            yield "meet", 0
            for vt in range(-1, steps):
                cs = gs + vt
                if vt >= 0:
                    yield self.wait(*([("doc", cs)] + ([("qr", cs + 1)] if vt + 1 < steps else [])))
                    yield self.wait(("p_ready", cs))
                    yield "work", "issue"
                    self.product("A", "dV", cs, self.cells("P") + both("do_col"), [], ["dv_done"])
                else:
                    yield self.wait(("qr", gs))
                if vt + 1 < steps:
                    if vt >= 0:
                        yield self.wait(("dq_empty", cs - 1))
                    yield "work", "issue"
                    # R0: over P^T and dQ^T
                    self.product("A", "S", cs + 1, both("q_row"), self.cells("S_lo") + self.cells("S_hi"), ["s_full"],
                                 self.cells("P") + self.cells("DQ"))
            gs += steps

    def issuer_b(self):
        gs = 0
        both = lambda n: [self.cell[n, r] for r in (0, 1)]
        for steps in self.items:
            yield "meet", 0
            yield self.wait(("dor", gs))
            if not self.skip("s_read ahead of dP"):
                yield self.wait(("s_read", gs))
            self.product("B", "dP", gs, both("do_row"), self.cells("DP_lo") + self.cells("DP_hi"), ["dp_full"], self.cells("DS"))
            for vt in range(steps):
                cs, more = gs + vt, vt + 1 < steps
                yield self.wait(*([("qc", cs)] + ([("dor", cs + 1)] if more else [])))
                yield self.wait(("ds_ready", cs))
                if self.skip("s_read ahead of dP") and vt == 0:
                    yield self.wait(("s_read", cs))
                yield "work", "issue"
                self.product("B", "dK", cs, self.cells("DS") + both("q_col"), [], ["dk_done"])
                if more:
                    self.product("B", "dP", cs + 1, both("do_row"), self.cells("DP_lo") + self.cells("DP_hi"), ["dp_full"], self.cells("DS"))
                last = [] if self.skip("last drain") else [("dq_empty", cs - 1)]
                yield self.wait(*([(("x_own", 0), cs)] + ([("s_read", cs + 1)] if more else last)))
                yield self.wait((("x_full", 0), cs), ("x_peer", cs))
                yield "work", "issue"
                self.product("B", "dQ", cs, self.cells("X"), self.cells("DQ"), ["dq_full"], self.cells("S_hi"))
            gs += steps

    def dq_warp(self, r, w):
        gs = 0
        for steps in self.items:
            yield "meet", 0
            for cs in range(gs, gs + steps):
                yield self.wait((("dq_full", r), cs))
                self.cell["DQ", r, w].check(cs)
                yield "work", "read"
                self.cell["DQ", r, w].check(cs)
                self.remote(r, "dq_empty")
                yield "work", "drain"
            gs += steps

    def softmax(self, r, w):
        keep = (w >= 4) == (r == 1)
        gs = 0
        C = lambda n: self.cell[n, r, w]
        for steps in self.items:
            yield "meet", 0
            for cs in range(gs, gs + steps):
                st = cs & 1
                yield self.wait((("ld_full%d" % st, r), cs >> 1), (("s_full", r), cs))
                C("S_lo").check(cs), C("S_hi").check(cs)
                yield "work", "read S"
                C("S_lo").check(cs), C("S_hi").check(cs)
                self.remote(r, "s_read")
                yield "work", "exp"
                self.cell["lse%d" % st, r].check(cs)
                C("S_lo").check(cs)
                C("P").write(cs)
                self.remote(r, "p_ready")
                yield self.wait((("dp_full", r), cs), (("dq_full", r), cs - 1))
                C("DP_lo").check(cs), C("DP_hi").check(cs)
                C("X").write(None)  # here, or on its way to the other CTA
                yield "work", "dS"
                C("DP_lo").check(cs), C("DP_hi").check(cs)
                self.cell["lse%d" % st, r].check(cs)
                C("DS").write(cs)
                self.remote(r, "ds_ready")
                self.bar["ld_empty%d" % st, r].arrive()
                yield "work", "fence"
                if keep:
                    C("X").write(cs)
                    self.bar["x_own", r].arrive()
                else:
                    def arrived(cs=cs):
                        C("X").write(cs)
                        self.bar["x_full", 1 - r].arrive()
                    self.at(0.1 + self.delay("copy%d" % r, w), arrived)
            gs += steps
            yield self.wait((("dv_done", r), gs - 1))
            yield self.wait((("dk_done", r), gs - 1))
            yield self.wait((("dq_full", r), gs - 1))
            yield "work", "epilogue"

    def run(self):
        roles = [("A", self.issuer_a()), ("B", self.issuer_b()), ("relay17", self.relay("x_own")), ("relay19", self.relay("x_full"))]
        for r in (0, 1):
            roles += [("producer%d" % r, self.producer(r)), ("loader%d" % r, self.loader(r))]
            roles += [("softmax%d.%d" % (r, w), self.softmax(r, w)) for w in range(8)]
            roles += [("dq%d.%d" % (r, w), self.dq_warp(r, w)) for w in range(8)]
        self.roles = len(roles)
        for who, gen in roles:
            self.role(who, gen)
        while self.queue:
            self.now, _, f = heapq.heappop(self.queue)
            f()
        if self.left:
            raise Fault("%d roles wait for good" % self.left)


def faults(runs, **kw):
    found = []
    for seed in range(runs):
        rng = random.Random(seed)
        items = [rng.choice([1, 2, 3, 4, 7]) for _ in range(rng.randint(1, 4))]
        try:
            Sim(items, seed, **kw).run()
        except Fault as e:
            found.append(str(e))
    return found


def test_no_wait_is_missing():
    assert faults(300) == []


@pytest.mark.parametrize("without", ["last drain", "s_read ahead of dP"])
def test_the_model_sees_a_missing_wait(without):
    assert faults(300, without=[without])


def test_the_kernel_has_the_waits_of_the_model():
    text = (Path(__file__).resolve().parent.parent / "paper_2609_22755_b200" / "csrc" / "nsp_bwd_pair.cu").read_text()
    b = text[text.index("const uint32_t v_km = smem_desc_addr"):text.index("if (!okm) {")]
    head, loop = b.split("#pragma unroll 1", 1)
    assert re.search(r"wait\w*\(&s\.bar_s_read, gs & 1.*issue_dp\(", head, re.S)  # ahead of the first dP^T
    # in front of dQ^T: S^T of the next step has been read, or, behind the last step's, dQ^T of the one before has been drained
    dq = loop[loop.index("issue_dp(true)"):loop.index("umma2_ss_lh(tDQ")]
    assert "bar_dq_empty" in dq and loop.count("bar_s_read") == dq.count("bar_s_read") == 1
