"""Host model of the barrier protocol of the fused score kernel: threads stand for the warp roles
of every CTA of one cluster, Python objects for the mbarriers.

What is modelled (names as in the kernel): per CTA a copy role (TMA), an MMA role, TWO exp roles
(the two groups of exp warps alternate heads: group g takes the heads g, g + 2, ...) and an add
role, joined by the barriers
    full / empty      staged keys of a head have landed / have been consumed        (n_q stages)
    tfull             logits of a head are in a tensor-memory buffer                 (n_buf buffers)
    eready            the exponentials of a head are in the buffer
    tempty            the buffer is free again
    sfull             every CTA's (max, sum) pair of a head has arrived in a slot    (n_slot slots)
    xempty            the place of a head's last columns is free again               (176-column tiles: 2 places)
with the phase-parity waits, the transaction counts of the asynchronous statistics stores, the
hand-over (an exp group hands a head's exponentials to the add role at once; ``handover="late"``
models the alternative - only when the group has got to its NEXT head, two heads on - which ends
in time-outs with two buffers: that next head needs the very same buffer), the
"tight" rule (the exp role stays within d heads of the local add role when there are only 2 d
slots) and the bounded waits: a wait that runs out raises the CTA's abort flag, every other wait
of that CTA then returns at once, the CTA records a time-out, tells its peers before the exit
barrier of the cluster, and the request is marked invalid (kept_cnt = -1).

Tiles of 176 columns (``extra=True``): the logits of a head's last columns go to one of two places of
their own, and the exp role gives a place back as soon as it has taken them into registers - behind its
wait for ``tfull``, and under the tight rule behind the wait for the add role as well; the MMA role
waits for the place that head h - 2 used.  ``keep_place=True``: the exp role gives it back only at its
next head, two heads on, whose MMAs wait for it - every wait runs out.

Grid plans (``grid=True``): the CTAs of the request are no cluster; the exp role leaves its pair in
the CTA's own memory and arrives on ``gsent``; a publishing role stores the pair to (modelled)
global memory and adds one to the head's counter; a fetch role waits until the counter shows every
CTA, copies the head's pairs into a statistics slot and completes the slot's barrier - it learns
that a slot is free from the buffer barrier (``tempty``) of the head that used it, by parity.  The
fetch role is a warp: one lane acquires each counter, all lanes copy.  ``lanes_meet=False`` leaves out
the warp barrier between the two, without which the other lanes' copies are not ordered behind it.

``Meeting`` models the end of the score part in the one-launch filter: who has stored its scores - and,
with head groups, staged its head sums - before whom they are read.

The model checks what the kernel relies on: no statistics slot is written before its previous
content has been read, no buffer is refilled before it was released, every head is processed
exactly once per CTA, and a missing arrive ends in a clean time-out everywhere instead of a hang.
"""
import threading
import time

OK, TIMEOUT = 0, 6          # MUSTDROP_OK, MUSTDROP_ERR_TIMEOUT
N_GROUPS = 2                # groups of exp warps per CTA; they alternate heads
LANES = 4                   # lanes of a (short) warp


class ProtocolError(AssertionError):
    pass


class Mbarrier:
    """An mbarrier with an arrival count and a transaction count; a phase completes when both
    reach zero.  Transactions may be counted before the phase's expectation is armed."""

    def __init__(self, count):
        self.count = count
        self.pending = count
        self.tx = 0
        self.phase = 0
        self.lock = threading.Lock()

    def _maybe_complete(self):
        if self.pending == 0 and self.tx == 0:
            self.phase ^= 1
            self.pending = self.count

    def arrive(self, expect_tx=0):
        with self.lock:
            self.tx += expect_tx
            self.pending -= 1
            if self.pending < 0:
                raise ProtocolError("more arrivals than the barrier was initialised for")
            self._maybe_complete()

    def complete_tx(self, n):
        with self.lock:
            self.tx -= n
            self._maybe_complete()

    def try_wait(self, parity):
        with self.lock:
            return self.phase != parity     # the phase with this parity has completed


class Cta:
    def __init__(self, cluster, rank, geo):
        self.cluster, self.rank, self.geo = cluster, rank, geo
        self.abort = False
        self.status = OK
        self.full = [Mbarrier(1) for _ in range(geo["n_q"])]
        self.empty = [Mbarrier(1) for _ in range(geo["n_q"])]
        self.tfull = [Mbarrier(1) for _ in range(geo["n_buf"])]
        self.eready = [Mbarrier(1) for _ in range(geo["n_buf"])]
        self.tempty = [Mbarrier(1) for _ in range(geo["n_buf"])]
        self.sfull = [Mbarrier(1) for _ in range(geo["n_slot"])]
        self.xempty = [Mbarrier(1) for _ in range(2)]
        self.place = [None] * 2             # head whose last columns' logits lie there
        self.gsent = [Mbarrier(1) for _ in range(geo["n_buf"])]     # grid plans: exp role -> publishing role
        self.own_pair = [None] * geo["n_buf"]
        self.stats = [[None] * geo["C"] for _ in range(geo["n_slot"])]   # head whose pair sits there
        self.stage_head = [None] * geo["n_q"]
        self.buf_state = [("free", None)] * geo["n_buf"]
        self.added = []                     # heads the add role finished, in order
        self.guard = threading.Lock()

    def wait(self, bar, parity, limit):
        """Bounded wait: False when it ran out or the CTA has already given up."""
        t0 = time.monotonic()
        while not bar.try_wait(parity):
            if self.abort or time.monotonic() - t0 > limit:
                self.abort = True
                return False
            time.sleep(0.0002)
        return True


class Cluster:
    """One request: C CTAs x 5 roles.  fault = (rank, role, head, what) makes that role skip one
    arrive ("full", "tfull", "eready", "tempty", "empty", "xempty") or one statistics store ("stats")."""

    def __init__(self, C=2, H=12, n_q=2, n_buf=3, n_slot=None, tight=0, limit=0.25, fault=None, jitter=None,
                 grid=False, handover="auto", lanes_meet=True, extra=False, keep_place=False):
        n_slot = (min(n_buf, 4) if grid else 2 * n_buf) if n_slot is None else n_slot
        self.grid = grid
        self.g_lock = threading.Lock()
        self.g_cnt = [0] * H                       # global memory: pairs published per head
        self.g_pairs = [[None] * C for _ in range(H)]
        self.geo = dict(C=C, H=H, n_q=n_q, n_buf=n_buf, n_slot=n_slot, tight=tight)
        # "auto": what the kernel does (at once); "late": one head of the group later
        self.eager = handover == "auto"
        self.limit, self.fault, self.jitter, self.lanes_meet = limit, fault, jitter or {}, lanes_meet
        self.extra, self.keep_place = extra, keep_place
        self.ctas = [Cta(self, r, self.geo) for r in range(C)]
        self.errors = []
        self.cluster_abort = False
        self.kept_cnt = None

    def _skips(self, rank, role, h, what):
        return self.fault == (rank, role, h, what)

    def _pause(self, rank, role):
        d = self.jitter.get((rank, role), 0.0)
        if d:
            time.sleep(d)

    # ---- the roles ---------------------------------------------------------------------------------
    def tma(self, c):
        g = self.geo
        for h in range(g["H"]):
            s = h % g["n_q"]
            if not c.wait(c.empty[s], ((h // g["n_q"]) & 1) ^ 1, self.limit):
                return
            self._pause(c.rank, "tma")
            if c.stage_head[s] is not None:
                raise ProtocolError("stage %d refilled before head %s was consumed" % (s, c.stage_head[s]))
            c.stage_head[s] = h
            if not self._skips(c.rank, "tma", h, "full"):
                c.full[s].arrive()

    def mma(self, c):
        g = self.geo
        for h in range(g["H"]):
            s, buf = h % g["n_q"], h % g["n_buf"]
            if not c.wait(c.full[s], (h // g["n_q"]) & 1, self.limit):
                return
            if not c.wait(c.tempty[buf], ((h // g["n_buf"]) & 1) ^ 1, self.limit):
                return
            if self.extra and not c.wait(c.xempty[h & 1], ((h >> 1) & 1) ^ 1, self.limit):
                return
            self._pause(c.rank, "mma")
            if c.stage_head[s] != h:
                raise ProtocolError("MMA of head %d found head %s staged" % (h, c.stage_head[s]))
            with c.guard:
                if c.buf_state[buf][0] != "free":
                    raise ProtocolError("buffer %d overwritten while %s" % (buf, c.buf_state[buf],))
                c.buf_state[buf] = ("logits", h)
                if self.extra:
                    if c.place[h & 1] is not None:
                        raise ProtocolError("place %d overwritten before head %s was taken" % (h & 1, c.place[h & 1]))
                    c.place[h & 1] = h
            c.stage_head[s] = None
            if not self._skips(c.rank, "mma", h, "empty"):
                c.empty[s].arrive()
            if self._skips(c.rank, "mma", h, "tfull"):
                return      # MMAs complete in order: if this head's never do, no later commit arrives either
            c.tfull[buf].arrive()

    def exp(self, c, grp=0):
        g = self.geo
        last = None                                   # head this group worked on before, not yet handed over
        for h in range(grp, g["H"], N_GROUPS):
            buf, slot = h % g["n_buf"], h % g["n_slot"]
            if g["tight"] and h >= g["tight"]:
                u = h - g["tight"]
                if not c.wait(c.tempty[u % g["n_buf"]], (u // g["n_buf"]) & 1, self.limit):
                    return
            if not c.wait(c.tfull[buf], (h // g["n_buf"]) & 1, self.limit):
                return
            if not self.grid:
                c.sfull[slot].arrive(expect_tx=g["C"])    # arm: every CTA will send one pair
            if self.extra:
                self._pause(c.rank, "take")
                with c.guard:
                    if c.place[h & 1] != h:
                        raise ProtocolError("exp role of head %d found the last columns of head %s" % (h, c.place[h & 1]))
                    c.place[h & 1] = None
                if not self.keep_place and not self._skips(c.rank, "exp", h, "xempty"):
                    c.xempty[h & 1].arrive()
            if last is not None:                          # late hand-over of the group's previous head
                if not self._skips(c.rank, "exp", last, "eready"):
                    c.eready[last % g["n_buf"]].arrive()
                last = None
            self._pause(c.rank, "exp")
            with c.guard:
                if c.buf_state[buf] != ("logits", h):
                    raise ProtocolError("exp role of head %d found %s" % (h, c.buf_state[buf],))
                c.buf_state[buf] = ("exps", h)
            if self.grid:
                if c.own_pair[buf] is not None:
                    raise ProtocolError("own pair of buffer %d overwritten before head %s was added" % (buf, c.own_pair[buf]))
                c.own_pair[buf] = h
                if not self._skips(c.rank, "exp", h, "stats"):
                    c.gsent[buf].arrive()
            elif not self._skips(c.rank, "exp", h, "stats"):
                for peer in self.ctas:                    # st.async into every CTA, counted on ITS barrier
                    with peer.guard:
                        if peer.stats[slot][c.rank] is not None:
                            raise ProtocolError("slot %d of CTA %d overwritten: head %s unread, head %d arrives"
                                                % (slot, peer.rank, peer.stats[slot][c.rank], h))
                        peer.stats[slot][c.rank] = h
                    peer.sfull[slot].complete_tx(1)
            if self.eager:
                if not self._skips(c.rank, "exp", h, "eready"):
                    c.eready[buf].arrive()
            else:
                last = h
        if last is not None and not self._skips(c.rank, "exp", last, "eready"):
            c.eready[last % g["n_buf"]].arrive()          # the last head the group worked on

    def exp1(self, c):
        self.exp(c, 1)

    def add(self, c):
        g = self.geo
        for h in range(g["H"]):
            buf, slot = h % g["n_buf"], h % g["n_slot"]
            if not c.wait(c.sfull[slot], (h // g["n_slot"]) & 1, self.limit):
                return
            with c.guard:
                if c.stats[slot] != [h] * g["C"]:
                    raise ProtocolError("add role of head %d read pairs of heads %s" % (h, c.stats[slot]))
                c.stats[slot] = [None] * g["C"]
                if self.grid:
                    if c.own_pair[buf] != h:
                        raise ProtocolError("add role of head %d found own pair of head %s" % (h, c.own_pair[buf]))
                    c.own_pair[buf] = None
            if not c.wait(c.eready[buf], (h // g["n_buf"]) & 1, self.limit):
                return
            self._pause(c.rank, "add")
            with c.guard:
                if c.buf_state[buf] != ("exps", h):
                    raise ProtocolError("add role of head %d found %s" % (h, c.buf_state[buf],))
                c.buf_state[buf] = ("free", None)
            c.added.append(h)
            if not self._skips(c.rank, "add", h, "tempty"):
                c.tempty[buf].arrive()

    def publish(self, c):
        g = self.geo
        for h in range(g["H"]):
            buf = h % g["n_buf"]
            if not c.wait(c.gsent[buf], (h // g["n_buf"]) & 1, self.limit):
                return
            self._pause(c.rank, "publish")
            with self.g_lock:
                self.g_pairs[h][c.rank] = h
                if not self._skips(c.rank, "publish", h, "count"):
                    self.g_cnt[h] += 1

    def fetch(self, c):
        g = self.geo
        ready = 0                                   # heads below are known to be published
        sees = [set() for _ in range(LANES)]        # heads whose pairs a lane is ordered behind
        for h in range(g["H"]):
            slot = h % g["n_slot"]
            self._pause(c.rank, "fetch_late")       # (a fetch role that gets to its next head late)
            if h >= g["n_slot"]:
                u = h - g["n_slot"]
                if not c.wait(c.tempty[u % g["n_buf"]], (u // g["n_buf"]) & 1, self.limit):
                    return
            t0 = time.monotonic()
            while h >= ready:
                with self.g_lock:                   # lane i looks at head h + i; the run of complete heads is taken
                    for lane in range(LANES):
                        if h + lane >= g["H"] or self.g_cnt[h + lane] < g["C"]:
                            break
                        sees[lane].add(h + lane)
                        ready = h + lane + 1
                if ready > h:
                    if self.lanes_meet:
                        every = set().union(*sees)
                        sees = [set(every) for _ in range(LANES)]
                    break
                if c.abort or time.monotonic() - t0 > self.limit:
                    c.abort = True
                    return
                time.sleep(0.0002)
            self._pause(c.rank, "fetch")
            if not all(h in s for s in sees):
                raise ProtocolError("a lane copies the pairs of head %d unordered behind its counter" % h)
            with c.guard:
                if c.stats[slot] != [None] * g["C"]:
                    raise ProtocolError("slot %d of CTA %d refilled for head %d before heads %s were read"
                                        % (slot, c.rank, h, c.stats[slot]))
                c.stats[slot] = list(self.g_pairs[h])
            c.sfull[slot].arrive()

    # ---- a run ---------------------------------------------------------------------------------------
    def run(self, join_limit=20.0):
        """Run all roles to their common exit.  Returns True when every thread came back."""
        def guarded(fn, c):
            try:
                fn(c)
            except ProtocolError as e:          # a broken invariant: remember it, let the others time out
                self.errors.append(str(e))
                c.abort = True

        roles = (self.tma, self.mma, self.exp, self.exp1, self.add) + ((self.publish, self.fetch) if self.grid else ())
        threads = [threading.Thread(target=guarded, args=(fn, c), daemon=True)
                   for c in self.ctas for fn in roles]
        for t in threads:
            t.start()
        t_end = time.monotonic() + join_limit
        for t in threads:
            t.join(max(0.0, t_end - time.monotonic()))
        if any(t.is_alive() for t in threads):
            return False
        # the common exit: each CTA records its own time-out and tells its peers, cluster barrier,
        # then rank 0 marks the request invalid if anyone gave up
        for c in self.ctas:
            if c.abort:
                c.status = TIMEOUT
                self.cluster_abort = True
        self.kept_cnt = -1 if self.cluster_abort else self.geo["H"]
        return True


class Meeting:
    """The end of the score part of one request in the one-launch filter: from the head sums of its CTAs
    to the selection, which every CTA runs on ALL of the request's scores.  A thread stands for a warp of
    the reducing (exp) warps; ``slow`` maps (CTA, warp) to a delay before that warp's stores.

    Grid plans (``groups`` = 1): a warp stores its share of the CTA's scores to global memory; the CTA's
    warps meet; warp 0 adds one to the request's counter and waits until it shows every CTA; the CTA's
    warps meet again and read all scores.  ``gathered=False`` leaves out the first of the two meetings.

    Head groups (a cluster of groups x C CTAs): the CTAs stage their head sums, meet, add the groups'
    sums for their part of the keys, push the scores into every CTA and meet again.  ``staged=False``
    leaves out the first of these two meetings."""

    def __init__(self, C=3, groups=1, warps=4, grid=True, slow=None, gathered=True, staged=True, limit=5.0):
        self.C, self.groups, self.warps, self.grid = C, groups, warps, grid
        self.n = C * groups
        self.slow, self.gathered, self.staged, self.limit = slow or {}, gathered, staged, limit
        self.cta = [threading.Barrier(warps) for _ in range(self.n)]
        self.cluster = threading.Barrier(self.n * warps)
        # scores[copy][CTA that reduced them][warp]: one copy in global memory, or one per CTA
        self.scores = [[[False] * warps for _ in range(self.n)] for _ in range(1 if grid else self.n)]
        self.sums = [[False] * warps for _ in range(self.n)]
        self.stored, self.lock = 0, threading.Lock()
        self.errors = []

    def _warp(self, cta, w):
        if not self.grid:
            time.sleep(self.slow.get((cta, w), 0.0))
            self.sums[cta][w] = True
            if self.staged:
                self.cluster.wait(self.limit)
            same_keys = range(cta % self.C, self.n, self.C)      # the CTAs of all groups that hold these keys
            if not all(self.sums[c][x] for c in same_keys for x in range(self.warps)):
                self.errors.append("CTA %d warp %d adds head sums that are not staged" % (cta, w))
            for copy in self.scores:
                copy[cta][w] = True
            self.cluster.wait(self.limit)
        else:
            time.sleep(self.slow.get((cta, w), 0.0))
            self.scores[0][cta][w] = True
            if self.gathered:
                self.cta[cta].wait(self.limit)
            if w == 0:
                with self.lock:
                    self.stored += 1
                t0 = time.monotonic()
                while self.stored < self.n and time.monotonic() - t0 < self.limit:
                    time.sleep(0.0002)
                # what the first warp could read as soon as the counter lets it through
                self._check(cta)
            self.cta[cta].wait(self.limit)
        self._check(cta)

    def _check(self, cta):
        if not all(all(ws) for ws in self.scores[0 if self.grid else cta]):
            self.errors.append("CTA %d selects from scores that are not stored" % cta)

    def run(self):
        threads = [threading.Thread(target=self._warp, args=(c, w), daemon=True) for c in range(self.n) for w in range(self.warps)]
        for t in threads:
            t.start()
        for t in threads:
            t.join(2 * self.limit)
        return not any(t.is_alive() for t in threads)
