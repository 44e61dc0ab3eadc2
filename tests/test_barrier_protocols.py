"""Models of the barrier traffic of k_gemm_tc (a pair of CTAs) and k_attn_tc (a CTA), run in random order on the CPU: every
agent ends, and when the last one has, no asynchronous arrival is under way any more.  An arrival that came in later would
land in the shared memory of the CTA that follows on the SM.  Without the closing waits the models show such arrivals."""
import heapq
import os
import random
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2505_19201_b200", "csrc")


class Clock:
    """Asynchronous completions, each after a delay of its own."""

    def __init__(self, rng):
        self.rng, self.now, self.queue, self.n = rng, 0.0, [], 0

    def at(self, when, f):
        self.n += 1
        heapq.heappush(self.queue, (when, self.n, f))

    def later(self, f, lo=0.1, hi=4.0):
        self.at(self.now + self.rng.uniform(lo, hi), f)


class Barrier:
    def __init__(self, count):
        self.count = self.pending = count
        self.tx = self.phase = 0

    def arrive(self):
        assert self.pending > 0
        self.pending -= 1
        self.add(0)

    def add(self, tx):
        self.tx += tx
        if self.pending == 0 and self.tx == 0:
            self.phase, self.pending = self.phase + 1, self.count

    def load(self, clock, boxes):            # expect_tx by one thread, the boxes land one by one
        self.add(boxes)
        self.arrive()
        for _ in range(boxes):
            clock.later(lambda: self.add(-1))

    def done(self, parity):
        return (self.phase & 1) != parity


class Committer:
    """tcgen05.commit: arrives behind the MMAs issued before it, barriers of one commit point at times of their own."""

    def __init__(self, clock):
        self.clock, self.last = clock, 0.0

    def __call__(self, *barriers):
        self.last = max(self.last, self.clock.now) + self.clock.rng.uniform(0.05, 0.6)
        for b in barriers:
            self.clock.at(self.last + self.clock.rng.uniform(0, 1.5), b.arrive)


def play(clock, agents):
    """Arrivals under way when the last agent has ended."""
    idle = 0
    while agents:
        clock.rng.shuffle(agents)
        alive = []
        for g in agents:
            try:
                next(g)
                alive.append(g)
            except StopIteration:
                pass
        agents = alive
        clock.now += 0.1
        while clock.queue and clock.queue[0][0] <= clock.now:
            heapq.heappop(clock.queue)[2]()
        idle = 0 if clock.queue else idle + 1
        assert idle < 500, "nothing under way and nobody moves"
    return len(clock.queue)


def until(cond):
    while not cond():
        yield


def some(rng, most):
    for _ in range(rng.randint(0, most)):
        yield


# ring depths by (head_dim, form): blocks of K and of V, score buffers, buffers of probabilities (AtShape in attn_tc.cuh)
ATTN = {(64, "paged"): (3, 3, 2), (64, "flat"): (4, 3, 2), (64, "prompt"): (3, 3, 2), (128, "paged"): (5, 4, 2), (128, "flat"): (2, 4, 2),
        (128, "prompt"): (2, 2, 1), (256, "paged"): (2, 4, 2), (256, "flat"): (1, 4, 2), (256, "prompt"): (2, 4, 2)}


def attention(shape, n_blk, early, seed, closing=True):
    rng = random.Random(seed)
    stages, s_bufs, p_bufs = ATTN[shape]
    clock = Clock(rng)
    bars = lambda n, count=1: [Barrier(count) for _ in range(n)]
    q_full, k_full, k_empty, v_full, v_empty = bars(1)[0], bars(stages), bars(stages), bars(stages), bars(stages)
    s_full, s_free, p_full, p_empty = bars(s_bufs), bars(s_bufs, 8), bars(p_bufs, 8), bars(p_bufs)
    n_pre = min(early, n_blk, stages)
    # what the buffers hold, to see that nobody reads or overwrites the wrong block
    held = dict(k=[None] * stages, v=[None] * stages, s=[None] * s_bufs, p=[[None] * 8 for _ in range(p_bufs)], o=-1)

    def load(what, full, st, it):
        held[what][st] = it
        full[st].load(clock, 2)

    def producer():
        for i in range(n_pre):
            load("k", k_full, i, i)
            load("v", v_full, i, i)
        q_full.load(clock, 2)
        ks = vs = n_pre % stages
        kph = vph = 0 if n_pre >= stages else 1
        for it in range(n_pre, n_blk + 1):
            if it < n_blk:
                yield from until(lambda: k_empty[ks].done(kph))
                load("k", k_full, ks, it)
                ks, kph = (ks + 1, kph) if ks + 1 < stages else (0, kph ^ 1)
            if it > n_pre:
                yield from until(lambda: v_empty[vs].done(vph))
                load("v", v_full, vs, it - 1)
                vs, vph = (vs + 1, vph) if vs + 1 < stages else (0, vph ^ 1)
        if not closing:
            return
        for _ in range(stages):
            yield from until(lambda: k_empty[ks].done(kph))
            yield from until(lambda: v_empty[vs].done(vph))
            ks, kph = (ks + 1, kph) if ks + 1 < stages else (0, kph ^ 1)
            vs, vph = (vs + 1, vph) if vs + 1 < stages else (0, vph ^ 1)
        for b in range(p_bufs):
            yield from until(lambda: p_empty[b].done(((n_blk + p_bufs - 1 - b) // p_bufs + 1) & 1))

    def s_issuer():
        commit = Committer(clock)
        yield from until(lambda: q_full.done(0))
        ks = sb = kph = 0
        sph = 1
        for it in range(n_blk):
            yield from until(lambda: s_free[sb].done(sph))
            yield from until(lambda: k_full[ks].done(kph))
            assert held["k"][ks] == it
            held["s"][sb] = it
            commit(k_empty[ks], s_full[sb])
            ks, kph = (ks + 1, kph) if ks + 1 < stages else (0, kph ^ 1)
            sb, sph = (sb + 1, sph) if sb + 1 < s_bufs else (0, sph ^ 1)

    def o_issuer():
        commit = Committer(clock)
        vs = vph = 0
        for it in range(n_blk):
            pb = it % p_bufs
            yield from until(lambda: v_full[vs].done(vph))
            yield from until(lambda: p_full[pb].done((it // p_bufs) & 1))
            assert held["v"][vs] == it and held["p"][pb] == [it] * 8
            commit(p_empty[pb], v_empty[vs])
            held["o"] = it
            vs, vph = (vs + 1, vph) if vs + 1 < stages else (0, vph ^ 1)

    def softmax(w):
        sb = sph = 0
        for it in range(n_blk):
            pb = it % p_bufs
            yield from until(lambda: s_full[sb].done(sph))
            assert held["s"][sb] == it
            yield from some(rng, 3)
            s_free[sb].arrive()
            sb, sph = (sb + 1, sph) if sb + 1 < s_bufs else (0, sph ^ 1)
            if it and rng.random() < 0.3:                     # the row's reference moves: behind the O of every earlier block, before this block's
                yield from until(lambda: p_empty[(it - 1) % p_bufs].done(((it - 1) // p_bufs) & 1))
                assert held["o"] == it - 1
                yield from some(rng, 2)
                assert held["o"] == it - 1
            if it >= p_bufs:
                yield from until(lambda: p_empty[pb].done((it // p_bufs - 1) & 1))
                assert held["o"] >= it - p_bufs
            held["p"][pb][w] = it
            yield from some(rng, 3)
            p_full[pb].arrive()
        yield from until(lambda: p_empty[(n_blk - 1) % p_bufs].done(((n_blk - 1) // p_bufs) & 1))
        assert held["o"] == n_blk - 1

    return play(clock, [producer(), s_issuer(), o_issuer()] + [softmax(w) for w in range(8)])


@pytest.mark.parametrize("shape", list(ATTN))
def test_attention(shape):
    for n_blk in (1, 2, 3, 4, 5, 6, 7, 11, 33):
        for early in ((0, 1, n_blk) if shape[1] == "paged" else (0,)):
            for seed in range(3):
                assert attention(shape, n_blk, early, seed) == 0


@pytest.mark.parametrize("shape", [(128, "paged"), (128, "prompt"), (256, "flat")])
def test_attention_without_closing_waits(shape):
    assert any(attention(shape, 5, 0, seed, closing=False) for seed in range(40))


def test_attention_shapes(tmp_path):
    """The depths above are those that AtShape gives to the forms that are launched."""
    src = open(os.path.join(CSRC, "attn_tc.cuh")).read()
    shape = src[src.index("template <int HD, bool FLAT, bool PF = false> struct AtShape"):]
    shape = shape[:shape.index("\n};") + 3]
    lines = ["#include <cstddef>", "#include <cstdio>"] + re.findall(r"^#define AT_[A-Z]+ .*$", src, re.M) + [shape, "int main() {"]
    for hd, form in ATTN:
        lines.append("  { using S = AtShape<%d, %s, %s>; printf(\"%%d %%d %%d\\n\", S::STAGES, S::S_BUFS, S::P_BUFS); }"
                     % (hd, str(form == "flat").lower(), str(form == "prompt").lower()))
    (tmp_path / "shape.cpp").write_text("\n".join(lines + ["}"]))
    subprocess.run(["g++", "-std=c++17", "-o", str(tmp_path / "shape"), str(tmp_path / "shape.cpp")], check=True)
    out = subprocess.run([str(tmp_path / "shape")], check=True, capture_output=True, text=True).stdout.split("\n")
    assert [tuple(map(int, line.split())) for line in out if line] == list(ATTN.values())


def gemm(panels, w_stages, x_stages, wp, chain, seed, closing=True):
    """panels: k panels of the pair's segments.  chain: panels per accumulator fill (0: a segment is one fill and only an arrival
    that the issuer waits for is sent, the forms of up to 128 rows)."""
    rng = random.Random(seed)
    clock = Clock(rng)
    bars = lambda n, count=1: [Barrier(count) for _ in range(n)]
    empty_w, full_w, full_x = [bars(w_stages), bars(w_stages)], bars(w_stages), bars(x_stages)
    acc_full, acc_empty = [bars(2), bars(2)], bars(2, 16)

    def w_producer(rank):
        s, ph = 0, 1
        for k in panels:
            for kb in range(0, k, wp):
                yield from until(lambda: empty_w[rank][s].done(ph))
                if rank == 0:
                    full_w[s].load(clock, 2 * min(wp, k - kb))      # its own boxes and the second CTA's
                s, ph = (s + 1, ph) if s + 1 < w_stages else (0, ph ^ 1)
        for _ in range(w_stages if closing else 0):
            yield from until(lambda: empty_w[rank][s].done(ph))
            s, ph = (s + 1, ph) if s + 1 < w_stages else (0, ph ^ 1)

    def x_producer(rank):
        yield from some(rng, 30)
        s = ws = wph = 0
        free = x_stages
        for k in panels:
            for kb in range(0, k, wp):
                if free:
                    free -= 1
                else:
                    yield from until(lambda: empty_w[rank][ws].done(wph))
                    ws, wph = (ws + 1, wph) if ws + 1 < w_stages else (0, wph ^ 1)
                if rank == 0:
                    full_x[s].load(clock, 2 * min(wp, k - kb))
                s = (s + 1) % x_stages

    fills = [[min(chain, k - a) for a in range(0, k, chain)] if chain else [k] for k in panels]

    def issuer():
        commit = Committer(clock)
        ws = xs = wph = xph = fill = 0
        for segment in fills:
            for k in segment:
                buf, use = fill & 1, fill >> 1
                fill += 1
                yield from until(lambda: acc_empty[buf].done((use & 1) ^ 1))
                for _ in range(0, k, wp):
                    yield from until(lambda: full_w[ws].done(wph) and full_x[xs].done(xph))
                    commit(empty_w[0][ws], empty_w[1][ws])
                    ws, wph = (ws + 1, wph) if ws + 1 < w_stages else (0, wph ^ 1)
                    xs, xph = (xs + 1, xph) if xs + 1 < x_stages else (0, xph ^ 1)
                commit(acc_full[0][buf], acc_full[1][buf])
        for buf in (0, 1) if chain and closing else ():
            yield from until(lambda: acc_empty[buf].done((((fill + 1 - buf) >> 1) & 1) ^ 1))

    def epilogue(rank):
        fill = 0
        for segment in fills:
            for _ in segment:
                buf = fill & 1
                yield from until(lambda: acc_full[rank][buf].done((fill >> 1) & 1))
                fill += 1
                yield from some(rng, 4)
                if chain or fill + 1 < len(panels):
                    clock.later(acc_empty[buf].arrive, 0, 3)         # relaxed and remote: it lands when it lands

    return play(clock, [w_producer(0), w_producer(1), x_producer(0), x_producer(1), issuer()] + [epilogue(r) for r in (0, 1) for _ in range(8)])


@pytest.mark.parametrize("panels", [[1], [3], [32], [25, 39], [7, 64, 46], [64, 64, 64, 20], [1, 1, 1]])
@pytest.mark.parametrize("w_stages,x_stages,wp,chain", [(6, 3, 2, 0), (10, 6, 1, 0), (9, 4, 1, 0), (7, 6, 1, 8), (5, 4, 1, 8), (5, 5, 1, 8)])
def test_gemm_pair(panels, w_stages, x_stages, wp, chain):
    for seed in range(2):
        assert gemm(panels, w_stages, x_stages, wp, chain, seed) == 0


def test_gemm_pair_without_closing_waits():
    assert any(gemm([25, 39], 5, 4, 1, 8, seed, closing=False) for seed in range(20))


def test_pair_holds_tmem_between_barriers_that_show_its_partner_running():
    """tcgen05.alloc and .dealloc of a pair are acts of both CTAs; with the first issued before the start barrier (and the second with
    nothing behind it) a launch hung once in some ten million."""
    src = open(os.path.join(CSRC, "gemm_tc.cuh")).read()
    body = src[src.index("k_gemm_tc(const __grid_constant__"):]
    alloc, release, free = (body.index("tcgen05." + op + ".cta_group::2") for op in ("alloc", "relinquish_alloc_permit", "dealloc"))
    assert body.index("cluster_sync_all();") < alloc
    closing = body.index("cluster_sync_relaxed();")
    assert alloc < release < closing < free < body.index("cluster_sync_relaxed();", closing + 1)
