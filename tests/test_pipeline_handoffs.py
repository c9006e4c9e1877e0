"""The hand-offs of attn_pipe_kernel, played through on the host: every stage's waits and arrivals in the order of the kernel, over
random pieces, restarts and orders of the warps' steps.  No warp may be left waiting, no buffer may be written before its readers have
left it -- the accumulators while a product adds to them or a group reads them, the P tiles that carry a group's sums at the end of a
piece, among them --, and no barrier may be two phases ahead of somebody who waits for it (a wait knows the parity of a phase only).  Barrier ids
and the order in which a CTA gives its memory back are read from the source."""
import os
import random
import re
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_01831_b200", "csrc")


def _code():
    return re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "attention_pipe.cuh")).read())


class Bar:
    """An mbarrier: completes a phase with every `count` arrivals."""
    def __init__(self, count):
        self.count, self.left, self.done = count, count, 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.done = self.count, self.done + 1


def _wait(bar, phase):
    """Waits for phase number `phase` (-1: one before the first) as the kernel does, by its parity."""
    while True:
        assert bar.done <= phase + 2, "two phases ahead of a waiter"
        if (bar.done - 1) % 2 == phase % 2:
            assert bar.done >= phase + 1, "let through before the phase"
            return
        yield


def _play(pieces, SG, NB, NV, PB, NT, ring_k, ring_v, rng):
    NP, n = 4 * PB, sum(pieces)
    B = lambda k, c: [Bar(c) for _ in range(k)]  # noqa: E731
    kfull, kempty, vfull, vempty = B(ring_k, 2), B(ring_k, 4), B(ring_v, 1), B(ring_v, 4)
    mfull, mfree, qfull, qempty, qready = B(NT, 1), B(NT, 4), B(2, 1), B(2, 4 * SG + 3), B(2, 2)
    kready, sfull, sfree = B(NB, 4), B(NB, 1), B(NB, 4)
    vready, pready, pvdone = B(NV, 4), B(SG * PB, 4), B(NP, 1)
    users = {}                      # buffer -> unit that is in it, and how many may still read it
    restart = [rng.random() < 0.3 for _ in range(n)]      # a unit that raises its group's references
    adding, reading, mail = [False] * SG, [0] * SG, [False] * SG   # a P.V, warps that read the sums, sums in the group's P tiles

    def put(buf, unit, readers, writers=1):
        old = users.get(buf)
        if old and old[0] == unit:
            return
        assert old is None or old[1] == 0, (buf, unit, old)
        users[buf] = [unit, readers]

    def get(buf, unit):
        assert users[buf][0] == unit and users[buf][1] > 0, (buf, unit, users[buf])
        users[buf][1] -= 1

    def producer(full, empty, ring, name, readers, publish):
        gs = 0
        for ic, m in enumerate(pieces):
            if publish:
                if ic >= 2:
                    yield from _wait(qempty[ic % 2], ic // 2 - 1)
                put(("item", ic % 2), ic, 4 * SG + 3)
                qfull[ic % 2].arrive()
            for _ in range(m):
                yield from _wait(empty[gs % ring], gs // ring - 1)
                put((name, gs % ring), gs, readers)
                yield
                full[gs % ring].arrive()
                gs += 1

    def k_warp():
        for gs in range(n):
            yield from _wait(kfull[gs % ring_k], gs // ring_k)
            yield from _wait(sfull[gs % NB], gs // NB - 1)
            put(("klev", gs % NB), gs, 1)
            yield
            get(("kraw", gs % ring_k), gs)
            kempty[gs % ring_k].arrive()
            yield
            kready[gs % NB].arrive()

    def v_warp():
        for gs in range(n):
            yield from _wait(vfull[gs % ring_v], gs // ring_v)
            yield from _wait(pvdone[(gs + NP - NV) % NP], (gs + NP - NV) // NP - 1)
            put(("vtile", gs % NV), gs, 1)
            yield
            get(("vraw", gs % ring_v), gs)
            vempty[gs % ring_v].arrive()
            vready[gs % NV].arrive()

    def qk():
        gs = 0
        for ic, m in enumerate(pieces):
            yield from _wait(qfull[ic % 2], ic // 2)
            yield from _wait(qready[ic % 2], ic // 2)
            for _ in range(m):
                yield from _wait(kready[gs % NB], gs // NB)
                yield from _wait(sfree[gs % NB], gs // NB - 1)
                put(("s", gs % NB), gs, 4)
                yield
                get(("klev", gs % NB), gs)
                sfull[gs % NB].arrive()
                gs += 1
            get(("item", ic % 2), ic)
            qempty[ic % 2].arrive()

    def pv():
        for gs in range(n):
            gb = gs % SG * PB + gs // SG % PB
            yield from _wait(vready[gs % NV], gs // NV)
            yield from _wait(pready[gb], gs // (SG * PB))
            assert reading[gs % SG] == 0, "a product into sums that are being read"
            adding[gs % SG] = True
            yield
            adding[gs % SG] = False
            get(("vtile", gs % NV), gs)
            get(("p", gb), gs)
            pvdone[gs % NP].arrive()

    def queries():
        for ic in range(len(pieces)):
            yield from _wait(qfull[ic % 2], ic // 2)
            yield
            qready[ic % 2].arrive()
            get(("item", ic % 2), ic)
            qempty[ic % 2].arrive()

    meet = {}

    def together(key, count):
        meet[key] = meet.get(key, 0) + 1
        while meet[key] < count:
            yield

    def read_sums(g):
        assert not adding[g], "sums read under a product"
        reading[g] += 1
        yield
        assert not adding[g]
        reading[g] -= 1

    def softmax(g, w):
        base = 0
        for ic, m in enumerate(pieces):
            yield from _wait(qfull[ic % 2], ic // 2)
            last = None
            if (g + SG - base % SG) % SG < m:
                yield from _wait(qready[ic % 2], ic // 2)
            for u in range((g + SG - base % SG) % SG, m, SG):
                last = gs = base + u
                gb = g * PB + gs // SG % PB
                yield from _wait(mfull[gs % NT], gs // NT)
                yield from _wait(sfull[gs % NB], gs // NB)
                yield
                get(("s", gs % NB), gs)
                get(("meta", gs % NT), gs)
                sfree[gs % NB].arrive()
                mfree[gs % NT].arrive()
                if gs >= SG * PB:
                    yield from _wait(pvdone[(gs - SG * PB) % NP], (gs - SG * PB) // NP)
                yield from together(("vote", gs), 4)
                if restart[gs] and gs - SG >= base:           # (not a piece's first unit: nothing to drain)
                    if PB > 1:
                        yield from _wait(pvdone[(gs - SG) % NP], (gs - SG) // NP)
                    yield from read_sums(g)
                assert not mail[g], "weights over sums that have not been read"
                put(("p", gb), gs, 1)
                yield
                pready[gb].arrive()
            if last is not None:
                yield from _wait(pvdone[last % NP], last // NP)
                yield from read_sums(g)
            tiles = [users.get(("p", g * PB + i)) for i in range(PB)]
            assert all(t is None or t[1] == 0 for t in tiles), "sums over weights that have not been read"
            mail[g] = True
            yield from together(("mail", ic), 4 * SG)
            assert all(mail), "sums of every group"
            yield from together(("left", ic), 4 * SG)
            mail[g] = False
            get(("item", ic % 2), ic)
            qempty[ic % 2].arrive()
            base += m

    todo = [producer(kfull, kempty, ring_k, "kraw", 4, False) for _ in range(2)]
    todo += [producer(vfull, vempty, ring_v, "vraw", 4, True), producer(mfull, mfree, NT, "meta", 4, False), qk(), pv(), queries(), queries()]
    todo += [k_warp() for _ in range(4)] + [v_warp() for _ in range(4)] + [softmax(g, w) for g in range(SG) for w in range(4)]
    idle = 0
    while todo:
        before = sum(b.done * 1000 - b.left for bars in (kfull, kempty, vfull, vempty, mfull, mfree, qfull, qempty, qready, kready, sfull, sfree,
                                                         vready, pready, pvdone) for b in bars) + len(meet) + sum(meet.values()) - 10 ** 6 * len(todo)
        rng.shuffle(todo)
        # (some warps are held up for a while, so that the others run as far ahead as the barriers let them)
        for t in todo[:rng.randint(1, len(todo))]:
            try:
                next(t)
            except StopIteration:
                todo.remove(t)
        after = sum(b.done * 1000 - b.left for bars in (kfull, kempty, vfull, vempty, mfull, mfree, qfull, qempty, qready, kready, sfull, sfree,
                                                        vready, pready, pvdone) for b in bars) + len(meet) + sum(meet.values()) - 10 ** 6 * len(todo)
        idle = idle + 1 if before == after else 0
        assert idle < 2000, "warps wait for one another"


# softmax groups, scores, V tiles, P tiles of a group, metadata, rings: PipeCfg's at full codes with 16 columns, Anchor with 16, full and
# Anchor below
CONFIGS = [(3, 3, 3, 2, 6, 3, 3), (3, 3, 3, 2, 8, 5, 6), (4, 4, 3, 1, 8, 4, 4), (4, 4, 3, 1, 8, 8, 8)]


@pytest.mark.parametrize("cfg", CONFIGS)
def test_no_warp_waits_for_ever_and_no_buffer_is_taken_early(cfg):
    for seed in range(12):
        rng = random.Random(seed)
        pieces = [rng.choice([1, 1, 2, 3, 5, 9, 20]) for _ in range(rng.randint(1, 8))]
        _play(pieces, *cfg, rng)


def test_the_games_configurations_are_the_kernels(tmp_path):
    """PipeCfg as it stands in the source, compiled for the host: every pair of full codes or not and columns."""
    text = open(os.path.join(CSRC, "attention_pipe.cuh")).read()
    cfg = re.search(r"template <bool FULL, int CP>\nstruct PipeCfg \{.*?\n\};\n", text, re.S).group(0)
    units = re.search(r"constexpr int kI8PieceUnits = \d+;", open(os.path.join(CSRC, "attention_i8.cuh")).read()).group(0)
    show = "".join(f"show<PipeCfg<{f}, {cp}>>();" for f in ("true", "false") for cp in (4, 8, 16))
    src, exe = tmp_path / "c.cpp", tmp_path / "c"
    src.write_text("#include <cstdint>\n#include <cstdio>\n" + units + "\n" + cfg + """
template <class C> void show() {
  std::printf("%d %d %d %d %d %d %d %d\\n", C::kSG, C::kNB, C::kNV, C::kPB, C::kNT, C::kRingK, C::kRingV, C::kNP);
}
int main() {""" + show + "}")
    subprocess.run(["g++", "-std=c++17", "-x", "c++", str(src), "-o", str(exe)], check=True)
    lines = [tuple(map(int, x.split())) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(lines) == 6 and {x[:7] for x in lines} == set(CONFIGS) and all(x[7] == 4 * x[3] for x in lines)


def test_memory_is_given_back_behind_what_is_in_flight():
    code = _code()
    done, land, free = (re.search(x, code).start() for x in (r"named_bar\(9, C::kDoneThreads\)", r"land_after_abort\(", r"tcgen05\.dealloc"))
    assert done < land < free
    assert len(re.findall(r"bar_arrive\(9, C::kDoneThreads\)", code)) == 3 and "abort_word, &maps, 9)" in code


def test_barrier_ids_are_distinct():
    code = _code()
    ids = {int(x) for x in re.findall(r"(?:named_bar|bar_arrive)\((\d+),", code)}
    assert "bar_g = 1 + g" in code and ids == {5, 6, 7, 9}        # 1..4 the softmax groups, 14 i8_join_shared's
