"""Host-side interpreter of the spine programs in the layout that the spine kernels read (emo_graph_spine_layout), in numpy,
vectorised over the policies.  It follows the kernels' division of work and their order: look-up chunks into words of sums, the
spine's operations a bundle at a time (all operands before any result), the pushers' records, backward the completion walk in
its streams, the storing workers' chunks.  Words that no one has written are poison, columns of rows without a policy random, and
what the kernels rely on is asserted: results of a bundle in different places, words that stay zero, records inside their ranges.

`late_stores` delays a stage's stores until just before the spine starts the stage two further on; `extra` takes the storing
form that also gives ES and LS (a tail for every member), else the form for slack alone (tails only in chunks with folds)."""
from __future__ import annotations

import numpy as np

NONE = 0xFFFFFFFF
M32 = np.uint64(0xFFFFFFFF)
POISON = np.uint64(0xA5A5A5A5)
FIRST, LAST, POP = 1, 2, 128


def _fs(x, d):
    """floor_sub: max(x, d) - d on unsigned 32-bit values held in uint64."""
    return np.maximum(x, np.uint64(d)) - np.uint64(d)


def _words(part, at, count):
    return [int(x) for x in part[at:at + 4 * count].view(np.uint32)]


class _Stage:
    """One stage's buffer of sums."""

    def __init__(self, words, zero, B):
        self.a = np.full((words, B), POISON, dtype=np.uint64)
        self.a[zero] = 0
        self.zero = zero

    def put(self, word, x):
        assert word != self.zero, "the word that stays zero was written"
        self.a[word] = x


def run(v: dict, n: int, lv: np.ndarray, late_stores: bool, extra: bool, seed: int = 0) -> dict:
    lanes, stages, Lp, NB, nlook, chunks = (v[k] for k in ("lanes", "stages", "Lp", "bundle", "nlook", "chunks"))
    B = lv.shape[1]
    rs = np.random.RandomState(seed)
    cols = np.arange(B)
    unread = v["unread_slot"]
    assert chunks + 1 <= v["most_chunks"]

    def column(d, st, e):
        row = int(v["rows"][d][st, e])
        return (lv[row] if row != NONE else rs.randint(0, 256, size=B)).astype(np.int64) & (Lp - 1)

    def bundles(d, st, slots, acc):
        """The spine's operations of a stage."""
        part = v["s"][d][st]
        ops = [_words(part, v["off_ops"][d] + 48 * i, 9) for i in range(int(part[:4].view(np.uint32)[0]) * NB)]
        for i in range(0, len(ops), NB):
            done = []
            for o in ops[i:i + NB]:
                assert all(x % 128 == 0 for x in (o[0], o[1], o[2], o[3], o[6], o[7], o[8]))
                q = np.maximum(_fs(slots[o[0] // 128], o[4]), _fs(slots[o[1] // 128], o[5]))
                done.append((o, q, (q + acc.a[o[2] // 128]) & M32))
            to = [s for o, _, _ in done for s in {o[6] // 128, o[7] // 128} | ({o[3] // 128} if d else set()) if s != unread]
            words = [o[8] // 128 for o, _, _ in done if o[8] // 128 != acc.zero + 1]
            assert len(to) == len(set(to)) and len(words) == len(set(words)), "two results of a bundle in one place"
            assert lanes not in to, "the slot that stays zero was written"
            for o, q, y in done:
                slots[o[6] // 128] = y
                slots[o[7] // 128] = y
                acc.put(o[8] // 128, q if d else y)
                if d:
                    slots[o[3] // 128] = 0

    # ---- forward ----------------------------------------------------------------------------------------
    slots = np.zeros((v["slots_fwd"], B), dtype=np.uint64)
    restore = np.full((int(v["pushes"]) + lanes, B), POISON, dtype=np.uint64)
    T, E = np.zeros(B, dtype=np.int64), np.zeros(B)
    for st in range(stages):
        w, s = v["w"][0][st], v["s"][0][st]
        pos = w[v["off_pos"][0]:].view(np.uint32)
        tab = w[v["off_tab"][0]:v["off_tab"][0] + nlook * Lp * 12].view(np.uint32).reshape(nlook, Lp, 3)
        acc = _Stage(v["words"][0], v["zero"][0], B)
        at = 0
        for c, ck in enumerate(_words(w, 0, chunks)):
            e0, cnt = ck & 0xFFFF, ck >> 16
            assert e0 == at and cnt % 4 == 0 and e0 + cnt <= nlook
            at += cnt
            runsum = np.full(B, POISON)
            for e in range(e0, e0 + cnt):
                pw, l = int(pos[e]), column(0, st, e)
                d = tab[e, l, 0].astype(np.uint64)
                E += ((tab[e, l, 1].astype(np.uint64) << np.uint64(32)) | tab[e, l, 2].astype(np.uint64)).view(np.float64)
                runsum = d if pw & FIRST else (runsum + d) & M32
                if pw & LAST:
                    acc.put(pw >> 16, runsum)
        bundles(0, st, slots, acc)
        _, n_term, n_rec = _words(s, 0, 3)
        for t in range(n_term):
            x, _, lo, hi = _words(s, 16 + 16 * t, 4)
            T = np.maximum(T, np.int64(lo | (hi << 32)) + slots[x // 128].astype(np.int64))
        assert n_rec % 4 == 0
        for i in range(n_rec):
            word, row = _words(s, v["off_rec"][0] + 8 * i, 2)
            if row != NONE:
                assert row < v["pushes"]
                restore[row] = acc.a[word // 128]
    restore[int(v["pushes"]):] = slots[:lanes]

    # ---- backward ---------------------------------------------------------------------------------------
    slots = np.zeros((v["slots_bwd"], B), dtype=np.uint64)
    slots[lanes + 2:2 * lanes + 2] = restore[int(v["pushes"]):]
    comp = v["max_segs"] + 2
    assert v["words"][1] == 2 * comp
    out = {k: np.full((n, B), -1, dtype=np.int64) for k in ("slack", "ES", "LS")}
    kept = {}

    def stores(st):
        acc, w = kept.pop(st), v["w"][1][st]
        tab = w[v["off_tab"][1]:v["off_tab"][1] + (nlook + 1) * Lp * 4].view(np.uint32).reshape(nlook + 1, Lp)
        assert not tab[nlook].any()
        first_bits = w[v["off_first"]:].view(np.uint32)
        at = 0
        for c, ck in enumerate(_words(w, 4 * v["most_chunks"], chunks + 1)):
            e0, cnt, folds = ck & 0xFFFF, (ck >> 16) & 0x7FFF, ck >> 31
            assert cnt % 4 == 0 and (e0 == at if c < chunks else e0 == nlook)
            at += cnt
            q, sl = np.full(B, POISON), np.zeros(B, dtype=np.int64)
            for e in range(e0, e0 + cnt):
                node, fold, corr, pw, a0, a1, b0, b1 = _words(w, v["off_mem"] + 32 * e, 8)
                d = tab[e if c < chunks else nlook][column(1, st, e) if c < chunks else np.zeros(B, np.int64)].astype(np.uint64)
                qn, cn = acc.a[pw >> 16], acc.a[(pw >> 16) + comp]
                first = bool((int(first_bits[e // 32]) >> (e % 32)) & 1)
                assert first == bool(pw & FIRST)
                if extra or not folds:      # everything for every member
                    sl = T - np.int64(a0 | (a1 << 32)) - ((qn + cn) & M32).astype(np.int64)
                elif first:                 # once per segment
                    sl = T - np.int64(a0 | (a1 << 32)) - ((qn + cn) & M32).astype(np.int64)
                q = ((qn if first else q) + d) & M32
                if extra or folds:
                    slots[fold // 128] = np.maximum(slots[fold // 128], _fs(q, corr))
                else:
                    assert fold // 128 == unread
                if node != NONE:
                    assert (out["slack"][node] == -1).all()
                    out["slack"][node] = sl
                    if extra:
                        out["ES"][node] = np.int64(b0 | (b1 << 32)) + ((qn + cn - q) & M32).astype(np.int64)
                        out["LS"][node] = out["ES"][node] + sl

    order = list(range(stages - 1, -1, -1))
    R = 4 if late_stores else 2          # records that a walker holds at once (either, by the policies per thread)
    for k, st in enumerate(order):
        w, s = v["w"][1][st], v["s"][1][st]
        acc = kept[st] = _Stage(v["words"][1], v["zero"][1], B)
        pos = w[v["off_pos"][1]:].view(np.uint32)
        tab = w[v["off_tab"][1]:v["off_tab"][1] + nlook * Lp * 4].view(np.uint32).reshape(nlook, Lp)
        for ck in _words(w, 0, chunks):
            runsum = np.full(B, POISON)
            for e in range(ck & 0xFFFF, (ck & 0xFFFF) + (ck >> 16)):
                pw, d = int(pos[e]), tab[e][column(1, st, e)].astype(np.uint64)
                runsum = d if pw & FIRST else (runsum + d) & M32
                if pw & LAST:
                    acc.put(pw >> 16, runsum)
        base, rows = int(v["push_base"][st]), int(v["push_base"][st + 1]) - int(v["push_base"][st])
        rounds = _words(s, 0, 3)[2]
        assert rounds % 4 == 0
        seen = []
        for stream in range(NB):
            co = np.zeros(B, dtype=np.uint64)
            for i in range(0, rounds, R):
                recs = [_words(s, v["off_rec"][1] + 16 * ((i + j) * NB + stream), 4) for j in range(R)]
                for r in recs:
                    if r[3] & POP:
                        assert (r[3] >> 8) < rows
                loaded = [(acc.a[r[1] // 128].copy(), slots[r[0] // 128].copy(), restore[base + (r[3] >> 8)].copy() if r[3] & POP else None) for r in recs]
                for r, (S, into, pop) in zip(recs, loaded):
                    if r[3] & FIRST:
                        co = into
                    acc.put(r[2] // 128 + comp, co)
                    if r[2] // 128 != acc.zero + 1:
                        seen.append(r[2] // 128)
                    co = pop if pop is not None else (co - S) & M32
                    if r[3] & LAST:
                        slots[r[0] // 128] = co
        assert len(seen) == len(set(seen)), "a segment walked twice"
        if late_stores and k >= 2:
            stores(order[k - 2])          # the spine waits for the stores of the stage two back, no earlier
        bundles(1, st, slots, acc)
        if not late_stores:
            stores(st)
    for st in list(kept):
        stores(st)
    return dict(out, makespan=T, energy=E)
