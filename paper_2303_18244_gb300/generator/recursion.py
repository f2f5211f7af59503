"""Emit the helicity-shared colour-ordered recursion of g g -> t t~ + gluons.

The per-helicity program (emit.py) evaluates every diagram of every helicity.
Here the colour-ordered amplitudes are built by the Berends-Giele recursion
(F. A. Berends, W. T. Giele, Nucl. Phys. B306 (1988) 759), which sums all
diagrams that share a sub-current, and every current is computed once per
helicity combination of its own external legs instead of once per helicity of
the event.  The group of threads that owns an event runs the stages below one
after the other (a group barrier between them), each stage a list of
independent tasks that read and write 4-component vectors of the event's
store:

  J(word)    off-shell gluon current of the ordered gluons `word`, computed for
             words that start with their smallest gluon; the other orders
             follow from the Kleiss-Kuijf relation
             J(a, m, b) = (-1)^|a| sum over shuffles s of (a reversed, b) J(m, s)
             (R. Kleiss, H. Kuijf, Nucl. Phys. B312 (1989) 616).  Momenta,
             couplings and gluon propagators are real and
             eps(-lambda) = -eps(lambda)*, so the current of m gluons with every
             helicity flipped is (-1)^m J*, bit for bit: half of the helicity
             combinations are computed, each writes its partner too (the lines
             have no such partners: the top's width is complex)
  R(word)    row spinor that left the outgoing top and absorbed `word`
  A(word)    the same before the last propagator (amputated)
  C(word)    column spinor that ends on the antitop, stored as the row of its
             charge conjugate (see mg_recursion.cuh)
  S(P|B)     R(P) Jslash_B, the block B across the cut, B in one order per
             Kleiss-Kuijf basis element
  V(P,S)     vector with V.J = R(P) Jslash C(S)

The amplitude of the ordering w is cut after its first p gluons: either no
gluon current spans the cut, A(w_1..w_p) . C(w_p+1..w_n), or one block does.
"""
from __future__ import annotations

import itertools

from .colour import colour_matrix_exact, common_denominator, words
from .diagrams import build_plan, count_diagrams

CUT = {2: 1, 3: 1, 4: 2, 5: 2}

# the calls that run an emitted header with one thread (host tests), by
# n > 4: currents and flows a[2][NCOL] of gluon bits hg and top spin s
HOST_CURRENTS = ("""P::currents<double>(st, kp, 0, 1, [] {});
    static cx<double> z[32][2][P::NCOL];
    for (int q = 0; q < 2 << P::N; q++)
      P::flows_open<double, 2>(st, q & ((1 << P::N) - 1), q >> P::N, 0, z[q]);
    P::late<double>(st, 0, 1);""",
                 """P::currents<double>(st, kp, 0, 1, [] {});
    static cx<double> z[64][2][P::NCOL];
    for (int q = 0; q < 64; q++)
      P::closings<double, 2>(st, q & 31, q >> 5, 0, [&](int ib, int k, cx<double> v) { z[q][ib][k] = v; });
    P::late<double>(st, kp, 0, 1);""")
HOST_FLOWS = ("""for (int q = 0; q < 2 * P::NCOL; q++) a[q / P::NCOL][q % P::NCOL] = z[hg + (s << P::N)][q / P::NCOL][q % P::NCOL];
        P::flows_block<double, 2>(st, hg, s, 0, a);""",
              """const int q = hg + 32 * s;
        P::all_flows<double, 2>(st, hg, s, 0, [&](int ib, int k) { return z[q][ib][k]; },
                                [&](int ib, int k, cx<double> v) { a[ib][k] = v; });""")


def shuffles(a: tuple, b: tuple):
    if not a or not b:
        yield a + b
        return
    for s in shuffles(a[1:], b):
        yield (a[0],) + s
    for s in shuffles(a, b[1:]):
        yield (b[0],) + s


def kk(word: tuple) -> tuple[int, list[tuple]]:
    """(sign, words starting with the smallest gluon) whose sum is J(word)."""
    m = min(word)
    i = word.index(m)
    a, b = word[:i], word[i + 1:]
    return (-1) ** len(a), [(m,) + s for s in shuffles(tuple(reversed(a)), b)]


def basis(gluons) -> list[tuple]:
    g = sorted(gluons)
    return [(g[0],) + s for s in itertools.permutations(g[1:])]


class Recursion:
    """Store layout, stage task tables and contraction terms for n gluons."""

    def __init__(self, n: int):
        self.n, self.p = n, CUT[n]
        self.full = (1 << n) - 1
        self.items: dict = {}      # key -> (gluons sorted, spin bits)
        self.tasks: dict = {}      # stage name -> list of items to compute
        self.base: dict = {}
        self._lev: dict = {}
        self._collect()
        self._layout()

    # -- what is needed -------------------------------------------------
    def _item(self, key, gluons, spins):
        if key in self.items:
            return False
        # helicity index bits: gluons in increasing order, but the last gluon of a
        # column (next to the antitop) last
        tail = ()
        if key[0] == "C" and key[1]:
            tail = key[1][-1:]
        elif key[0] == "V" and key[2]:
            tail = key[2][-1:]
        self.items[key] = (tuple(sorted(g for g in gluons if g not in tail)) + tail, spins)
        return True

    def jkey(self, word):
        """Store key of J(word): triples are equal to their reversal."""
        word = tuple(word)
        if len(word) == 3 and (word[2] < word[0]):
            word = word[::-1]
        return ("J", word)

    def need_j(self, word):
        key = self.jkey(word)
        word = key[1]
        if not self._item(key, word, 0):
            return
        m = len(word)
        if m == 1:
            return
        if m == 2:
            self.need_j(word[::-1])
            for i in word:
                self.need_j((i,))
            if word[0] < word[1]:
                self.tasks.setdefault("J2", []).append(key)
            return
        if word[0] == min(word):
            for i in range(m):
                for j in range(i + 1, m + 1):
                    if j - i < m:
                        self.need_j(word[i:j])
            self.tasks.setdefault(f"J{m}", []).append(key)
        else:
            for w in kk(word)[1]:
                self.need_j(w)
            self.tasks.setdefault(f"K{m}", []).append(key)

    def need_line(self, kind, word):
        key = (kind, tuple(word))
        if not self._item(key, word, 1):
            return
        m = len(word)
        for i in range(m):  # block next to the cut, the rest next to the top
            if kind == "C":
                self.need_j(word[:m - i])
                self.need_line("C", word[m - i:])
            else:
                self.need_j(word[i:])
                self.need_line("R", word[:i])
        if m:
            self.tasks.setdefault(f"{kind}{m}", []).append(key)

    def spanning(self):
        """(prefix, block set, suffix, closing kind) of every term with a block across the cut."""
        n, p = self.n, self.p
        for lp in range(p):
            for ls in range(n - p):
                m = n - lp - ls
                if m < 2:
                    continue
                for pre in itertools.permutations(range(n), lp):
                    rest = [g for g in range(n) if g not in pre]
                    for suf in itertools.permutations(rest, ls):
                        yield pre, tuple(g for g in rest if g not in suf), suf

    def closing(self, lp, ls, m):
        """"S": spinor R(P)Jslash_B dotted with C(S); "V": V(P,S) dotted with J_B."""
        return "S" if (self.n, lp, ls) in ((4, 1, 1), (5, 1, 2), (5, 0, 2)) else "V"

    def _collect(self):
        n, p = self.n, self.p
        for i in range(n):
            self.need_j((i,))
        for w in itertools.permutations(range(n), p):
            self.need_line("A", w)
        for w in itertools.permutations(range(n), n - p):
            self.need_line("C", w)
        for pre, blk, suf in self.spanning():
            for b in basis(blk):
                self.need_j(b)
            self.need_line("R", pre)
            self.need_line("C", suf)
            if self.closing(len(pre), len(suf), len(blk)) == "S":
                for b in basis(blk):
                    if self._item(("S", pre, b), pre + b, 1):
                        self.tasks.setdefault("S", []).append(("S", pre, b))
            elif self._item(("V", pre, suf), pre + suf, 2):
                self.tasks.setdefault("V", []).append(("V", pre, suf))

    # -- layout ----------------------------------------------------------
    def _size(self, key):
        g, sp = self.items[key]
        return 1 << (len(g) + sp)

    def _layout(self):
        """Store positions.  Items written after others are dead share space
        (`late`).  Four gluons: the spinors S, over A and C of two gluons, once
        the flows without a block across the cut are closed.  Five: the columns C of three gluons, over the currents that
        only the full-length closing and the longer currents read."""
        def dead_early(key):
            m = len(key[1])
            if self.n == 4:
                return m == 2 and key[0] in "AC"
            return self.n == 5 and key[0] == "J" and (m == 5 or (m == 4 and key[1][0] != min(key[1])))

        def order(key):
            """Five gluons: items that the closing of one last gluon e reads
            together are consecutive, so that their positions are affine in e."""
            if self.n < 5:
                return ()
            w = key[1]
            if key[0] == "C" and w:
                return ("C", len(w), w[-1:] + w[:-1])
            if key[0] == "V":
                return ("V", len(w) + 10 * len(key[2]), key[2][-1:] + w)
            if key[0] == "J" and len(w) == 4 and w[0] == min(w):
                return ("J", 4, (min(set(range(5)) - set(w)),) + w)
            return (key[0], len(w), w)

        def place(keys, pos):
            for key in sorted(keys, key=order):
                self.base[key] = pos
                pos += self._size(key)
            return pos
        first = place([k for k in self.items if dead_early(k)], 0)
        second = place([k for k in self.items if self.late(k)], 0) if first else 0
        self.nlate = second
        self.nvec = place([k for k in self.items if k not in self.base], max(first, second))

    def late(self, key) -> bool:
        """Computed in the last stage, over space that is read until then."""
        return (self.n == 4 and key[0] == "S") or (self.n == 5 and key[0] == "C" and len(key[1]) == 3)

    # -- vector index of an item for one helicity combination -------------
    def index(self, key, hel: dict, s: int = 0, b: int = 0) -> int:
        g, sp = self.items[key]
        i = sum(hel[x] << q for q, x in enumerate(g))
        spin = 0
        if sp == 2:
            spin = s + 2 * b
        elif sp == 1:
            spin = b if key[0] == "C" else s
        return self.base[key] + i + (spin << len(g))

    @staticmethod
    def mask(word) -> int:
        return sum(1 << i for i in word)

    def _combos(self, key):
        g, sp = self.items[key]
        for c in range(1 << (len(g) + sp)):
            hel = {x: c >> q & 1 for q, x in enumerate(g)}
            spin = c >> len(g)
            if sp == 2:
                yield hel, spin & 1, spin >> 1
            else:
                yield hel, spin, spin

    def _task_combos(self, key):
        """Combinations that have a task of their own: of the gluon currents
        the half whose last gluon has helicity bit 0."""
        for hel, s, b in self._combos(key):
            if key[0] != "J" or not hel[self.items[key][0][-1]]:
                yield hel, s, b

    # -- task tables -------------------------------------------------------
    def table(self, stage, keys):
        """Rows of 16-bit numbers, one per task (item x helicity combination)."""
        rows = []
        for key in keys:
            for hel, s, b in self._task_combos(key):
                flip = {g: 1 - x for g, x in hel.items()}
                ix = lambda k: self.index(k, hel, s, b)  # noqa: E731
                dst = ix(key)
                if stage[0] == "J":
                    w = key[1]
                    m = len(w)
                    row = [ix(self.jkey(w[i:j])) for i in range(m) for j in range(i + 1, m + 1) if j - i < m]
                    for i in range(1, m):
                        row += [self.mask(w[:i]), self.mask(w[i:])]
                    row += [dst, self.index(key, flip)]
                    if m == 2:
                        row += [self.index(self.jkey(w[::-1]), x) for x in (hel, flip)]
                elif stage[0] == "K":
                    sg, ws = kk(key[1])
                    row = [ix(self.jkey(w)) for w in ws]
                    row += [row[0]] * (3 - len(row)) + [dst, len(ws), 1 if sg < 0 else 0]
                    row += [self.index(key, flip), len(key[1]) % 2]
                elif stage[0] in "RAC":
                    w = key[1]
                    m = len(w)
                    row = []
                    for i in range(m):
                        if stage[0] == "C":
                            row += [ix(("C", w[m - i:])), ix(self.jkey(w[:m - i]))]
                        else:
                            row += [ix(("R", w[:i])), ix(self.jkey(w[i:]))]
                    row.append(dst)
                    if stage[0] == "R":
                        row += [0, self.mask(w), self.mask(w)]
                    elif stage[0] == "C":
                        row += [1, self.mask(w), self.full ^ self.mask(w)]
                elif stage[0] == "S":
                    row = [ix(("R", key[1])), ix(self.jkey(key[2])), dst]
                else:
                    row = [ix(("R", key[1])), ix(("C", key[2])), dst]
                rows.append(row)
        return rows

    # -- stages -------------------------------------------------------------
    def deps(self, key):
        kind = key[0]
        w = key[1]
        m = len(w)
        if kind == "J":
            if m == 1:
                return []
            if m == 2:
                return [self.jkey(w[:1]), self.jkey(w[1:])]
            if w[0] == min(w):
                return [self.jkey(w[i:j]) for i in range(m) for j in range(i + 1, m + 1) if j - i < m]
            return [self.jkey(x) for x in kk(w)[1]]
        if kind == "S":
            return [("R", w), self.jkey(key[2])]
        if kind == "V":
            return [("R", w), ("C", key[2])]
        if kind == "C":
            return [k for i in range(m) for k in (("C", w[m - i:]), self.jkey(w[:m - i]))]
        return [k for i in range(m) for k in (("R", w[:i]), self.jkey(w[i:]))]

    def level(self, key) -> int:
        """Stage of an item.  The currents of one length are one list (their
        code is the longest, so it is there and fetched once), the Kleiss-Kuijf
        sums of one length another."""
        if key not in self._lev:
            w = key[1]
            group = [key]
            if key[0] == "J" and len(w) > 2:
                group = self.tasks[("J" if w[0] == min(w) else "K") + str(len(w))]
            self._lev[key] = 1 + max([self.level(d) for k in group for d in self.deps(k)], default=-1)
        return self._lev[key]

    def routine(self, key) -> str:
        """The task call of an item ({row}: its table line)."""
        kind, m = key[0], len(key[1])
        if kind == "J":
            return f"j_task<{m}, R>(st, {{row}}, kr)" if m < 3 or key[1][0] == min(key[1]) else "comb_task<R>(st, {row})"
        if kind in "RC":
            return f"line_task<{m}, R>(st, {{row}}, kr)"
        if kind == "A":
            return f"amp_task<{m}, R>(st, {{row}})"
        if kind == "S":
            return "amp_task<1, R>(st, {row})"
        return "vec_task<R>(st, {row})"

    def stages(self):
        """[(level, routine, row width, rows)]: task lists in dependency order;
        lists of one level are independent of each other."""
        lists: dict = {}
        for stage, keys in self.tasks.items():
            for key in keys:
                lev = 99 if self.late(key) else self.level(key)
                fn = "rec::" + self.routine(key)
                lists.setdefault((lev, fn), []).extend(self.table(stage, [key]))
        return sorted([(lev, fn, rows) for (lev, fn), rows in lists.items()], key=lambda x: x[0])


# ---------------------------------------------------------------------------
# emission
# ---------------------------------------------------------------------------

def colour_blocks(n: int, K):
    """The colour form block by block: C(pi s, pi t) = C(s, t) for a common
    relabelling pi of the gluons, so the characters of a group of commuting
    relabellings, here H = {1, (01)} x {1, (23)} (n >= 4), split the flows into
    |H| blocks that the form does not mix:
      J^T K J = (1/|H|) sum_chi sum_r,r' F_chi(r) M_chi(r, r') F_chi(r'),
      F_chi(r) = sum_h chi(h) J(h r),  M_chi(r, r') = sum_h chi(h) K(r, h r'),
    r over the orbits of H.  Returns (orbits [[flow index of h r]], characters, M)."""
    ws = words(n)
    ix = {w: i for i, w in enumerate(ws)}
    swaps = [(0, 1), (2, 3)]

    def act(bits, w):
        rel = list(range(n))
        for q, (a, b) in enumerate(swaps):
            if bits >> q & 1:
                rel[a], rel[b] = rel[b], rel[a]
        return tuple(rel[x] for x in w)
    seen, orbits = set(), []
    for w in ws:
        if w in seen:
            continue
        orb = [act(h, w) for h in range(4)]
        seen.update(orb)
        assert len(set(orb)) == 4
        orbits.append([ix[x] for x in orb])
    M = []
    for chi in range(4):
        sg = [(-1) ** bin(chi & h).count("1") for h in range(4)]
        M.append([[sum(sg[h] * K[r[0]][t[h]] for h in range(4)) for t in orbits] for r in orbits])
    return orbits, M


class _Emit:
    def __init__(self, rec: Recursion):
        self.rec = rec
        self.masks: set = set()

    def addr(self, key, ib=True):
        """Vector index of an item for the thread's helicities (code)."""
        rec = self.rec
        g, sp = rec.items[key]
        a = f"{rec.base[key]} + {self.offset(g)}" if g else f"{rec.base[key]}"
        if sp == 2:
            a += f" + ((s + 2 * (b0 + ib)) << {len(g)})"
        elif sp == 1:
            a += f" + (({'b0 + ib' if key[0] == 'C' else 's'}) << {len(g)})"
        return a

    def offset(self, g) -> str:
        """Packed helicity bits of the gluons g (increasing, or all but the last)."""
        if list(g) == sorted(g):
            self.masks.add(self.rec.mask(g))
            return f"o{self.rec.mask(g)}"
        self.masks.update((self.rec.mask(g[:-1]), self.rec.mask(g[-1:])))
        return f"o{self.rec.mask(g[:-1])} + (o{self.rec.mask(g[-1:])} << {len(g) - 1})"

    def offsets(self):
        n = self.rec.n
        return [f"  const int o{m} = hel_bits<{m}, {n}>(hg);" for m in sorted(self.masks) if m]

    def spread(self, out, xs, pre, blk, suf, flows, tag):
        """Add the closed basis values xs[word] (arrays over ib) to the flows
        of every order of the block."""
        sums: dict = {}
        for w in itertools.permutations(blk):
            k = flows.get(pre + w + suf)
            if k is None:
                continue
            if len(w) == 2:
                sg, terms = (1, (w,)) if w in xs else (-1, (w[::-1],))
            else:
                sg, t = kk(w)
                terms = tuple(sorted(t))
            if len(terms) == 1:
                nm = xs[terms[0]]
            else:
                if terms not in sums:
                    nm = f"{tag}_{len(sums)}"
                    sums[terms] = nm
                    out.append(f"    cx<R> {nm}[NB];")
                    out.append("    for (int ib = 0; ib < NB; ib++) "
                               f"{nm}[ib] = " + " + ".join(f"{xs[t]}[ib]" for t in terms) + ";")
                nm = sums[terms]
            op = "+" if sg > 0 else "-"
            out.append(f"    for (int ib = 0; ib < NB; ib++) a[ib][{k}] = a[ib][{k}] {op} {nm}[ib];")

    def contraction(self, flows: dict, skip=lambda lp, ls: False):
        """Code that adds every term of the given flows (word -> accumulator index) to a[ib][.]."""
        return self.open_terms(flows) + self.block_terms(flows, skip)

    def open_terms(self, flows: dict):
        rec = self.rec
        p = rec.p
        out: list[str] = []
        # no block across the cut
        heads: dict = {}
        for w in flows:
            heads.setdefault(w[:p], []).append(w)
        for h, ws in heads.items():
            out.append(f"  {{ const V4<R> r = st.ld({self.addr(('A', h))});")
            for w in ws:
                out.append("    for (int ib = 0; ib < NB; ib++) "
                           f"close_rc(a[ib][{flows[w]}], r, st.ld({self.addr(('C', w[p:]))}));")
            out.append("  }")
        return out

    def block_terms(self, flows: dict, skip=lambda lp, ls: False):
        rec = self.rec
        n, p = rec.n, rec.p
        out: list[str] = []
        done = set()
        cols: dict = {}
        for w in flows:
            for lp in range(p):
                for ls in range(n - p):
                    if n - lp - ls < 2 or skip(lp, ls):
                        continue
                    pre, blk, suf = w[:lp], tuple(sorted(w[lp:n - ls])), w[n - ls:]
                    if (pre, blk, suf) in done:
                        continue
                    done.add((pre, blk, suf))
                    kind = rec.closing(lp, ls, len(blk))
                    group = (kind, suf) if kind == "S" else (kind, blk)
                    cols.setdefault(group, []).append((pre, blk, suf))
        q = 0
        for (kind, shared), terms in cols.items():
            if kind == "S":
                out.append(f"  {{ V4<R> c[NB]; for (int ib = 0; ib < NB; ib++) c[ib] = st.ld({self.addr(('C', shared))});")
                for pre, blk, suf in terms:
                    xs = {}
                    for b in basis(blk):
                        nm = f"x{q}"
                        q += 1
                        xs[b] = nm
                        out.append(f"    cx<R> {nm}[NB]; {{ const V4<R> r = st.ld({self.addr(('S', pre, b))});")
                        out.append("      for (int ib = 0; ib < NB; ib++) { "
                                   f"{nm}[ib] = {{R(0), R(0)}}; close_rc({nm}[ib], r, c[ib]); }} }}")
                    self.spread(out, xs, pre, blk, suf, flows, f"y{q}")
                out.append("  }")
            else:
                vs = []
                out.append("  {")
                for pre, blk, suf in terms:
                    nm = f"v{q}"
                    q += 1
                    vs.append(nm)
                    out.append(f"    V4<R> {nm}[NB]; for (int ib = 0; ib < NB; ib++) {nm}[ib] = "
                               f"st.ld({self.addr(('V', pre, suf))});")
                xs = [dict() for _ in terms]
                for b in basis(shared):
                    out.append(f"    cx<R> {', '.join(f'x{q}_{t}[NB]' for t in range(len(terms)))};")
                    out.append(f"    {{ const V4<R> j = st.ld({self.addr(rec.jkey(b))});")
                    for t, nm in enumerate(vs):
                        xs[t][b] = f"x{q}_{t}"
                        out.append(f"      for (int ib = 0; ib < NB; ib++) x{q}_{t}[ib] = vdot({nm}[ib], j);")
                    out.append("    }")
                    q += 1
                for t, (pre, blk, suf) in enumerate(terms):
                    self.spread(out, xs[t], pre, blk, suf, flows, f"y{q}_{t}")
                out.append("  }")
        return out


class _EmitLast(_Emit):
    """The closing of the flows that end on gluon e, for a variable e: written
    for e = 4 with the others renamed 0..3 in increasing order, which keeps
    every canonical order; positions affine in e, the others from a table."""

    def __init__(self, rec: Recursion):
        super().__init__(rec)
        self.rows: list = []  # table columns: positions for e = 0..4

    def renamed(self, key, e):
        ab = {**{i: i if i < e else i + 1 for i in range(4)}, 4: e}
        return tuple(tuple(ab[g] for g in x) if isinstance(x, tuple) else x for x in key)

    def offset(self, g) -> str:
        rest = [x for x in g if x != 4]
        parts = []
        if rest:
            self.masks.add(self.rec.mask(rest))
            parts.append(f"o{self.rec.mask(rest)}")
        if 4 in g:
            assert g[-1] == 4
            parts.append(f"(he << {len(rest)})" if rest else "he")
        return " + ".join(parts)

    def addr(self, key, ib=True):
        rec = self.rec
        g, sp = rec.items[key]
        pos = [rec.base[self.renamed(key, e)] for e in range(5)]
        step = pos[1] - pos[0]
        if all(pos[e] == pos[0] + e * step for e in range(5)):
            a = f"{pos[0]} + {step} * e"
        else:
            if pos not in self.rows:
                self.rows.append(pos)
            a = f"tb[{self.rows.index(pos)}]"
        if g:
            a += f" + {self.offset(g)}"
        if sp == 2:
            a += f" + ((s + 2 * (b0 + ib)) << {len(g)})"
        elif sp == 1:
            a += f" + (({'b0 + ib' if key[0] == 'C' else 's'}) << {len(g)})"
        return a


def flow_order(n: int) -> list[tuple]:
    """Order of the flows in the emitted code: lexicographic, but for five
    gluons grouped by the last gluon."""
    return sorted(words(n), key=lambda w: (w[-1:] + w) if n > 4 else w)


def _thread_sum(rec: Recursion) -> list[str]:
    """Two gluons: every helicity of an event by one thread, straight line in
    registers, the antitop spins one after the other (the columns and closing
    vectors of one spin at a time)."""
    L = ["  // sum over the helicities whose bit of `good` is set, one thread per event",
         "  template <typename R, typename D, typename A>",
         "  __device__ static __forceinline__ A thread_sum(const double* p, const double* kp, const unsigned good) {",
         "    using namespace rec;",
         f"    const RegStore<R, {rec.n}, {rec.nvec}> st{{}};",
         "    const R kr[2] = {R(kp[0]), R(kp[1])};",
         "    setup_thread<" + "P_SELF" + ", R, D>(st, p, kp, kr);", "    A acc = A(0);"]
    calls: dict = {None: [], 0: [], 1: []}
    for stage, keys in rec.tasks.items():
        for key in keys:
            rows = rec.table(stage, [key])
            for row, (hel, s, b) in zip(rows, rec._task_combos(key), strict=True):
                w = ((len(row) + 7) // 8) * 8
                lit = f"Row<{w}>{{{{" + ", ".join(str(x) for x in row + [0] * (w - len(row))) + "}}"
                when = b if key[0] in "CV" else None
                calls[when].append((rec.level(key), rec.routine(key).format(row=lit)))
    L += ["    " + c + ";" for _, c in sorted(calls[None], key=lambda x: x[0])]
    for b in range(2):
        L += ["    " + c + ";" for _, c in sorted(calls[b], key=lambda x: x[0])]
        for s in range(2):
            for hg in range(1 << rec.n):
                L.append(f"    {{ cx<R> a[1][2]; flows_open<R, 1>(st, {hg}, {s}, {b}, a); flows_block<R, 1>(st, {hg}, {s}, {b}, a);")
                L.append("      const R v = colour_form<R>(a[0]);")
                L.append(f"      if (good >> helicity({hg}, {s}, {b}) & 1u) acc += (A)v; }}")
    L += ["    return acc;", "  }"]
    return L


def _grouped_flows(rec: Recursion, head, tag, late) -> list[str]:
    """Five gluons: 120 flows do not fit in registers, so they are closed in
    five groups by their last gluon e, all by the same code (a loop over e; the
    straight-line code of all groups does not stay in the instruction cache).
    The closings of one gluon + a block of four, and of the block of all five,
    serve several groups: they come first and start the flows."""
    n = rec.n
    fo = flow_order(n)
    L = []
    L.append("  // columns of three gluons, over the store space that closings() read")
    L.append("  template <typename R, class ST>")
    L.append("  __device__ static __forceinline__ void late(const ST& all, const R* kr, const int tid, const int nt,")
    L.append("                                              const int per = 1) {")
    L += late
    L.append("  }")
    em = _Emit(rec)
    xname, code = {}, []
    for pre in [()] + [(a,) for a in range(n)]:
        blk = [g for g in range(n) if g not in pre]
        code.append(f"  {{ V4<R> v[NB]; for (int ib = 0; ib < NB; ib++) v[ib] = st.ld({em.addr(('V', pre, ()))});")
        for b in basis(blk):
            xname[(pre, b)] = len(xname)
            code.append(f"    {{ const V4<R> j = st.ld({em.addr(rec.jkey(b))}); for (int ib = 0; ib < NB; ib++) "
                        f"x[ib][{xname[(pre, b)]}] = vdot(v[ib], j); }}")
        code.append("  }")
    for k, w in enumerate(fo):
        val = ""
        for lp in (0, 1):
            sg, t = kk(w[lp:])
            e = " + ".join(f"x[ib][{xname[(w[:lp], q)]}]" for q in sorted(t))
            val += (" - " if sg < 0 else " + " if lp else "") + f"({e})"
        code.append(f"  for (int ib = 0; ib < NB; ib++) put(ib, {k}, {val.strip()});")
    L.append("  // put(ib, k, value) stores the first part of flow k of antitop spin b0 + ib")
    L.append("  template <typename R, int NB, class ST, class PUT>")
    L.append("  __device__ static __forceinline__ void closings(const ST& st, const int hg, const int s, const int b0,")
    L.append("                                                  const PUT& put) {")
    L.append("    using namespace rec;")
    L.append(f"    cx<R> x[NB][{len(xname)}];")
    L += ["  " + q for q in em.offsets() + code]
    L.append("  }")
    em = _EmitLast(rec)
    mine = [w for w in fo if w[-1] == 4]
    flows = {w: i for i, w in enumerate(mine)}
    body = em.contraction(flows, skip=lambda lp, ls: ls == 0)
    head.insert(head.index(f"struct {tag}_rec {{"), f"MG_REC_CONST unsigned short {tag}_RECE[5][{len(em.rows)}] = {{"
                + ", ".join("{" + ", ".join(str(r[e]) for r in em.rows) + "}" for e in range(5)) + "};")
    L.append("  // get(ib, k) returns the first part of flow k, put(ib, k, value) stores the flow")
    L.append("  template <typename R, int NB, class ST, class GET, class PUT>")
    L.append("  __device__ static __forceinline__ void all_flows(const ST& st, const int hg, const int s, const int b0,")
    L.append("                                                   const GET& get, const PUT& put) {")
    L.append("    using namespace rec;")
    L.append("#pragma unroll 1")
    L.append("    for (int e = 0; e < 5; e++) {")
    L.append("      const int hr = ((hg >> (e + 1)) << e) | (hg & ((1 << e) - 1)), he = hg >> e & 1;")
    L.append(f"      const unsigned short* tb = {tag}_RECE[e];")
    L += [f"      const int o{m} = hel_bits<{m}, 4>(hr);" for m in sorted(em.masks) if m]
    L.append(f"      cx<R> a[NB][{len(mine)}];")
    L.append(f"      for (int ib = 0; ib < NB; ib++) for (int k = 0; k < {len(mine)}; k++) a[ib][k] = get(ib, {len(mine)} * e + k);")
    L += ["    " + q for q in body]
    L.append(f"      for (int ib = 0; ib < NB; ib++) for (int k = 0; k < {len(mine)}; k++) put(ib, {len(mine)} * e + k, a[ib][k]);")
    L.append("    }")
    L.append("  }")
    return L


def _colour_form_looped(head, tag, n, K, ws) -> list[str]:
    """The colour form of 120 flows: one block after the other (the same code
    over four tables of block numerators), the flows anywhere in memory."""
    ws = flow_order(n)
    orbits, M = colour_blocks(n, K)
    pos = {w: i for i, w in enumerate(ws)}
    orbits = [[pos[w] for w in (words(n)[k] for k in o)] for o in orbits]
    no = len(orbits)
    tri = [M[chi][i][j] * (1 if i == j else 2) for chi in range(4) for i in range(no) for j in range(i, no)]
    head.insert(head.index(f"struct {tag}_rec {{"),
                f"MG_REC_TABLE double {tag}_RECM[{len(tri)}] = {{" + ", ".join(str(x) for x in tri) + "};")
    L = [f"  // the flows' components in the four blocks of {no}, in their place", f"  static constexpr int NBLOCK = {no};",
         "  template <typename R>",
         f"  __device__ static __forceinline__ void colour_blocks(cx<R> (&a)[{len(ws)}]) {{"]
    for o in orbits:
        L.append(f"    {{ const cx<R> p0 = a[{o[0]}] + a[{o[1]}], m0 = a[{o[0]}] - a[{o[1]}], "
                 f"p1 = a[{o[2]}] + a[{o[3]}], m1 = a[{o[2]}] - a[{o[3]}];")
        L.append(f"      a[{o[0]}] = p0 + p1; a[{o[1]}] = m0 + m1; a[{o[2]}] = p0 - p1; a[{o[3]}] = m0 - m1; }}")
    L.append("  }")
    L += ["  // those of block CHI", "  template <int CHI, typename R>",
          f"  __device__ static __forceinline__ void colour_block(const cx<R> (&a)[{len(ws)}], cx<R> (&f)[{no}]) {{"]
    for chi in range(4):
        L.append(f"    if constexpr (CHI == {chi}) {{ "
                 + " ".join(f"f[{r}] = a[{o[chi]}];" for r, o in enumerate(orbits)) + " }")
    L.append("  }")
    L += ["  // sum_ij KNUM_ij (Re J_i Re J_j + Im J_i Im J_j); |M|^2 colour sum = result / CDEN.",
          "  // a[k]: flow k; overwritten by its block components.  The sum of four blocks' values:",
          "  template <typename R>",
          f"  __device__ static __forceinline__ R block_value(int chi, const cx<R> (&f)[{no}]) {{",
          f"    return R(0.25) * block_form<R>({tag}_RECM + {no * (no + 1) // 2} * chi, f);", "  }",
          "  template <typename R>",
          f"  __device__ static __forceinline__ R colour_form(cx<R> (&a)[{len(ws)}]) {{",
          "    colour_blocks<R>(a);", "    R acc = R(0);", f"    cx<R> f[{no}];"]
    L += [f"    colour_block<{chi}, R>(a, f); acc = acc + block_value<R>({chi}, f);" for chi in range(4)]
    L += ["    return acc;", "  }"]
    B = ["  // one block: numerators M_ii and 2 M_ij (j > i) row by row",
         "  template <typename R>",
         f"  __device__ static __noinline__ R block_form(const double* __restrict__ m, const cx<R> (&f)[{no}]) {{",
         "    R acc = R(0);", "    int q = 0;", "    MG_REC_UNROLL", f"    for (int i = 0; i < {no}; i++) {{",
         "      R yr = R(0), yi = R(0);", "    MG_REC_UNROLL", f"      for (int j = i; j < {no}; j++) {{",
         "        const R k = R(__ldg(m + q++));",
         "        yr = rec::fmad(k, f[j].re, yr);", "        yi = rec::fmad(k, f[j].im, yi);", "      }",
         "      acc = rec::fmad(f[i].re, yr, acc);", "      acc = rec::fmad(f[i].im, yi, acc);", "    }",
         "    return acc;", "  }"]
    lex = words(n)
    vals = [K[i][j] * (1 if i == j else 2) if j >= i else 0 for i in range(len(ws)) for j in range(len(ws))]
    head.insert(head.index(f"struct {tag}_rec {{"),
                f"MG_REC_TABLE short {tag}_RECK[{len(vals)}] = {{" + ", ".join(str(x) for x in vals) + "};")
    Q = ["  // the same in FP32 (diagrams in FP64): rows i, numerators K_ii and 2 K_ij (j > i)",
         f"  __device__ static __noinline__ float colour_form_paper(const cx<double> (&a)[{len(ws)}]) {{",
         f"    float fr[{len(ws)}], fi[{len(ws)}];",
         f"    for (int k = 0; k < {len(ws)}; k++) {{ fr[lex_flow(k)] = (float)a[k].re; fi[lex_flow(k)] = (float)a[k].im; }}",
         "    float q = 0.f;",
         f"    for (int i = 0; i < {len(ws)}; i++) {{",
         "      float yr = 0.f, yi = 0.f;",
         f"      for (int j = i; j < {len(ws)}; j++) {{",
         f"        const float k = (float)__ldg({tag}_RECK + i * {len(ws)} + j);",
         "        yr = rec::fmad(k, fr[j], yr); yi = rec::fmad(k, fi[j], yi);", "      }",
         "      q = rec::fmad(fr[i], yr, q); q = rec::fmad(fi[i], yi, q);", "    }",
         "    return q;", "  }"]
    head.insert(head.index(f"struct {tag}_rec {{"), f"MG_REC_TABLE unsigned char {tag}_RECL[{len(ws)}] = {{"
                + ", ".join(str(lex.index(w)) for w in ws) + "};")
    O = ["  // flow index (lexicographic order of the gluons) of the emitted code's flow k",
         f"  __device__ static __forceinline__ int lex_flow(int k) {{ return __ldg({tag}_RECL + k); }}",
         f"  static constexpr int KNUM_ORDERED[{len(ws) ** 2}] = {{"
         + ", ".join(str(K[lex.index(a)][lex.index(b)]) for a in ws for b in ws) + "};  // in the emitted order"]
    return O + B + L + Q


def emit_recursion(n: int, tag: str) -> str:
    """Header of the recursion of one process: store sizes, stage tables, the
    stage driver, the closing contraction of one helicity and the colour form."""
    rec = Recursion(n)
    ws = words(n)
    cden, K = common_denominator(colour_matrix_exact(n))
    iden = 256
    for i in range(2, n - 1):
        iden *= i
    T, body, late = [], [], []
    # five gluons: a task's table line is fetched one task ahead, a list's first
    # one before the barrier of its stage (60 KB of lines come from L2: the store
    # leaves little L1; 8229 mixed events, flow kernel 1.49 -> 1.44 ms; the
    # smaller tables stay in L1, where it cost FP64 2 %).  A list runs over the
    # tasks of all events of the CTA, so that its last, partly filled round is
    # one of the CTA and not one of every warp.
    levels: dict = {}
    for q, (lev, fn, rows) in enumerate(rec.stages()):
        w = ((len(rows[0]) + 7) // 8) * 8
        flat = [x for r in rows for x in r + [0] * (w - len(r))]
        assert all(0 <= x < 65536 for x in flat)
        name = f"{tag}_REC{q}"
        T.append(f"MG_REC_TABLE rec::Row<{w}> {name}[{len(rows)}] = {{"
                 + ", ".join("{{" + ", ".join(str(x) for x in flat[i:i + w]) + "}}" for i in range(0, len(flat), w))
                 + "};")
        if n < 5:
            levels.setdefault(lev, []).append((None, [
                f"    MG_REC_LOOP for (int t = tid; t < {len(rows)} * per; t += nt) {{",
                f"      const ST st = all.at(t / {len(rows)});",
                f"      {fn.format(row=f'{name}[t % {len(rows)}]')};", "    }"]))
            continue
        levels.setdefault(lev, []).append((
            f"    rec::Row<{w}> r{q} = {name}[tid % {len(rows)}];",
            [f"    MG_REC_LOOP for (int t = tid; t < {len(rows)} * per; t += nt) {{",
             f"      const rec::Row<{w}> row = r{q};", f"      const ST st = all.at(t / {len(rows)});",
             f"      r{q} = {name}[(t + nt) % {len(rows)}];",
             f"      {fn.format(row='row')};", "    }"]))
    for lev in sorted(levels):
        out = late if lev == 99 else body
        out += [first for first, _ in levels[lev] if first]
        if lev != 99 and body and lev != min(levels):
            out.append("    sync();")
        for _, loop in levels[lev]:
            out += loop
    L = [f"// generated by paper_2303_18244_gb300.generator for 'g g > t t~{' g' * (n - 2)}':",
         "// helicity-shared colour-ordered recursion", "#pragma once", '#include "mg_recursion.cuh"', "namespace mg {"]
    L += T
    L.append(f"struct {tag}_rec {{")
    L.append(f"  static constexpr int N = {n}, NPAR = {n + 2}, NHEL = {1 << (n + 2)}, NCOL = {len(ws)};")
    L.append("  template <typename R>")
    L.append(f"  static constexpr int NVEC = {rec.nvec};")
    L.append(f"  static constexpr double IDEN = {iden}.0;")
    L.append(f"  static constexpr int CDEN = {cden}, NDIAG = {count_diagrams(n)}, NAMP = {len(build_plan(n).amps)};")
    L.append("  // colour numerators, flows in lexicographic order")
    L.append(f"  static constexpr int KNUM[{len(ws) ** 2}] = {{{', '.join(str(x) for r in K for x in r)}}};")
    L.append(f"  static constexpr int R0 = {rec.base[('R', ())]}, C0 = {rec.base[('C', ())]};")
    j1 = [rec.base[("J", (i,))] for i in range(n)]
    assert all(j1[i] == j1[0] + 2 * i for i in range(n))
    L.append(f"  __device__ static __forceinline__ int j1_base(int i) {{ return {j1[0]} + 2 * i; }}")
    L.append("  // helicity index (bit NPAR - 1 - slot of a particle set: helicity +1) of the gluon")
    L.append("  // helicity bits hg (bit i: gluon i) and the spin bits s (top) and b (antitop)")
    L.append("  __device__ static __forceinline__ int helicity(int hg, int s, int b) {")
    L.append(f"    int h = (s << {n - 1}) | (b << {n - 2});")
    L.append("#pragma unroll")
    L.append(f"    for (int i = 0; i < {n}; i++) h |= (hg >> i & 1) << ({n + 1} - (i < 2 ? i : i + 2));")
    L.append("    return h;")
    L.append("  }")
    L.append("  // the currents of `per` events (all: the store of the first), by nt threads")
    L.append("  template <typename R, class ST, class SYNC>")
    L.append("  __device__ static __forceinline__ void currents(const ST& all, const R* kr, const int tid, const int nt,")
    L.append("                                                  const SYNC& sync, const int per = 1) {")
    L += body
    L.append("  }")
    if n <= 4:
        L.append(f"  static constexpr bool LATE = {'true' if late else 'false'};")
        L.append("  template <typename R, class ST>")
        L.append("  __device__ static __forceinline__ void late([[maybe_unused]] const ST& all, [[maybe_unused]] const int tid,")
        L.append("                                              [[maybe_unused]] const int nt,")
        L.append("                                              [[maybe_unused]] const int per = 1) {")
        L += late
        L.append("  }")
        flows = {w: i for i, w in enumerate(ws)}
        L.append("  // the colour-ordered amplitudes of NB helicities (gluon bits hg, top spin s, antitop spins")
        L.append("  // b0 ..): the terms without a block across the cut, then (after late()) those with one")
        for name, get in (("flows_open", lambda e: e.open_terms(flows)), ("flows_block", lambda e: e.block_terms(flows))):
            em = _Emit(rec)
            code = get(em)
            L.append("  template <typename R, int NB, class ST>")
            L.append(f"  __device__ static __forceinline__ void {name}(const ST& st, const int hg, const int s, const int b0,")
            L.append(f"                                                 cx<R> (&a)[NB][{len(ws)}]) {{")
            L.append("    using namespace rec;")
            L += ["  " + x for x in em.offsets()]
            if name == "flows_open":
                L.append("    for (int ib = 0; ib < NB; ib++)")
                L.append(f"      for (int k = 0; k < {len(ws)}; k++) a[ib][k] = {{R(0), R(0)}};")
            L += ["  " + x for x in code]
            L.append("  }")
    else:
        L += _grouped_flows(rec, L, tag, late)
    # colour form
    if n == 2:
        L += [x.replace("P_SELF", f"{tag}_rec") for x in _thread_sum(rec)]
    if n > 4:
        L += _colour_form_looped(L, tag, n, K, ws)
        L += ["};", "}  // namespace mg"]
        return _unrolled(L)
    L.append("  // sum_ij KNUM_ij (Re J_i Re J_j + Im J_i Im J_j); |M|^2 colour sum = result / CDEN")
    L.append("  template <typename R>")
    L.append(f"  __device__ static __forceinline__ R colour_form(const cx<R> (&a)[{len(ws)}]) {{")
    if n == 4:
        orbits, M = colour_blocks(n, K)
        L.append("    R acc = R(0);")
        no = len(orbits)
        L.append(f"    cx<R> f[4][{no}];")
        for r, o in enumerate(orbits):
            L.append(f"    {{ const cx<R> p0 = a[{o[0]}] + a[{o[1]}], m0 = a[{o[0]}] - a[{o[1]}], "
                     f"p1 = a[{o[2]}] + a[{o[3]}], m1 = a[{o[2]}] - a[{o[3]}];")
            L.append(f"      f[0][{r}] = p0 + p1; f[1][{r}] = m0 + m1; f[2][{r}] = p0 - p1; f[3][{r}] = m0 - m1; }}")
        for chi in range(4):
            for i in range(no):
                terms = [(M[chi][i][j] * (1 if j == i else 2), j) for j in range(i, no)]
                terms = [t for t in terms if t[0]]
                if not terms:
                    continue
                L.append(f"    {{ cx<R> y = R({terms[0][0]}) * f[{chi}][{terms[0][1]}];")
                for k, j in terms[1:]:
                    L.append(f"      y = fma(R({k}), f[{chi}][{j}], y);")
                L.append(f"      acc = rec::fmad(f[{chi}][{i}].re, y.re, acc); acc = rec::fmad(f[{chi}][{i}].im, y.im, acc); }}")
        L.append("    return R(0.25) * acc;")
    else:
        from .emit import _colour_quadratic
        L.append("#define JAMP(k) a[k]")
        L += ["  " + x.replace("fmaf_t<R>", "rec::fmad") for x in _colour_quadratic(K, len(ws))]
        L.append("#undef JAMP")
    L.append("  }")
    # the FP32 form of MG_MIXED_PAPER, in the order of sigma_paper_kernel
    L.append("  // the same in FP32 (diagrams in FP64): rows i, numerators K_ii and 2 K_ij (j > i)")
    L.append(f"  __device__ static __forceinline__ float colour_form_paper(const cx<double> (&a)[{len(ws)}]) {{")
    L.append("    float q = 0.f;")
    for i in range(len(ws)):
        L.append("    { float yr = 0.f, yi = 0.f;")
        for j in range(i, len(ws)):
            k = K[i][j] * (1 if i == j else 2)
            if k:
                L.append(f"      yr = rec::fmad({k}.f, (float)a[{j}].re, yr); yi = rec::fmad({k}.f, (float)a[{j}].im, yi);")
        L.append(f"      q = rec::fmad((float)a[{i}].re, yr, q); q = rec::fmad((float)a[{i}].im, yi, q); }}")
    L.append("    return q;")
    L.append("  }")
    L.append("};")
    L.append("}  // namespace mg")
    return _unrolled(L)


def _unrolled(L: list[str]) -> str:
    out = []
    for x in L:  # every per-antitop-spin loop is unrolled
        if "for (int ib" in x or "for (int k" in x:
            x = x.replace("for (int ib = 0; ib < NB; ib++)", "MG_REC_UNROLL for (int ib = 0; ib < NB; ib++)")
            x = x.replace("for (int k = 0", "MG_REC_UNROLL for (int k = 0")
        out.append(x)
    return "\n".join(out) + "\n"
