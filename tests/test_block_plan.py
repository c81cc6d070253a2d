"""Host-side check of the on-chip mode of one block per SM (csrc/bte_grid.cu),
no GPU needed: the kernel's partition into blocks, its split of a block into
interior and boundary cells and its edge exchange, mirrored for blocks of one
row or one column group up to several, with ragged last blocks.

Every cell is made once per half-step; interior cells read no halo; every
halo cell that a boundary cell reads and that lies in the grid is polled, from
the exchange entry that the cell's owner publishes; a block polls entries only
of blocks that poll its own (so an entry is read before it is written again);
and no index leaves its array.
"""
import pytest


def cdiv(a, b):
    return -(-a // b)


class Block:
    def __init__(self, b, N1, M1, R, W, V):
        self.GR, self.GC = cdiv(N1, R), cdiv(M1, W)
        self.bi, self.bj = divmod(b, self.GC)
        self.r0, self.c0 = self.bi * R, self.bj * W
        self.R, self.W = min(R, N1 - self.r0), min(W, M1 - self.c0)
        self.N1, self.M1, self.V, self.Wmax = N1, M1, V, W
        self.ncg = cdiv(self.W, V)
        self.nri, self.nci = max(self.R - 2, 0), max(self.ncg - 2, 0)

    def interior(self, threads):
        cpp = max(min(self.nci, threads), 1)
        split = threads // cpp
        nrow = cdiv(self.nri, split)
        if not (self.nci and self.nri):
            return
        for tid in range(threads):
            gl, part = tid % cpp, tid // cpp
            lo = 1 + part * nrow
            for g0 in range(0, self.nci, cpp):
                g = g0 + gl
                on_g = part < split and g < self.nci
                for ch in range(2):
                    for ii in range((nrow + 1 - ch) // 2):
                        i = lo + ch + 2 * ii
                        if on_g and i < self.R - 1:
                            yield i, g + 1

    def boundary(self):
        nrb, ncb = (2 if self.R >= 2 else 1), (2 if self.ncg >= 2 else 1)
        nb_rows = nrb * self.ncg
        for u in range(nb_rows + ncb * self.nri):
            if u < nb_rows:
                yield (0, u) if u < self.ncg else (self.R - 1, u - self.ncg)
            else:
                v = u - nb_rows
                il = 1 + v // ncb
                yield il, (self.ncg - 1 if v - (il - 1) * ncb else 0)

    def published(self):
        """{exchange entry: global cell}"""
        out = {}
        for il, g in self.boundary():
            m, n = g * self.V, self.r0 + il
            for q in range(self.V):
                if m + q < self.W:
                    cell = (n, self.c0 + m + q)
                    if il == 0 and self.bi > 0:
                        out["row", self.bi, 0, self.c0 + m + q] = cell
                    if il == self.R - 1 and self.bi + 1 < self.GR:
                        out["row", self.bi, 1, self.c0 + m + q] = cell
            if g == 0 and self.bj > 0:
                out["col", self.bj, 0, n] = (n, self.c0)
            if g == self.ncg - 1 and self.bj + 1 < self.GC:
                out["col", self.bj, 1, n] = (n, self.c0 + m + self.V - 1)
        return out

    def polled(self):
        """{local halo cell: exchange entry}"""
        out = {}
        for q in range(2 * (self.W + 2) + 2 * self.R):
            if q < 2 * (self.W + 2):
                bot = q >= self.W + 2
                lc = (q - (self.W + 2) if bot else q) - 1
                li = self.R if bot else -1
                if not (0 <= self.r0 + li < self.N1 and 0 <= self.c0 + lc < self.M1):
                    continue
                out[li, lc] = ("row", self.bi + 1 if bot else self.bi - 1, 0 if bot else 1, self.c0 + lc)
            else:
                q2 = q - 2 * (self.W + 2)
                rgt = q2 >= self.R
                li, lc = (q2 - self.R if rgt else q2), (self.W if rgt else -1)
                if not 0 <= self.c0 + lc < self.M1:
                    continue
                out[li, lc] = ("col", self.bj + 1 if rgt else self.bj - 1, 0 if rgt else 1, self.r0 + li)
        return out


@pytest.mark.parametrize("N1,M1,R,W,V,threads", [
    (31, 201, 8, 6, 1, 64), (31, 201, 8, 6, 2, 64), (23, 41, 1, 4, 4, 64), (9, 37, 3, 4, 4, 64),
    (10, 38, 4, 8, 4, 96), (17, 250, 6, 12, 4, 64), (2, 3, 1, 1, 1, 64), (2, 3, 2, 4, 4, 64),
    (51, 101, 51, 104, 4, 512), (40, 333, 13, 112, 2, 128)])
def test_blocks_cover_the_grid_and_their_exchange_is_complete(N1, M1, R, W, V, threads):
    GR, GC = cdiv(N1, R), cdiv(M1, W)
    blocks = [Block(b, N1, M1, R, W, V) for b in range(GR * GC)]
    owner, made, pub = {}, set(), {}
    for b in blocks:
        assert b.R >= 1 and b.W >= 1 and (b.W == W or b.c0 + b.W == M1)
        cells = list(b.interior(threads)) + list(b.boundary())
        assert len(cells) == len(set(cells)) == b.R * b.ncg
        for il, g in cells:
            assert 0 <= il < b.R and 0 <= g < b.ncg
            for e in range(b.V):
                if g * V + e < b.W:
                    made.add((b.r0 + il, b.c0 + g * V + e))
                    owner[b.r0 + il, b.c0 + g * V + e] = b
        for il, g in b.interior(threads):  # reads rows il -+ 1, columns one beyond the group
            assert 1 <= il <= b.R - 2 and g * V - 1 >= 0 and g * V + V < b.W
        p = b.published()
        assert not set(p) & set(pub)
        pub.update(p)
    assert len(made) == N1 * M1
    P, arr = W + 2 * V, (R + 2) * (W + 2 * V)
    polls = []
    for b in blocks:
        polled = b.polled()
        polls.append({id(owner[pub[e]]) for e in polled.values()})
        for (li, lc), e in polled.items():
            assert pub[e] == (b.r0 + li, b.c0 + lc)
            assert owner[pub[e]] is not b
            kind, blk, side, at = e
            assert 0 <= blk < (GR if kind == "row" else GC) and 0 <= at < (M1 if kind == "row" else N1)
            assert 0 <= (li + 1) * P + V + lc < arr
        for il, g in b.boundary():
            for di in (-1, 1):
                for col in range(g * V - 1, g * V + V + 1):
                    n, m = b.r0 + il + di, b.c0 + col
                    if 0 <= n < N1 and 0 <= m < M1:
                        own = 0 <= il + di < b.R and 0 <= col < b.W
                        # of a ragged group only the columns up to M + 1 are read in earnest
                        if not own and col <= b.W:
                            assert (il + di, col) in polled
                    assert 0 <= (il + di + 1) * P + V + col < arr
    for k, b in enumerate(blocks):
        for j, c in enumerate(blocks):
            assert (id(c) in polls[k]) == (id(b) in polls[j])
