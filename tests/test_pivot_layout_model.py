"""Models of index arithmetic, checked on the CPU: the pivot's tiles and mailboxes (PivotDim, FusedLayout in
csrc/pivot.cu) and the stacking of digit planes in the tensor-memory kernels (csrc/tc_digits.cu)."""
import pytest

T = 8  # digits


def dims(KM):
    LPP = 4
    return dict(LPP=LPP, R=KM // LPP, P2=KM // 2, NT=4 * KM, LDT=KM + 4, LDW=KM + 4, TX=KM // 4, RU=KM // 16)


@pytest.mark.parametrize("KM", [32, 64])
def test_cholesky_tiles_and_published_column(KM):
    d = dims(KM)
    TX, RU = d["TX"], d["RU"]
    at = sorted((RU * (t // TX) + u, 4 * (t % TX) + j) for t in range(d["NT"]) for u in range(RU) for j in range(4))
    assert at == [(i, j) for i in range(KM) for j in range(KM)]  # every entry in one thread
    for p in range(KM):  # the threads of column p write row i of colh, entry p & 3 of their four columns
        own = [t for t in range(d["NT"]) if t % TX == p >> 2]
        assert sorted(RU * (t // TX) + u for t in own for u in range(RU)) == list(range(KM))
        assert all(4 * (t % TX) + (p & 3) == p for t in own)
    assert (d["LDT"] * 4) % 16 == 0 and (RU * 4) % 8 == 0


@pytest.mark.parametrize("KM", [32, 64])
def test_mailboxes(KM):
    d = dims(KM)
    LPP, R, P2 = d["LPP"], d["R"], d["P2"]
    box = lambda q, sl, l: (q * P2 + sl) * LPP + l  # noqa: E731  16-byte chunk q of lane l in the box of slot sl
    chunks = [box(q, sl, l) for q in range(R // 4) for sl in range(P2) for l in range(LPP)]
    assert sorted(chunks) == list(range(KM * P2 // 4))  # fills the box of a column per slot, no overlap
    for q in range(R // 4):  # a quarter warp reads 128 consecutive bytes of its own slots
        for w in range(2 * KM // 32):
            for quarter in range(4):
                lanes = [32 * w + 8 * quarter + x for x in range(8)]
                a = [box(q, t // LPP, t % LPP) for t in lanes]
                assert a == list(range(a[0], a[0] + 8))
    # rows l R + u of the two halves of the threads: every row of a column once
    assert sorted(l * R + u for l in range(LPP) for u in range(R)) == list(range(KM))


@pytest.mark.parametrize("KM,MF", [(32, 96), (64, 192)])
def test_fused_step_maps(KM, MF):
    d = dims(KM)
    LDX = LDB = KM + 4
    NT, CT = d["NT"], KM // 4
    work = max(KM * d["LDT"], 4 * KM * d["P2"], KM * LDB + 64 * LDX)
    assert KM * LDB + 64 * LDX <= work and (KM * LDB * 4) % 16 == 0 and (LDX * 4) % 16 == 0
    assert NT // CT == 16
    RPT = KM // 16
    gram = sorted((RPT * (t // CT) + u, 4 * (t % CT) + v) for t in range(NT) for u in range(RPT) for v in range(4))
    assert gram == [(i, j) for i in range(KM) for j in range(KM)]
    upd = sorted((4 * (t // CT) + u, 4 * (t % CT) + v) for t in range(NT) for u in range(4) for v in range(4))
    assert upd == [(r, j) for r in range(64) for j in range(KM)]
    # the chunk of V: element e is row e % 64 of column e / 64
    assert sorted((e % 64, e // 64) for u in range(KM * 64 // NT) for e in range(u * NT, u * NT + NT)) == \
        [(r, c) for r in range(64) for c in range(KM)]
    for m in range(16, MF + 1, 16):  # rows of X_P: lanes and six chunks cover the m rows, the update only them
        rows = [rr + lane + 32 * u for rr in range(0, m, 192) for u in range(6) for lane in range(32)]
        assert [r for r in sorted(rows) if r < m] == list(range(m))
        done = [r0 + 4 * ty + u for r0 in range(0, m, 64) for ty in range(16) if 4 * ty < min(64, m - r0) for u in range(4)]
        assert done == list(range(m))


def test_update_planes():
    """k_update_oz_tc: X_t against planes u .. u + nb - 1 of V~, into blocks t + u ..: levels 0..7 hold every
    product once, and the first MMAs on a block (t = 0) overwrite it; level 8 then goes to block 0."""
    blocks, first = {}, {}
    for t in range(T):
        for u in range(0, T - t, 4):
            nb = min(4, T - t - u)
            assert 64 * nb <= 256 and t + u + nb <= 8
            for j in range(nb):
                first.setdefault(t + u + j, t)
                blocks.setdefault(t + u + j, []).append((t, u + j))
    assert set(first.values()) == {0}
    for L in range(T):
        assert sorted(blocks[L]) == [(t, L - t) for t in range(L + 1)]
    assert sorted((t, 8 - t) for t in range(1, T)) == [(t, 8 - t) for t in range(1, T)] and max(8 - t for t in range(1, T)) < T


def test_gram_planes_and_halves():
    """k_gram_oz_tc: an M = 128 operand of planes a, a + 1 (a even) against planes v .. v + nb - 1.  Lanes 0..63 of
    block B hold level B, lanes 64..127 level B + 1; together every (t, u), t + u <= 7, once."""
    low, high, first, mmas = {}, {}, {}, 0
    for a in range(0, T, 2):
        for v in range(0, T - a, 4):
            nb = min(4, T - a - v)
            mmas += 1
            for j in range(nb):
                B = a + v + j
                assert B < 8
                first.setdefault(B, a)
                low.setdefault(B, []).append((a, v + j))
                high.setdefault(B, []).append((a + 1, v + j))
    assert mmas == 6 and set(first.values()) == {0}
    for L in range(T):
        got = low[L] + (high[L - 1] if L else [])
        assert sorted(got) == [(t, L - t) for t in range(L + 1)]
    # epilogue: warp w reads lanes 32 (w & 3) .. and finishes 8 of the 16 columns of its strip, the other
    # half the rest; what it passes on is what the other finishes
    fin = {}
    for w in range(16):
        upper, c0 = (w & 3) < 2, 16 * (w >> 2)
        cf, cs = c0 + (0 if upper else 8), c0 + (8 if upper else 0)
        for lane in range(32):
            i = (32 * (w & 3) + lane) & 63
            for j in range(8):
                assert (i, cf + j) not in fin
                fin[(i, cf + j)] = (upper, cs)
    assert sorted(fin) == [(i, c) for i in range(64) for c in range(64)]
    for (i, c), (upper, _) in fin.items():  # the partner of the same row passes this column
        assert upper == (c % 16 < 8)
