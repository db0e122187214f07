"""Host-side model of the index arithmetic of the one-thread-per-element stage
(csrc/dg_stage_ept.cuh): for every tile of whole meshes and latitude bands, the
16-byte blocks read and written lie inside the state array padded to 16 bytes,
the shared-memory regions neither overlap nor overflow, every value of the tile
and of its halo ring lands where its thread reads it, and the whole and partial
output blocks of all tiles together write every own value exactly once."""
import numpy as np
import pytest

GEOMETRY = [(2, 32, 4), (3, 32, 4), (4, 16, 8), (5, 16, 8), (5, 32, 4)]   # N, tile columns, rows
MESHES = [(1, 3), (2, 9), (4, 2), (15, 19), (16, 8), (33, 5), (35, 19), (67, 9), (64, 13)]


class Geo:
    def __init__(self, geometry):
        N, self.TX, self.TY = geometry
        self.N, self.EL = N, 3 * N * N
        self.VEC = (N * N) % 4 == 0
        EL = self.EL
        self.ES = (EL if (EL // 4) % 2 else EL + 4) if self.VEC else EL
        self.ROW = self.TX * self.ES if self.VEC else self.TX * EL + 32
        s0 = self.ES if self.VEC else (EL + 6) // 4 * 4
        self.SLOT = s0 if (s0 // 4) % 2 else s0 + 4
        c1, r1 = self.TX + 1, self.TY + 1
        self.TE = self.TY * self.ROW
        self.TN = self.TE + 3 * N * self.TY * c1
        self.RW = self.TN + 3 * N * r1 * self.TX
        self.RS = self.RW + 3 * N * self.TY
        self.U = (self.RS + 3 * N * self.TX + 3) // 4 * 4
        self.RING = 2 * self.ROW + 2 * self.TY * self.SLOT
        self.LEN = self.U + max(self.RING, 3 * N * (self.TY * c1 + r1 * self.TX))

    def block(self, c):
        """Shared-memory position of 16-byte block c of a row."""
        return (c // (self.EL // 4)) * self.ES + c % (self.EL // 4) * 4 if self.VEC else 4 * c


@pytest.mark.parametrize("geometry", GEOMETRY)
def test_shared_memory_fits(geometry):
    g = Geo(geometry)
    ctas = {(2, 32): 6, (3, 32): 5, (4, 16): 4, (5, 16): 3, (5, 32): 2}[geometry[:2]]
    assert g.U % 4 == 0 and g.ROW % 4 == 0 and g.SLOT % 4 == 0
    assert ctas * (4 * g.LEN + 1024) <= 228 * 1024
    # the lanes of a warp read word m of 32 elements (or 16-byte block m of 8)
    if g.VEC:
        assert len({(k * g.ES // 4) % 8 for k in range(8)}) == 8
    else:
        lanes = [(k // g.TX) * g.ROW + (k % g.TX) * g.ES for k in range(32)]
        assert len({a % 32 for a in lanes}) == 32


@pytest.mark.parametrize("gs,gn", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("nlon,nlat", MESHES)
@pytest.mark.parametrize("geometry", GEOMETRY)
def test_tiles(geometry, nlon, nlat, gs, gn):
    g = Geo(geometry)
    EL, TX, TY = g.EL, g.TX, g.TY
    row = nlon * EL
    base = gs * row                                        # own row 0; the array starts 16-byte aligned
    end = ((nlat + gs + gn) * row + 3) // 4 * 4            # padded length
    written = np.zeros(end, dtype=int)

    def copy(sm, at, o, count):
        """Blocks holding values o .. o + count, placed from shared position at; returns the lead."""
        lead = 0 if g.VEC else (base + o) % 4
        assert (base + o - lead) % 4 == 0                  # aligned source (VEC: every row starts on a block)
        for c in range((lead + count + 3) // 4):
            a = base + o - lead + 4 * c
            assert 0 <= a and a + 4 <= end
            p = at + (g.block(c) if count > EL or not g.VEC else 4 * c)
            assert p + 4 <= len(sm)
            sm[p:p + 4] = np.arange(a, a + 4)
        return lead

    for j0 in range(0, nlat, TY):
        for i0 in range(0, nlon, TX):
            Gv, Wv = min(TX, nlon - i0), min(TY, nlat - j0)
            off = lambda j, i: (j * nlon + i) * EL  # noqa: E731
            for r in range(Wv):
                sm = np.full(g.ROW, -1)
                o = off(j0 + r, i0)
                lead = copy(sm, 0, o, Gv * EL)
                for k in range(Gv):
                    at = lead + k * g.ES
                    assert np.array_equal(sm[at:at + EL], base + o + k * EL + np.arange(EL))
                stop = lead + Gv * EL
                for c in range((stop + 3) // 4):           # output blocks
                    a = base + o - lead + 4 * c
                    if g.VEC or (4 * c >= lead and 4 * c + 4 <= stop):
                        written[a:a + 4] += 1
                    else:
                        for t in range(4):
                            if lead <= 4 * c + t < stop:
                                written[a + t] += 1
            ring = np.full(g.RING, -1)
            for there, at, jj in ((j0 > 0 or gs, 0, j0 - 1), (j0 + Wv < nlat or gn, g.ROW, j0 + Wv)):
                if there:
                    lead = copy(ring, at, off(jj, i0), Gv * EL)
                    for k in range(Gv):
                        p = at + lead + k * g.ES
                        assert np.array_equal(ring[p:p + EL], base + off(jj, i0 + k) + np.arange(EL))
            for s in range(2 * TY):
                w = s % TY
                if w < Wv:
                    i = (i0 - 1) % nlon if s < TY else (i0 + Gv) % nlon
                    at = 2 * g.ROW + s * g.SLOT
                    lead = copy(ring, at, off(j0 + w, i), EL)
                    assert lead + EL <= g.SLOT
                    assert np.array_equal(ring[at + lead:at + lead + EL], base + off(j0 + w, i) + np.arange(EL))
    assert np.all(written[base:base + nlat * row] == 1)
    assert written.sum() == nlat * row
