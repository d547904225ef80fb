"""Output tiles of the pair contraction in the residue form (256 x 256), no GPU: they
cover every element the pass needs exactly once, none is listed without one, and the
largest workload pads little."""
import numpy as np
import pytest

import paper_2312_07008_gb300 as pkg

T = 256
FORM = 10      # moduli of the residue form


@pytest.mark.parametrize("nc,na,nv", [(3, 0, 40), (4, 2, 61), (2, 5, 130), (5, 3, 7), (2, 1, 255), (3, 0, 256), (2, 2, 300)])
@pytest.mark.parametrize("energy_only", [False, True])
def test_tiles_cover_each_needed_element_once(nc, na, nv, energy_only):
    nh, np_ = nc + na, na + nv
    rng = np.random.default_rng(nc * 100 + na * 10 + nv)
    allp = [(i, j) for i in range(nh) for j in range(i, nh)]
    pick = rng.choice(len(allp), size=max(1, len(allp) // 2), replace=False)
    pairs = [allp[k] for k in sorted(pick)]
    need = np.zeros((nh * np_, nh * np_), dtype=bool)
    for i, j in pairs:
        blk = np.ones((np_, np_), dtype=bool)
        blk[:na, :na] = False
        if energy_only:
            blk[:na, :] = blk[:, :na] = False
        need[i * np_:(i + 1) * np_, j * np_:(j + 1) * np_] |= blk
    tiles = pkg.dsrg_fno_debug_pair_tiles(FORM, nc, na, nv, pairs, energy_only)
    assert len(set(tiles)) == len(tiles)
    cover = np.zeros_like(need, dtype=np.int32)
    for mt, nt in tiles:
        assert 0 <= mt * T < nh * np_ and 0 <= nt * T < nh * np_
        assert need[mt * T:(mt + 1) * T, nt * T:(nt + 1) * T].any(), (mt, nt)
        cover[mt * T:(mt + 1) * T, nt * T:(nt + 1) * T] += 1
    assert np.all(cover[need] == 1)
    band = [mt // 8 for mt, _ in tiles]
    assert band == sorted(band)


def test_padding_of_a_whole_workload():
    """nvir 1200, CAS(10,10), 60 core: the listed tiles hold the needed elements of all
    pairs with under 2 % padding (half a tile along the diagonal and the last rows)."""
    nc, na, nv = 60, 10, 1200
    nh, np_ = nc + na, na + nv
    pairs = [(i, j) for i in range(nh) for j in range(i, nh)]
    tiles = pkg.dsrg_fno_debug_pair_tiles(FORM, nc, na, nv, pairs, False)
    needed = len(pairs) * (np_ * np_ - na * na)
    assert needed <= len(tiles) * T * T <= 1.02 * needed
