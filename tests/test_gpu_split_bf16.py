"""The split-bf16 contractions (csrc/k_tc.cu) against the oracle at sizes where
their K blocks, M tiles and N tiles end: products past the last element are not
issued, the last M tile has boxes of its own height, wide right-hand sides
are cut into tiles of equal height, and the last stage takes two core states
per thread from 40,000 (k, band, state pairs) on.  Bounds: those of
parity_check.py for this arithmetic."""
import numpy as np
import pytest

from oracle import bse_oracle as O
from paper_1601_07728_gb300 import bse, synth as S
from parity_check import close

pytestmark = pytest.mark.gpu


# bands: 2 Nb around 64-element K blocks and 128-row M tiles; grid points: around
# K blocks of 64, K steps of 16 and M tiles of 128; columns (core states x
# vectors): B rows 2 to 576 in one, two and three tiles
@pytest.mark.parametrize("case", [
    ((2, 2, 2), (5, 5, 5), 65, 1, 0, 1), ((2, 2, 2), (8, 8, 2), 64, 6, 4, 1), ((2, 2, 2), (43, 3, 1), 63, 6, 4, 2),
    ((2, 2, 1), (11, 12, 1), 70, 6, 9, 22), ((1, 2, 2), (7, 7, 7), 129, 6, 4, 32), ((2, 1, 2), (17, 8, 1), 9, 6, 4, 43),
    ((1, 1, 2), (5, 13, 9), 33, 4, 4, 33), ((2, 2, 2), (257, 1, 1), 8, 6, 4, 48), ((1, 1, 1), (9, 9, 9), 193, 10, 4, 13),
    # around the rule for pairs of core states: 39,960 and 40,080
    ((2, 2, 2), (6, 6, 6), 37, 6, 4, 45), ((2, 5, 2), (6, 6, 3), 4, 6, 4, 167)])
def test_apply_matches_oracle(case):
    nk, nx, nb, na, npj, nv = case
    s = S.make_system_from(dict(id=971, n_alpha=na, nk=nk, n_bands=nb, nx=nx, cell=7.4, eps=5.0, n_proj=npj,
                                so_split=5.7, m_scale=0.5, kshift=(0.1, 0.0, 0.2)), 5)
    psi = S.make_start_vectors(s, nv)
    out = bse.System(s, precision="split_bf16", max_vec=nv).apply_h(psi)
    for v in {0, nv // 2, nv - 1}:
        close("split_bf16/%s/v%d" % (case, v), out[v], O.apply_h(s, psi[v]), "split_bf16")
