"""1/r of the FP64 energy pass from a single-precision root and one third-order
step: two opposite charges without Lennard-Jones terms, E = f q q' / eps_r (1/r +
k_rf r^2 - c_rf), at distances from 1/20 of the cutoff to the cutoff.

With u = 2^-53 and exact coordinates (x = L i / 2^32 for the integer offset i),
r^2 carries 2 u from each of its squares' factors and 3 u from its sums, 1/r half
of that and the 2 u of one unit in the last place; the rest of the formula five
roundings of at most its largest term: below 10 u of f q q' / eps_r (1/r + k_rf r^2
+ c_rf).  Without the third-order term the error would be 2^-41 of 1/r."""
import math
from fractions import Fraction

import numpy as np
import pytest

from _systems import beads
from paper_2005_08348_gb300 import mdas

pytestmark = pytest.mark.gpu
RC = 1.1


def _root(x):
    """sqrt of a positive fraction to 2^-200 of 1."""
    s = 1 << 400
    return Fraction(math.isqrt(x.numerator * s // x.denominator), 1 << 200)


@pytest.mark.parametrize("box", [(4.0, 4.0, 4.0), (4.0, 5.6, 4.7)])
def test_one_pair_to_the_last_place(box):
    rng = np.random.default_rng(7)
    m = beads([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0]], [0, 1], box=box, eps=np.zeros((10, 10)))
    s = mdas.System(m, precision="fp64")
    qq = Fraction(138.935458) * -1 / Fraction(m.eps_r)
    krf, crf = Fraction(1, 2) / Fraction(RC) ** 3, Fraction(3, 2) / Fraction(RC)
    st = s.get_state()
    for k in range(300):
        r = RC * math.exp(rng.uniform(math.log(0.05), 0.0)) * 0.9999
        d = rng.normal(size=3) if k % 2 else np.eye(3)[k // 2 % 3]
        d = d * (r / np.linalg.norm(d))
        off = np.rint(d / np.asarray(box) * 2.0 ** 32).astype(np.int64)
        base = rng.integers(0, 2 ** 32, 3)
        pos = np.stack([base, base + off]) % 2 ** 32
        s.set_state(pos_u=pos.astype(np.uint32), vel=st["vel"], ltype=st["ltype"])
        e = s.energy()
        r2 = sum((Fraction(int(o)) * Fraction(float(L)) / 2 ** 32) ** 2 for o, L in zip(off, box))
        ri = 1 / _root(r2)
        want = qq * (ri + krf * r2 - crf)
        scale = abs(qq) * (ri + krf * r2 + crf)
        assert e["pairs"] == 1 and e["lj"] == 0.0
        assert abs(Fraction(e["rf"]) - want) <= 10 * scale / 2 ** 53, (k, r)
    s.close()
