"""The bond-weight kernels at the edges of their work split: few (qz, w) rows, column counts around a block, so many
columns that a thread walks down several rows, one to eight bonds around the four of an adjoint step, more bonds than the
adjoint's table of reverse bonds holds, and lists in which some bonds have no reverse (zero weight, zero gradient, status
reported). The reference adds the same terms in numpy in the order of Eq. (3): the forward is equal to the bit,
and so is the adjoint (slot sums of two terms, self blocks subtracted bond by bond)."""
import numpy as np
import pytest
import torch

from paper_1912_10024_gb300 import binding as B

pytestmark = pytest.mark.gpu


def reverse_slots(nbr):
    NA, NB = nbr.shape
    rev = -np.ones((NA, NB), dtype=int)
    for a in range(NA):
        for s in range(NB):
            hit = [k for k in range(NB) if nbr[nbr[a, s], k] == a]
            rev[a, s] = hit[0] if hit else -1
    return rev


@pytest.mark.parametrize("NA,NB,Nqz,Nw,steps", [
    (3, 1, 1, 1, [1]), (2, 1, 1, 3, [1]), (13, 2, 2, 2, [1, -1]), (15, 2, 5, 1, [1, -1]), (7, 4, 3, 3, [1, -1, 2, -2]),
    (12, 3, 2, 4, [1, -1, 3]), (33, 3, 1, 7, [2, -2, 5]),
    (17, 5, 1, 3, [1, -1, 2, -2, 4]), (19, 7, 2, 2, [1, -1, 2, -2, 3, -3, 5]), (20, 8, 1, 5, [1, -1, 2, -2, 3, -3, 4, -4]),
    (66, 65, 1, 3, [s for k in range(1, 33) for s in (k, -k)] + [33]),
    (3000, 2, 1, 13, [1, -1]),  # 211 and 106 blocks across: 5 and 11 of the 13 rows at once
], ids=str)
def test_row_and_column_remainders(NA, NB, Nqz, Nw, steps):
    nbr = np.array([[(a + s) % NA for s in steps] for a in range(NA)], dtype=np.int32)
    rev = reverse_slots(nbr)
    rng = np.random.default_rng(NA + NB)

    def draw(n):
        return rng.standard_normal((Nqz, Nw, NA, n, 3, 3)) + 1j * rng.standard_normal((Nqz, Nw, NA, n, 3, 3))

    raw, g = [draw(NB + 1) for _ in range(2)], [draw(NB) for _ in range(2)]
    n = torch.from_numpy(nbr).cuda()
    fwd = B.dcomb(*[torch.from_numpy(x).cuda() for x in raw], n)
    bwd = B.dcomb_grad(*[torch.from_numpy(x).cuda() for x in g], n)
    for t in range(2):
        ref, adj = np.zeros_like(g[t]), np.zeros_like(raw[t])
        for a in range(NA):
            for s in range(NB):
                b, r = nbr[a, s], rev[a, s]
                if r < 0:
                    continue
                R, G = raw[t], g[t]
                ref[:, :, a, s] = R[:, :, b, r] - R[:, :, b, NB] - R[:, :, a, NB] + R[:, :, a, s]
                both = G[:, :, a, s] + G[:, :, b, r]
                adj[:, :, a, s] = both
                adj[:, :, a, NB] -= both
        assert np.array_equal(fwd[t].cpu().numpy(), ref) and np.array_equal(bwd[t].cpu().numpy(), adj)
    if (rev < 0).any():
        with pytest.raises(B.SseError):
            B.dcomb_grad(*[torch.from_numpy(x).cuda() for x in g], n, check=True)
