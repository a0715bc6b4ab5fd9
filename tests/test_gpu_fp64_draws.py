"""FP64 draws from tables and FP64 hops decided by an FP32 filter, through the public calls.

Draws: with no springs, no forces (all beads at the origin) and amp = sqrt(2 kT dt / zeta)
= 1, the positions after one step are the Box-Muller normals themselves, exactly.

Hops: beads that do not move (zeta = 1e300) and one step with springs three beads apart,
whose anchors and neighbours are placed so that a move's probability lies within 1e-10 to
1e-5 of the slot's uniform, far inside the error of FP32: the filter has to hand these to
the FP64 probabilities.
"""
import math

import numpy as np
import pytest

import oracle
from paper_1106_2899_gb300 import SlipSpring

pytestmark = pytest.mark.gpu

MASK = 0xFFFFFFFF


def _philox_step(idx, chain, seed, step=0):
    """Words of Philox4x32-10 of counter (idx, step, 1, chain): int64 tensors."""
    import torch
    c = [idx, torch.full_like(idx, step), torch.full_like(idx, 1), chain.expand_as(idx)]
    k0, k1 = seed & MASK, seed >> 32
    for _ in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57
        c = [((p1 >> 32) & MASK) ^ c[1] ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c[3] ^ k1, p0 & MASK]
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c


def _pair(wa, wb):
    """(radius, r cos, r sin) of a pair in FP64: the angle -pi + 2 pi k / 2^24 reduced to
    an eighth of a turn in integers."""
    import torch
    r = torch.sqrt(-2.0 * torch.log(((wa >> 8) + 1).double() / 2**24))
    k = wb >> 8
    q = (k + (1 << 21)) >> 22
    x = (k - (q << 22)).double() * (2.0 * math.pi / 2**24)
    c, s = torch.cos(x), torch.sin(x)
    q = (q + 2) & 3  # less half a turn
    cos = torch.where(q == 0, c, torch.where(q == 1, -s, torch.where(q == 2, -c, s)))
    sin = torch.where(q == 0, s, torch.where(q == 1, c, torch.where(q == 2, -s, -c)))
    return r, r * cos, r * sin


def test_normals_over_the_lattice(cuda_ok):
    import torch
    M, N, seed = 131072, 128, 9
    g = SlipSpring([(M, N)], precision="fp64", seed=seed)
    g.set_params(N0=math.inf, zeta_s=1.0, dt=0.5, kT=1.0, zeta=1.0, k_b=1e-3, k_s=1e-3, corr_levels=-1)
    dev = dict(device="cuda")
    R = torch.zeros(M, N, 3, dtype=torch.float64, **dev)
    zm = 64
    Z, S = torch.zeros(M, dtype=torch.int32, **dev), torch.full((M, zm), -1, dtype=torch.int32, **dev)
    A = torch.zeros(M, zm, 3, dtype=torch.float64, **dev)
    g.set_state_dev(R, Z, S, A)
    g.run(1)
    g.get_state_dev(R, Z, S, A)
    g.synchronize()
    assert g.status() == 0
    g.close()
    idx = torch.arange(N, **dev)[None, :].expand(M, N).contiguous()
    w = _philox_step(idx, torch.arange(M, **dev)[:, None], seed)
    for m, i in ((0, 0), (5, 127), (131071, 64)):
        assert [int(x[m, i]) for x in w] == [int(x) for x in oracle.philox([i, 0, 1, m], [seed, 0])]
    # every interval of the logarithm's table and every angle of the other one
    lattice = (w[0] >> 8) + 1
    e = torch.floor(torch.log2(lattice.double())).long()
    assert len(torch.unique(e)) >= 22 and len(torch.unique((lattice << 10 >> e).flatten())) >= 1024
    assert len(torch.unique((w[1] >> 8) >> 14)) == 1024
    # Bound relative to the radius.  Tables: radius 2.6e-16, sine and cosine 2.2e-16,
    # product 1.1e-16.  Here: logarithm 1 ulp, halved by the root, 1.1e-16, the root's
    # rounding 1.1e-16, sine and cosine 1.1e-16 and the angle's rounding 1.2e-16, product
    # 1.1e-16.  Sum 1.15e-15.
    for wa, wb, cols in ((w[0], w[1], (0, 1)), (w[2], w[3], (2,))):
        r, c, s = _pair(wa, wb)
        for d, ref in zip(cols, (c, s)):
            err = torch.abs(R[:, :, d] - ref)
            assert bool(torch.all(err <= 1.2e-15 * r)), float((err / r.clamp(min=1e-300)).max())


@pytest.mark.parametrize("N", [128, 30])  # lane layouts of four and of two beads
def test_hops_at_the_edge_of_their_probabilities(cuda_ok, N):
    M, seed = 4000, 77
    rng = np.random.default_rng(3)
    s0 = np.arange(4, N - 5, 3)  # the springs' beads
    Z = len(s0)
    pref, chop = 0.25, 1.0  # dt kT / zeta_s, k_s / (4 kT)
    import torch
    w = _philox_step(torch.arange(Z)[None, :].expand(M, Z).contiguous(), torch.arange(M)[:, None], seed)
    k = ((w[0] & 255) | ((w[1] & 255) << 8) | ((w[2] & 255) << 16)).numpy()
    u = k / 2.0**24
    # probability pref (1 - tanh y) of a move with y = chop (change of squared length)
    def change_for(p):
        return np.arctanh(1.0 - p / pref) / chop

    R = np.zeros((M, N, 3))
    R[:, :, 0] = 1.0 + 0.1 * np.arange(N)
    R[:, :, 1:] = 0.5
    delta = 10.0 ** rng.uniform(-10, -5, (M, Z)) * rng.choice([-1.0, 1.0], (M, Z))
    first = rng.random((M, Z)) < 0.5  # the edge between up and the rest, or between down and none
    p_up = np.where(first, u * (1.0 + delta), u * rng.uniform(0.2, 0.8, (M, Z)))
    p_dn = np.where(first, 0.1, u * (1.0 + delta) - p_up)
    edge = (u > 1e-3) & (p_up < 0.495) & (p_dn > 1e-4) & (p_dn < 0.495)
    p_up, p_dn = np.where(edge, p_up, 0.2), np.where(edge, p_dn, 0.1)

    def unit():
        v = rng.normal(size=(M, Z, 3))
        return v / np.linalg.norm(v, axis=-1, keepdims=True)

    d0 = rng.uniform(2.5, 4.0, (M, Z))  # larger than any change of squared length is negative
    A = R[:, s0] + unit() * np.sqrt(d0)[..., None]
    R[:, s0 + 1] = A + unit() * np.sqrt(d0 + change_for(p_up))[..., None]
    R[:, s0 - 1] = A + unit() * np.sqrt(d0 + change_for(p_dn))[..., None]

    def prob(b):  # from the rounded coordinates
        x = np.longdouble(1.0) * (R[:, b] - A)
        y = np.longdouble(1.0) * (R[:, s0] - A)
        t = 2.0 * chop * ((x * x).sum(-1) - (y * y).sum(-1))
        return np.minimum(2.0 * pref / (1.0 + np.exp(t)), 0.5)

    pp, pm = prob(s0 + 1), prob(s0 - 1)
    assert edge.mean() > 0.2 and np.all(np.isfinite(pp)) and np.all(np.isfinite(pm))
    near = np.minimum(np.abs(u - pp), np.abs(u - (pp + pm)))
    clear = near > 1e-13  # the probabilities of FP64 are good to 1e-14
    assert clear.mean() > 0.999 and (near < 1e-6).mean() > 0.2
    want = np.where(u < pp, s0 + 1, np.where(u < pp + pm, s0 - 1, s0))

    g = SlipSpring([(M, N)], precision="fp64", seed=seed)
    g.set_params(N0=1e6, zeta_s=1.0, dt=0.25, kT=1.0, zeta=1e300, k_b=1.0, k_s=4.0, z_max=Z, corr_levels=-1)
    S = np.broadcast_to(s0, (M, Z)).astype(np.int32)
    g.set_state({"R": R, "Z": np.full(M, Z, dtype=np.int32), "S": S, "A": A})
    g.run(1)
    got = g.get_state()
    assert g.status() == 0
    g.close()
    assert np.array_equal(got["R"], R) and np.array_equal(got["A"], A) and np.all(got["Z"] == Z)
    assert np.array_equal(got["S"][clear], want[clear])
    assert 0.05 < np.mean(want > s0) < 0.95 and np.mean(want < s0) > 0.02
