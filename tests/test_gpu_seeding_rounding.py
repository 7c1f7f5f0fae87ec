"""K-means++ seeding (csrc/seeding.cu): a point of weight 0 is never chosen while another has weight.

The running sums of the weights come from scans, so the sum up to a point of weight 0 can exceed the
one before it by a rounding.  Both scans (over a block's points, over the blocks) are repeated here in
float64, and u is chosen so that the target falls into such a gap.  Linear kernel, d = 1, first point 0:
the weights are p^2, exact in float64."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _scan(v):
    """Inclusive running sums over the 32 lanes of a warp, in the order of shuffles by 1, 2, 4, 8, 16."""
    v = np.array(v, dtype=np.float64)
    o = 1
    while o < 32:
        u = v.copy()
        u[o:] = v[o:] + v[:-o]
        v = u
        o *= 2
    return v


def _draw_for(target, W):
    """u in [0, 1) with fl(u W) == target, or None."""
    u = target / W
    for _ in range(8):
        if u * W == target:
            return u if u < 1 else None
        u = np.nextafter(u, 1.0 if u * W < target else 0.0)
    return None


def _seed(p, first, u):
    import paper_2501_05587_gb300 as pc
    P = torch.from_numpy(p.astype(np.float32).reshape(-1, 1)).cuda()
    n = len(p)
    r = pc.popcorn_kmeanspp(P, 2, pc.kernel_spec("linear"), np.array([(first + 0.5) / n, u]))
    c = r["centers"]
    assert c[0] == first
    return c[1]


def test_a_gap_between_the_points_of_a_block():
    G = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(0)
    n, tried = 32 * G, 0                       # 32 points a block, a lane each
    while tried < 6:
        p = np.zeros(n, dtype=np.float32)
        p[:32] = rng.uniform(0.5, 2.0, 32)
        z = int(rng.integers(2, 31))
        p[z] = 0.0
        inc = _scan(p[:32].astype(np.float64) ** 2)
        if not inc[z] > inc[z - 1]:
            continue
        u = _draw_for(inc[z - 1], inc[31])     # the other blocks add nothing: W = inc[31]
        if u is None:
            continue
        tried += 1
        c = _seed(p, n - 1, u)
        assert p[c] != 0.0, (z, c)


def test_a_gap_between_blocks():
    G = torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.default_rng(1)
    per, m = (G + 31) // 32, 8                 # blocks a lane; points a block
    n, tried = m * G, 0
    while tried < 6:
        w = np.zeros(32 * per)
        q = np.zeros(32 * per, dtype=np.float32)
        q[:G - 1] = rng.uniform(0.5, 2.0, G - 1)   # the last block holds the first point and no weight
        lane = int(rng.integers(1, (G - 1) // per - 1))
        q[per * (lane + 1)] = 0.0
        w[:] = q.astype(np.float64) ** 2
        s = np.zeros(32)
        for x in range(32):
            for b in range(per * x, min(per * (x + 1), G)):
                s[x] += w[b]
        upto = _scan(s)
        run = upto[lane - 1]
        for b in range(per * lane, per * (lane + 1)):
            run += w[b]
        if not run < upto[lane]:               # the lane's own running sum ends below the scan's
            continue
        u = _draw_for(run, upto[31])
        if u is None:
            continue
        tried += 1
        p = np.zeros(n, dtype=np.float32)
        p[3::m][:G] = q[:G]                    # one weighted point a block
        c = _seed(p, n - 1, u)
        assert p[c] != 0.0, (lane, c)
