"""The resident solve's index arithmetic (csrc/resident.cu), replayed on the
CPU: how a mesh's slabs (2D rows, 3D planes) are dealt to the CTAs of a
cluster, the multiply-high division of a thread's node number, the slabs a
stencil, a restriction and a prolongation read, and the shared memory they
need. Every interior node is visited once, and every slab a CTA reads lies in
the band of the CTA it is read from, or is the slab of zeros."""
import pytest

THREADS, BAND, MAX_V, PORTABLE, MAX_LEVELS, SMEM, SHARE = 256, 512, 16, 8, 7, 224 * 1024, 74 * 1024


def layout(dim, n, K, V, C, mixed, solve=True):
    """(levels, nd, bytes): the geometry and shared memory of one CTA."""
    size = 4 if mixed else 8
    off = 0

    def take(count, sz):
        nonlocal off
        off = (off + 15) // 16 * 16 + count * sz
    nv = V // C
    rv = max(1, n // V) if K > 1 else -(-(n - 1) // V)
    nd, lv = 0, []
    for l in range(K):
        nl = n >> l
        N1 = nl + 1
        S = N1 if dim == 2 else N1 * N1
        split = C > 1 and nd == l and (l == 0 or (nl >= C and nl > (16 if dim == 2 else 4)))
        if split:
            nd = l + 1
        R = (max(1, nl // C) if K > 1 else -(-nv * (n - 1) // V)) if split else nl - 1
        m = max(1, nl - 1)
        lv.append(dict(n=nl, N1=N1, S=S, R=R, m1=-(-2 ** 32 // m) % 2 ** 32, m2=-(-2 ** 32 // (m * m)) % 2 ** 32))
        for _ in range((0 if K > 1 and l == K - 1 else 2) + (1 if K > 1 else 0)):
            take(R * S, size)
    take(lv[0]["S"], size)
    if solve:
        for _ in range(2):
            take(lv[0]["R"] * lv[0]["S"], size)
        take(4 * 2 * MAX_V, 8)
        take((1 if K > 1 else 2) * nv * THREADS, 8)
        take(48, 1)
    lv[0]["edge"] = [v * (n - 1) // V if K == 1 else min(v * rv, n - 1) for v in range(V + 1)]
    lv[0]["nv"] = nv
    return lv, nd, (off + 15) // 16 * 16


def cells(dim, K, mixed):
    """Largest mesh whose solves run resident."""
    if K > 1:
        return 128 if dim == 2 else 16
    return (256 if mixed else 170) if dim == 2 else (30 if mixed else 24)


def bands(dim, n, K, mixed):
    if n < 2 or K > MAX_LEVELS or n > cells(dim, K, mixed):
        return 0
    V = 1
    while V < PORTABLE and (n - 1) ** dim > V * BAND and 2 * V <= n:
        V *= 2
    if K == 1 and V == PORTABLE and (n - 1) ** dim > V * BAND and n >= MAX_V:
        V = MAX_V
    return V if layout(dim, n, K, V, V, mixed)[2] <= SMEM else 0


def band(lv, nd, C, l, rank):
    """(first slab, slabs) of a CTA on level l."""
    if l >= nd and rank:
        return 1, 0
    if l == 0:
        edge, nv = lv[0]["edge"], lv[0]["nv"]
        return edge[rank * nv] + 1, edge[(rank + 1) * nv] - edge[rank * nv]
    z0 = rank * lv[l]["R"] + 1 if l < nd else 1
    return z0, max(0, min(lv[l]["R"], lv[l]["n"] - z0))


CASES = [(2, 1 << k, k, mx) for k in range(2, 9) for mx in (False, True)] + \
        [(3, 1 << k, k, mx) for k in range(2, 7) for mx in (False, True)] + \
        [(2, n, 1, mx) for n in (2, 3, 9, 31, 45, 67, 100, 129, 170, 171, 200, 235, 256, 257) for mx in (False, True)] + \
        [(3, n, 1, mx) for n in (2, 3, 9, 17, 24, 25, 30, 31, 40) for mx in (False, True)]


@pytest.mark.parametrize("dim,n,K,mixed", CASES)
def test_bands_slabs_and_shared_memory(dim, n, K, mixed):
    V = bands(dim, n, K, mixed)
    # every mesh up to the largest has its bands: none is left out by its shared memory
    assert (V > 0) == (n <= cells(dim, K, mixed))
    if V == 0:
        return
    C = V
    while C >= 1:
        check(dim, n, K, mixed, V, C)
        C //= 2
        if C and layout(dim, n, K, V, C, mixed)[2] > SHARE:
            break


def check(dim, n, K, mixed, V, C):
    lv, nd, bytes_ = layout(dim, n, K, V, C, mixed)
    assert bytes_ <= SMEM and nd <= max(1, K - 1) and (C == 1) == (nd == 0)
    # the bands of the sums: rv slabs each, together every slab of level 0, V / C per CTA
    edge = lv[0]["edge"]
    assert edge[0] == 0 and edge[V] == n - 1 and all(a < b or (K > 1 and b == n - 1) for a, b in zip(edge, edge[1:]))
    for l, L in enumerate(lv):
        nl, m, R, S = L["n"], L["n"] - 1, L["R"], L["S"]
        if K > 1 and l < nd:
            assert R & (R - 1) == 0 and R * C == nl
        owner = {}
        for r in range(C):
            z0, own = band(lv, nd, C, l, r)
            assert own <= R
            per = m if dim == 2 else m * m
            seen = set()
            for x in range(own * per):
                js = (x * (L["m1"] if dim == 2 else L["m2"])) >> 32
                rem = x - js * per
                j = 0 if dim == 2 else ((rem * L["m1"]) >> 32) + 1
                i = rem - (j - 1) * m + 1 if dim == 3 else rem + 1
                assert 0 <= js < own and 1 <= i <= m and (dim == 2 or 1 <= j <= m)
                o = i if dim == 2 else j * L["N1"] + i
                # the row (plane) neighbours of the node lie in its slab
                assert o - (1 if dim == 2 else L["N1"] + 1) >= 0 and o + (1 if dim == 2 else L["N1"] + 1) < S
                seen.add((js, o))
            assert len(seen) == own * per
            for js in range(own):
                assert z0 + js not in owner
                owner[z0 + js] = (r, js)
        assert sorted(owner) == list(range(1, nl))

        def slab(z):
            """(CTA, slab in its band) as the kernel addresses it, None for the zeros."""
            if z <= 0 or z >= nl:
                return None
            return ((z - 1) // R, (z - 1) % R) if l < nd else (0, z - 1)
        if K > 1:   # one level alone has no transfers: its bands are even shares, read by before and after only
            for z in range(1, nl):
                assert slab(z) == owner[z]
        for r in range(C):
            z0, own = band(lv, nd, C, l, r)
            if own == 0:
                continue
            # the slabs before and after the band: the last of CTA r - 1, the first of CTA r + 1
            last = (band(lv, nd, C, 0, r - 1)[1] if l == 0 and r else R) - 1
            assert owner.get(z0 - 1) == (None if r == 0 or l >= nd else (r - 1, last))
            assert owner.get(z0 + own) == (None if z0 + own >= nl else (r + 1, 0))
        if K > 1 and l + 1 < K:
            nc = lv[l + 1]["n"]
            for z in range(1, nc):       # full weighting reads fine slabs 2z - 1 .. 2z + 1, columns 2I - 1 .. 2I + 1
                assert all(slab(f) is not None for f in (2 * z - 1, 2 * z, 2 * z + 1)) and 2 * (nc - 1) + 1 <= nl
            for z in range(1, nl):       # prolongation reads coarse slabs z / 2 (and z / 2 + 1 for odd z)
                assert 0 <= z >> 1 and (z >> 1) + (z & 1) <= nc and ((nl - 1) >> 1) + 1 <= nc


BOTTOM_SLOTS = 152 * 3


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("dim,n,K", [(2, 1 << k, k) for k in range(2, 7)] + [(3, 1 << k, k) for k in range(2, 5)])
def test_bottom_levels_fit_every_batch(dim, n, K, mixed):
    """The V-cycle's fused levels: the CTAs a batch gives a sample, each with room for its arrays."""
    top = 1
    while top < PORTABLE and (n - 1) ** dim > top * THREADS and 2 * top <= n:
        top *= 2
    for B in (1, 40, 57, 58, 100, 500, 60000):
        C = top
        while C > 1 and B * C > BOTTOM_SLOTS and layout(dim, n, K, C // 2, C // 2, mixed, False)[2] <= SHARE:
            C //= 2
        lv, nd, bytes_ = layout(dim, n, K, C, C, mixed, False)
        assert bytes_ <= SMEM and nd <= K - 1 and (C == 1) == (nd == 0)
        for l in range(nd):
            assert lv[l]["R"] * C == lv[l]["n"]
