"""The codebook search on the tensor cores gives the codes of the FP32 scan.

Every code is the first entry with the smallest d2 = fma chain of (x_d - c_d)^2 in FP32, computed here
with the squares and sums of each step formed in float64 and rounded to float32 (a double rounding
would have to fall on the smallest d2 of a point to be seen). Point counts at the edges of the
256-point tiles, entries that are all different, few and many times repeated, walls of equal points, and
values that are NaN, infinite or huge (those points scan every entry; with no finite distance the
code is 0).
"""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu
GROUPS = {"sggx": (7, 6), "material": (13, 16)}   # offset and width in a codebook row


@pytest.fixture(scope="module")
def ugp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp as U
    build.build()
    U.lib()
    return U


def _scan(torch, X, B):
    """First entry of smallest d2, in the arithmetic of the FP32 scan; 0 when no d2 is finite."""
    code = torch.zeros(X.shape[0], dtype=torch.long, device="cuda")
    for i in range(0, X.shape[0], 256):
        x = X[i:i + 256]
        d2 = torch.zeros(x.shape[0], B.shape[0], device="cuda")
        for d in range(B.shape[1]):
            v = (x[:, d:d + 1] - B[None, :, d]).double()
            d2 = (v * v + d2.double()).float()
        d2 = torch.where(torch.isfinite(d2), d2, torch.full_like(d2, float("inf")))
        m = d2.min(1, keepdim=True).values
        first = (d2 == m).to(torch.int32).argmax(1)
        code[i:i + 256] = torch.where(torch.isinf(m[:, 0]), torch.zeros_like(first), first)
    return code


@pytest.mark.parametrize("kind", ["spread", "few", "extreme"])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 12_345])
def test_codes_are_those_of_the_scan(ugp, n, kind):
    import torch
    rng = np.random.Generator(np.random.Philox(1000 * n + len(kind)))
    s = scenes.with_disney(scenes.room_scene(max(n, 100), seed=n, n_clusters=5), 0.5, seed=2).subset(np.arange(n))
    sggx, alb, emi, dis = s.sggx.copy(), s.albedo.copy(), s.emission.copy(), s.disney.copy()
    if kind == "spread":
        sggx = rng.normal(size=sggx.shape).astype(np.float32)
        alb = rng.random(alb.shape).astype(np.float32)
    elif kind == "few":   # three materials and one normal: nearly every entry is a repetition
        pick = rng.integers(0, 3, n)
        alb, emi, dis = alb[pick % n], emi[pick % n], dis[pick % n]
        sggx = np.repeat(sggx[:1], n, 0)
    else:
        alb[rng.random(n) < 0.02, 0] = np.nan
        emi[rng.random(n) < 0.02, 1] = np.inf
        emi[rng.random(n) < 0.02, 2] = 1e25
        sggx[rng.random(n) < 0.02, 3] = -3e18
        sggx[rng.random(n) < 0.02, 2] = 1e13
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    rough = t(s.roughness)
    mats = ugp.Materials(t(sggx), torch.from_numpy(s.mtype.copy()).cuda(), t(alb), rough, t(emi), t(dis))
    book, rec = ugp.codebook_encode(t(s.mean), t(s.quat), t(s.scale), t(s.magnitude), mats, iters=2)
    torch.cuda.synchronize()
    codes = rec.cpu().numpy()[:, 16:24].copy().view(np.uint16).astype(np.int64)
    got = {"sggx": codes[:, 2], "material": codes[:, 3] & 0xfff}
    X = {"sggx": t(sggx), "material": torch.cat([t(alb), rough[:, None], t(emi), t(dis)], 1)}
    for g, (o, w) in GROUPS.items():
        ref = _scan(torch, X[g], book[:, o:o + w].contiguous()).cpu().numpy()
        assert np.array_equal(got[g], ref), (g, np.flatnonzero(got[g] != ref)[:5])


@pytest.mark.parametrize("n", [1, 4097, 1_400_000])
def test_entries_are_the_means_of_their_points(ugp, n):
    """Sums of values that fit the words of shared memory, at their limit (512) and beyond, over more points
    than one pass holds: the fixed-point sums are whole numbers, so the entries are equal."""
    import torch
    rng = np.random.Generator(np.random.Philox(n))
    row = rng.normal(size=(300, 22)).astype(np.float32)
    row[:, 10:13] = rng.choice(np.array([-600, -511.99, 0, 300, 511.99, 512, 1e5], np.float32), (300, 3))
    row[:, 0] *= np.where(rng.random(300) < 0.1, np.float32(700), np.float32(1))
    pick = np.where(np.arange(n) < n // 2, np.arange(n) * 100 // max(n, 1), rng.integers(0, 300, n))
    x = row[pick]                                       # runs of equal points, then points in any order
    s = scenes.room_scene(100, seed=1, n_clusters=3).subset(np.arange(100)[:1])
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    rep = lambda a: t(np.repeat(a, n, 0))
    mats = ugp.Materials(t(x[:, :6]), torch.zeros(n, dtype=torch.uint8).cuda(), t(x[:, 6:9]), t(x[:, 9]),
                         t(x[:, 10:13]), t(x[:, 13:22]))
    book, _ = ugp.codebook_encode(rep(s.mean), rep(s.quat), rep(s.scale), rep(s.magnitude), mats, iters=1)
    got = book.cpu().numpy()
    first = x[np.arange(4096, dtype=np.int64) * n // 4096]
    for o, w, c in ((7, 6, 0), (13, 16, 6)):
        code = _scan(torch, t(row[:, c:c + w]), t(first[:, c:c + w])).cpu().numpy()[pick]
        num = np.bincount(code, minlength=4096)
        want = first[:, c:c + w].copy()
        for d in range(w):
            v = np.rint(x[:, c + d] * np.float32(2 ** 24)).astype(np.int64)
            total = np.zeros(4096, np.int64)
            np.add.at(total, code, v)
            want[num > 0, d] = (total[num > 0].astype(np.float64) / (2.0 ** 24 * num[num > 0])).astype(np.float32)
        assert np.array_equal(got[:, o:o + w], want), o
