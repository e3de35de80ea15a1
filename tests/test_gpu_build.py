"""The BVH build's per-primitive records and its 4-wide nodes.

* The records hold W = S^-1 R^T as two floats and g0 as one. Against float64 (numpy) the first float
  is W to half an ulp, the pair to 2^-46 of its row's 1 / s (float64's own rounding, a few 2^-53 of
  the unit rotation, is far below), g0 to 1.5 ulp. Quaternions come with lengths from 1e-9 to 1e15 and
  scales over 20 decades, where products of the raw values would over- or underflow.
* The binary nodes are the radix tree over the sorted codes, with exact boxes.
* Every primitive is hit by the ray through its centre, whatever the shape of the tree: one, two
  and a few primitives (fewer children than a 4-wide node has), equal centres (ties in the code).
"""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ugp():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp as U
    build.build()
    U.lib()
    return U


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()


@pytest.mark.parametrize("n", [1, 2, 5, 257, 20_000])
def test_records_hold_the_whitening_matrix(ugp, n):
    import torch
    rng = np.random.Generator(np.random.Philox(n))
    q = (scenes.random_quaternions(rng, n) * 10.0 ** rng.uniform(-9, 15, (n, 1))).astype(np.float32)
    s = (10.0 ** rng.uniform(-12, 8, (n, 3))).astype(np.float32)
    mean = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    mag = rng.uniform(0.1, 2.0, n).astype(np.float32)
    bvh = ugp.build_bvh(_dev(mean), _dev(q), _dev(s), _dev(mag))
    torch.cuda.synchronize()
    ws = bvh.workspace.cpu().numpy()
    up = lambda x: (x + 255) // 256 * 256
    ni = max(n - 1, 1)
    off_lo = up(up(up(n * 64) + ni * 64) + ni * 64)
    rec = ws[: n * 64].view(np.float32).reshape(n, 4, 4)
    low = ws[off_lo: off_lo + n * 48].view(np.float32).reshape(n, 3, 4)
    idx = rec[:, 3, 1].copy().view(np.int32)
    assert sorted(idx.tolist()) == list(range(n))
    qd = q[idx].astype(np.float64)
    qd /= np.linalg.norm(qd, axis=1, keepdims=True)
    w, x, y, z = qd.T
    R = np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                  2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                  2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(n, 3, 3)
    sd = s[idx].astype(np.float64)
    W = R.transpose(0, 2, 1) / sd[:, :, None]
    row = 1.0 / sd[:, :, None]
    hi, lo = rec[:, :3, :3].astype(np.float64), low[:, :, :3].astype(np.float64)
    assert (np.abs(hi - W) <= 2.0 ** -24 * np.abs(W) + 2.0 ** -46 * row).all()
    assert (np.abs(hi + lo - W) <= 2.0 ** -46 * row).all()
    g0 = mag[idx].astype(np.float64) / ((2 * np.pi) ** 1.5 * sd.prod(1))
    ok = (g0 > 1e-37) & (g0 < 3e38)   # representable as a normal float
    got = rec[:, 3, 0].astype(np.float64)
    assert (np.abs(got - g0)[ok] <= 1.5 * 2.0 ** -24 * g0[ok]).all()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 9, 33, 1000])
@pytest.mark.parametrize("spread", [0.0, 1.0])
def test_every_primitive_is_reached(ugp, n, spread):
    """The ray through each centre meets exactly the primitives that brute force finds (round ones, so
    that the test is |closest approach| < k s)."""
    import torch
    rng = np.random.Generator(np.random.Philox(100 + n))
    mean = (spread * rng.uniform(0, 1, (n, 3)) + 0.25).astype(np.float32)
    s = np.repeat(rng.uniform(0.01, 0.05, (n, 1)), 3, 1).astype(np.float32)
    q = np.tile(np.array([1, 0, 0, 0], np.float32), (n, 1))
    mag = (1e-4 * rng.uniform(0.5, 1.0, n)).astype(np.float32)
    bvh = ugp.build_bvh(_dev(mean), _dev(q), _dev(s), _dev(mag))
    d = scenes.unit_vectors(rng, n)
    o = (mean - 3.0 * d).astype(np.float32)
    t0, t1 = np.zeros(n, np.float32), np.full(n, 8.0, np.float32)
    T, st = ugp.trace_transmittance(bvh, _dev(o), _dev(d), _dev(t0), _dev(t1))
    _, _, _, cnt, _ = ugp.collect_hits(bvh, _dev(o), _dev(d), _dev(t0), _dev(t1), 0)
    torch.cuda.synchronize()
    assert int(st.max()) == 0
    p = o.astype(np.float64)[:, None] - mean.astype(np.float64)[None]
    dd = d.astype(np.float64)[:, None]
    u = dd / np.linalg.norm(dd, axis=2, keepdims=True)
    c = p - (p * u).sum(2, keepdims=True) * u
    d2 = (c * c).sum(2) / s[None, :, 0].astype(np.float64) ** 2
    k2 = -2 * np.log(0.01)
    # 1/2 I of a round Gaussian over its chord, g0 s sqrt(pi/2) e^{-d2/2} erf(sqrt((k2 - d2) / 2)), per unit of |d|
    from scipy.special import erf
    g0 = mag.astype(np.float64) / ((2 * np.pi) ** 1.5 * s.astype(np.float64).prod(1))
    v = np.where(d2 < k2, g0 * s[:, 0] * np.sqrt(np.pi / 2) * np.exp(-0.5 * d2)
                 * erf(np.sqrt(np.maximum(k2 - d2, 0) / 2)), 0.0) / np.linalg.norm(dd, axis=2)
    ref = np.maximum(0.0, 1.0 - v.sum(1))
    assert np.abs(T.cpu().numpy() - ref).max() <= 1e-5
    edge = np.abs(d2 - k2) < 1e-3
    assert (np.abs(cnt.cpu().numpy() - (d2 < k2).sum(1)) <= edge.sum(1)).all()


@pytest.mark.parametrize("n", [2, 3, 128, 255, 256, 257, 512, 513, 4096, 4097, 30_011])
@pytest.mark.parametrize("kind", ["spread", "ties"])
def test_nodes_are_the_radix_tree_and_its_boxes(ugp, n, kind):
    """The binary nodes equal the radix tree over (code, position), split at the highest differing bit and
    numbered by the end of the leaves nearest the sibling; every box is the exact union of its leaves'."""
    import torch
    rng = np.random.Generator(np.random.Philox(n + (kind == "ties")))
    mean = rng.uniform(-1, 1, (n, 3)).astype(np.float32)
    if kind == "ties":   # a few positions, runs of equal codes longer than a block among them
        mean = mean[np.minimum(rng.integers(0, 40, n), rng.integers(0, 40, n)) % n]
    s = rng.uniform(0.01, 0.05, (n, 3)).astype(np.float32)
    bvh = ugp.build_bvh(_dev(mean), _dev(scenes.random_quaternions(rng, n)), _dev(s), _dev(np.ones(n)))
    torch.cuda.synchronize()
    ws = bvh.workspace.cpu().numpy()
    up = lambda x: (x + 255) // 256 * 256
    rec = ws[: n * 64].view(np.float32).reshape(n, 4, 4)
    node = ws[up(n * 64): up(n * 64) + (n - 1) * 64].view(np.float32).reshape(n - 1, 16)
    child = node.view(np.int32)[:, 12:14]
    assert (node[:, 14:] == 0).all()
    leaf = np.zeros((n, 6), np.float32)
    boxes = node[:, :12].reshape(-1, 6)
    is_leaf = child.reshape(-1) < 0
    assert sorted((~child.reshape(-1)[is_leaf]).tolist()) == list(range(n))
    leaf[~child.reshape(-1)[is_leaf]] = boxes[is_leaf]
    # codes of the leaves in order, from their boxes' centres between the means' extremes
    lo, hi = mean.min(0), mean.max(0)
    c = np.float32(0.5) * (leaf[:, :3] + leaf[:, 3:])
    ext = hi - lo
    t = np.where(ext > 0, (c - lo) / np.where(ext > 0, ext, 1), np.float32(0.5)).astype(np.float32)
    t = np.clip(t * np.float32(1024), 0, 1023).astype(np.uint64)
    code = np.zeros(n, np.uint64)
    for b in range(10):
        for a in range(3):
            code |= ((t[:, a] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + 2 - a)
    assert (np.diff(code.astype(np.int64)) >= 0).all()
    key = [int(x) << 32 | i for i, x in enumerate(code)]
    arr = np.array(key, np.uint64)
    todo = [(0, 0, n - 1)]
    seen = 0
    while todo:
        i, l, r = todo.pop()
        seen += 1
        h = (key[l] ^ key[r]).bit_length() - 1
        g = int(np.searchsorted(arr, np.uint64(key[r] >> h << h))) - 1
        assert child[i].tolist() == [~g if l == g else g, ~(g + 1) if r == g + 1 else g + 1], (i, l, r)
        for side, (p, q) in enumerate(((l, g), (g + 1, r))):
            box = np.concatenate([leaf[p:q + 1, :3].min(0), leaf[p:q + 1, 3:].max(0)])
            assert np.array_equal(node[i, 6 * side:6 * side + 6], box), (i, side)
            if p < q:
                todo.append(((g, g + 1)[side], p, q))
    assert seen == n - 1
    idx = rec[:, 3, 1].copy().view(np.int32)
    for k in np.flatnonzero(np.diff(code.astype(np.int64)) == 0):   # equal codes keep the arrays' order
        assert idx[k] < idx[k + 1]
