"""The error bound of the codebook search's product.

The product of BF16 pieces must not be off by more than the search allows for, or an entry that wins by d2 is not
among the candidates. The parts of the bound, each relative to |x||c| (Cauchy, dimension by dimension) or
to |x||c| + |c|^2 / 2: the products of pieces that are left out, formed here for values over a binade (the
worst lies at 1.01173); the additions in the accumulator, 2^-22 each; the rounding of the two
moved coordinates, 2^-24 each and their product; that of |c|^2 / 2, D + 1 roundings and its third piece.
"""
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _bf16(v):
    """Nearest BF16 value, ties to even, of float32 values."""
    b = np.asarray(v, np.float32).view(np.uint32).astype(np.uint64)
    return ((b + 0x7fff + ((b >> 16) & 1)) >> 16 << 16).astype(np.uint32).view(np.float32)


def _pieces(v):
    h = _bf16(v)
    m = _bf16(v - h)
    return [p.astype(np.float64) for p in (h, m, _bf16(v - h - m))]


def _left_out(terms):
    v = np.concatenate([np.linspace(1, 2, 1500, endpoint=False), [1.01173], 1.01173 + np.arange(-60, 60) * 2.0 ** -20])
    v = v.astype(np.float32)
    x, c = _pieces(v), _pieces(v)
    kept = [(0, 0), (0, 1), (1, 0)] + ([(1, 1), (0, 2), (2, 0)] if terms == 6 else [])
    got = sum(np.multiply.outer(x[i], c[j]) for i, j in kept)
    exact = np.multiply.outer(v.astype(np.float64), v.astype(np.float64))
    return np.abs(got / exact - 1).max()


@pytest.mark.parametrize("D", [3, 4, 6, 16])
def test_bound_covers_its_parts(D):
    src = open(os.path.join(ROOT, "paper_2406_09733_gb300", "csrc", "ugp_nearest.cuh")).read()
    few, many = re.search(r"kErr = D <= 6 \? ([\d.e+-]+)f : ([\d.e+-]+)f", src).groups()
    terms = 6 if D <= 6 else 3
    need = _left_out(terms) + (D * terms + 3) * 2.0 ** -22 + 3 * 2.0 ** -24 + (D + 2) * 2.0 ** -24
    assert float(few if D <= 6 else many) >= need


@pytest.mark.gpu
@pytest.mark.parametrize("far", [1.0, 64.0, 4096.0])
def test_codes_of_the_worst_mantissas(far):
    """Entries a few ulps apart whose coordinates have the worst mantissa, in one dimension or in all, seen from
    points of the same directions, near and far: the codes are those of the FP32 scan."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, scenes, ugp
    from test_gpu_nearest import _scan
    build.build()
    rng = np.random.Generator(np.random.Philox(int(far)))
    n = 8192
    c = np.full((n, 16), 1.01173, np.float32) + rng.integers(-8, 9, (n, 16)).astype(np.float32) * np.float32(2.0 ** -23)
    c *= np.where(rng.random((n, 1)) < 0.5, np.float32(1), np.float32(-1))
    c[n // 2:, :4] *= np.float32(2.0 ** -12)     # half of them: the other dimensions, one in ten a single one
    c[n // 2:, 5:] *= np.where(rng.random((n - n // 2, 1)) < 0.2, np.float32(2.0 ** -12), np.float32(1))
    c[1::2] *= np.float32(far)                   # even rows are the starting entries, odd ones are looked up
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    s = scenes.tiny_scene(n=n, seed=1)
    X = t(c)
    mats = ugp.Materials(t(s.sggx), torch.zeros(n, dtype=torch.uint8).cuda(), X[:, :3].contiguous(),
                         X[:, 3].contiguous(), X[:, 4:7].contiguous(), X[:, 7:].contiguous())
    book, rec = ugp.codebook_encode(t(s.mean), t(s.quat), t(s.scale), t(s.magnitude), mats, iters=0)
    torch.cuda.synchronize()
    got = rec.cpu().numpy()[:, 16:24].copy().view(np.uint16)[:, 3].astype(np.int64) & 0xfff
    ref = _scan(torch, X, book[:, 13:29].contiguous()).cpu().numpy()
    assert np.array_equal(got, ref)
