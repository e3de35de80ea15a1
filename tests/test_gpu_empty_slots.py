"""Nodes with empty child slots, seen from far away.

The node test allows for rounding by 4e-7 of the distance. A ray enters any box of a node smaller than that, and
an empty slot must still count as a miss. One to six
primitives around the origin, rays along (1, 1, 1) from 7.9 units away in each coordinate (exactly through the
origin), against float64: primitives of 3e-7 are smaller than the allowance and still longer than the spacing of
floats at 7.9 (4.8e-7), those of 1e-7 are not, and only end with status 0.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 5, 6])
@pytest.mark.parametrize("size", [1e-7, 3e-7, 1e-2])
@pytest.mark.parametrize("rays", [5, 400_000])   # a group of lanes per ray, a lane each
def test_tiny_primitives_are_seen_from_afar(n, size, rays):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from scipy.special import erf
    from paper_2406_09733_gb300 import build, ugp
    build.build()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    rng = np.random.Generator(np.random.Philox(n))
    mean = (size * rng.uniform(-1, 1, (n, 3))).astype(np.float32)
    s = np.full((n, 3), size, np.float32)
    mag = (size * size * rng.uniform(0.1, 0.9, n)).astype(np.float32)
    bvh = ugp.build_bvh(t(mean), t(np.tile([1, 0, 0, 0], (n, 1))), t(s), t(mag))
    o, d = t(np.full((rays, 3), -7.9)), t(np.ones((rays, 3)))
    t0, t1 = t(np.zeros(rays)), t(np.full(rays, 20.0))
    T, st = ugp.trace_transmittance(bvh, o, d, t0, t1)
    u = t(np.linspace(0, 1, rays, endpoint=False))
    prim, _, _, sf = ugp.sample_free_flight(bvh, o, d, t0, t1, u, u)
    rgb, sr = ugp.render_radiance_field(bvh, o, d, t0, t1, t(np.ones((n, 3))), (0.0, 0.0, 0.0))
    torch.cuda.synchronize()
    assert int(st.max()) == 0 and int(sf.max()) == 0 and int(sr.max()) == 0
    if size < 2e-7:
        return
    # 1/2 I of a round Gaussian over its chord, per unit of |d|
    m, w = mean.astype(np.float64), float(s[0, 0])
    c = m - m.sum(1, keepdims=True) / 3
    d2, k2 = (c * c).sum(1) / w ** 2, -2 * np.log(0.01)
    g0 = mag.astype(np.float64) / ((2 * np.pi) ** 1.5 * w ** 3)
    tau = (g0 * w * np.sqrt(np.pi / 2) * np.exp(-0.5 * d2) * erf(np.sqrt((k2 - d2) / 2)) / np.sqrt(3)).sum()
    assert 0 < tau < 1
    assert float((T.double() - (1 - tau)).abs().max()) <= 1e-5
    assert float((rgb.double() - tau).abs().max()) <= 1e-5
    if size > 1e-3:
        assert abs(float((prim >= 0).double().mean()) - tau) <= 1.0 / rays + 1e-5
