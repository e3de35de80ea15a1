"""Scenes of any width, and rays along the axes.

Positions and scales times w = 2^k, directions times l = 2^m and magnitudes times w^2 l leave every optical
depth the same, bit for bit: the tests of the primitives scale exactly, and the boxes only decide which of
them are tested. So transmittances of the scaled scenes equal those of the unit one, for rays along +-x, +-y,
+-z (zero components of either sign), with one zero component and without. Free flights and the radiance field
use absolute slacks of 1e-6 along the ray, so they are compared in scenes that are not small against those: distances
to 1e-5 of the segment of 4, radiances to what a shift of 4e-5 can move (half densities below 10, emissions below 1).
"""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu
N = 1500


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp
    build.build()
    ugp.lib()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    rng = np.random.Generator(np.random.Philox(8))
    s = scenes.tiny_scene(n=700, seed=6)
    d = scenes.unit_vectors(rng, N).astype(np.float32)
    kind = np.arange(N) % 3
    axis = np.arange(N) // 3 % 3
    zero = np.where(rng.random(N) < 0.5, np.float32(0.0), np.float32(-0.0))
    for i in range(N):
        if kind[i] == 0:     # along an axis
            keep = d[i, axis[i]]
            d[i] = zero[i]
            d[i, axis[i]] = np.sign(keep)
        elif kind[i] == 1:   # in a coordinate plane
            d[i, axis[i]] = zero[i]
    through = s.mean[rng.integers(0, s.n, N)] + 0.01 * rng.normal(size=(N, 3))
    o = (through - rng.uniform(0.0, 2.0, (N, 1)) * d).astype(np.float32)
    u, u2 = scenes.uniforms24(3, N), scenes.uniforms24(4, N)
    em = rng.random((s.n, 3)).astype(np.float32)

    def run(k, m=0):
        w, l = np.float32(2.0 ** k), np.float32(2.0 ** m)
        bvh = ugp.build_bvh(t(s.mean * w), t(s.quat), t(s.scale * w), t(s.magnitude * (w * w * l)))
        O, D, a, b = t(o * w), t(d * l), t(np.zeros(N)), t(np.full(N, 4 * w / l))
        T = ugp.trace_transmittance(bvh, O, D, a, b)
        ff = ugp.sample_free_flight(bvh, O, D, a, b, t(u), t(u2))
        rad = ugp.render_radiance_field(bvh, O, D, a, b, t(em), (0.1, 0.2, 0.3))
        torch.cuda.synchronize()
        return [x.cpu().numpy() for x in (*T, *ff, *rad)], float(w / l)

    return run, run(0)[0]


@pytest.mark.parametrize("k,m", [(-20, 0), (18, 0), (21, 0), (22, 0), (30, 0), (0, -30), (0, 20), (22, -4), (22, 15)])
def test_rays_see_the_same_in_scenes_of_any_width(env, k, m):
    run, (T1, st1, prim1, tu1, tsp1, sf1, rgb1, sr1) = env
    (T, st, prim, tu, tsp, sf, rgb, sr), unit = run(k, m)
    assert st.max() == 0 and sf.max() == 0 and sr.max() == 0
    assert (T1 < 1).mean() > 0.9
    assert np.array_equal(T, T1)
    if unit < 1:   # the segment is short against the absolute slacks
        return
    same = prim == prim1
    assert same.mean() >= 0.995   # u within rounding of a boundary between two primitives
    assert np.abs(tu[same].astype(np.float64) / unit - tu1[same]).max() <= 4e-5
    assert np.abs(rgb.astype(np.float64) - rgb1).max() <= 4e-4
