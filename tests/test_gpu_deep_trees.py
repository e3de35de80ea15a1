"""Trees whose paths need a deep traversal stack.

Primitives whose sizes span decades around one place put one small child beside large ones at every level, so a
ray through that place holds several entries per level: 40 to 80, above the rows that the kernels
keep in shared memory. Every ray must end with status 0, and transmittances and free flights (sums of
integers) give the same bits in calls of few rays, which share deeper stacks among lanes, and in one large
call. Nothing saturates, so no ray ends early. Equal boxes must not make the 4-wide tree deeper than two
binary levels a node.
"""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu
N = 360_000


def _decades(rng, n):
    r = 10.0 ** rng.uniform(-5, 0, n)
    return r[:, None] * scenes.unit_vectors(rng, n), 0.15 * r


def _plume(rng, n):
    y = 10.0 ** rng.uniform(-4, 0, n)
    return np.stack([0.3 * y * rng.normal(size=n), y, 0.3 * y * rng.normal(size=n)], 1), 0.1 * y


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp
    build.build()
    ugp.lib()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    made = {}

    def scene(kind):
        if kind not in made:
            rng = np.random.Generator(np.random.Philox(21))
            mean, size = _decades(rng, 20_000) if kind == "decades" else _plume(rng, 100_000)
            n = len(mean)
            s = size[:, None] * rng.uniform(0.7, 1.3, (n, 3))
            mag = 4 * np.pi * s.prod(1) ** (2 / 3) * rng.uniform(0.5, 1, n) * 10 / n   # all of them together: tau 5
            bvh = ugp.build_bvh(t(mean), t(scenes.random_quaternions(rng, n)), t(s), t(mag))
            d = scenes.unit_vectors(rng, N)
            aim = mean[rng.integers(0, n, N)] * 10.0 ** rng.uniform(-2, 0, (N, 1))
            o = aim - np.where(rng.random((N, 1)) < 0.5, 0.0, rng.uniform(0, 3, (N, 1))) * d
            rays = [t(o), t(d), t(np.zeros(N)), t(np.full(N, 8.0))]
            us = [t(scenes.uniforms24(1, N)), t(scenes.uniforms24(2, N))]
            made[kind] = (bvh, rays, us, t(rng.random((n, 3))),
                          ugp.trace_transmittance(bvh, *rays) + ugp.sample_free_flight(bvh, *rays, *us))
        return made[kind]

    return torch, ugp, t, scene


@pytest.mark.parametrize("kind", ["decades", "plume"])
@pytest.mark.parametrize("n", [500, 4000, 20_000, 100_000, 200_000])
def test_small_and_large_calls_agree(env, kind, n):
    torch, ugp, _, scene = env
    bvh, rays, us, _, full = scene(kind)
    q, v = [x[:n] for x in rays], [x[:n] for x in us]
    part = ugp.trace_transmittance(bvh, *q) + ugp.sample_free_flight(bvh, *q, *v)
    torch.cuda.synchronize()
    assert int(full[1].max()) == 0 and int(full[5].max()) == 0
    assert float(full[0].min()) > 0 and float((full[2] >= 0).float().mean()) > 0.01
    for a, b in zip(part, full):
        assert torch.equal(a, b[:n])


@pytest.mark.parametrize("kind", ["decades", "plume"])
def test_radiance_field_reaches_every_primitive(env, kind):
    """With emission 1 and no background an unsaturated ray sees 1 - T."""
    torch, ugp, _, scene = env
    bvh, rays, _, em, full = scene(kind)
    rgb, st = ugp.render_radiance_field(bvh, *rays, torch.ones_like(em), (0.0, 0.0, 0.0))
    torch.cuda.synchronize()
    assert int(st.max()) == 0
    tau = 1 - full[0].double()[:, None]
    # float32 sums of up to a few thousand terms against the integer sum
    assert bool(((rgb.double() - tau).abs() <= 2e-6 + 1e-4 * tau).all())


@pytest.mark.parametrize("m", [2, 5, 12])
def test_equal_boxes_give_two_levels_a_node(env, m):
    torch, ugp, t, _ = env
    n = 1 << m
    bvh = ugp.build_bvh(t(np.full((n, 3), 0.25)), t(np.tile([1, 0, 0, 0], (n, 1))), t(np.full((n, 3), 0.05)),
                        t(np.full(n, 1e-6)))
    torch.cuda.synchronize()
    ws = bvh.workspace.cpu().numpy()
    up = lambda x: (x + 255) // 256 * 256
    off = up(up(n * 64) + (n - 1) * 64)
    ref = ws[off: off + (n - 1) * 64].view(np.int32).reshape(n - 1, 16)[:, 12:]
    level, depth = [0], 0
    while level:
        depth += 1
        level = [c for i in level for c in ref[i] if c >= 0]
    assert depth == (m + 1) // 2
