"""A radiance-field ray gives the same bits whichever rays share its call.

One call of 120,001 rays against calls of its first n rays and against the same rays in another order, on a room
(most rays saturate) and on a few thousand primitives (few do).
"""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu
N = 120_001


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp
    build.build()
    ugp.lib()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    r = scenes.random_rays(N, seed=31)
    rays = [t(r.o), t(r.d), t(r.t0), t(r.t1)]
    made = {}

    def scene(kind):
        if kind not in made:
            s = scenes.room_scene(20_000, seed=4, n_clusters=6) if kind == "room" else scenes.tiny_scene(3000, seed=5)
            bvh = ugp.build_bvh(t(s.mean), t(s.quat), t(s.scale), t(s.magnitude))
            em = t(np.random.default_rng(6).uniform(0, 3, (s.n, 3)))
            made[kind] = (bvh, em, ugp.render_radiance_field(bvh, *rays, em, (0.2, 0.5, 0.9)))
        return made[kind]

    return torch, ugp, rays, scene


@pytest.mark.parametrize("kind", ["room", "tiny"])
@pytest.mark.parametrize("n", [1, 33, 4863, 4865, 30_400, 100_000])
def test_first_rays_alone_give_the_same_bits(env, kind, n):
    torch, ugp, rays, scene = env
    bvh, em, (rgb, st) = scene(kind)
    a, b = ugp.render_radiance_field(bvh, *[x[:n].contiguous() for x in rays], em, (0.2, 0.5, 0.9))
    torch.cuda.synchronize()
    assert torch.equal(a, rgb[:n]) and torch.equal(b, st[:n]) and int(st.max()) == 0


@pytest.mark.parametrize("kind", ["room", "tiny"])
def test_order_of_the_rays_does_not_matter(env, kind):
    torch, ugp, rays, scene = env
    bvh, em, (rgb, st) = scene(kind)
    p = torch.randperm(N, generator=torch.Generator().manual_seed(7)).cuda()
    a, _ = ugp.render_radiance_field(bvh, *[x[p].contiguous() for x in rays], em, (0.2, 0.5, 0.9))
    torch.cuda.synchronize()
    assert torch.equal(a, rgb[p])
