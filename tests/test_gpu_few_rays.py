"""A ray's result does not depend on how many rays its call has.

Calls of few rays give each ray a group of lanes (2 to 5 powers of two, by the count), larger ones a lane each;
transmittances and free flights are sums of integers, so the same ray must give the same bits. One call
of 360,000 rays (a lane each) against calls of its first n rays, n at the edges of warps and of the group
sizes' ranges, on a room, on a few primitives, and on a heap of dense primitives whose shares exceed the
bins (the large-share path of the grouped scan) and whose rays cross hundreds of them.
"""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu
N = 360_000
SIZES = [1, 2, 31, 33, 1000, 4863, 4865, 9120, 9121, 12_161, 30_400, 30_401, 76_001, 77_825, 182_400, 182_401, 350_208,
         350_209]


def _heap(n):
    """Dense primitives around one point: interval masses from 10^-6 to 100."""
    rng = np.random.Generator(np.random.Philox(5))
    s = scenes.tiny_scene(n=n, seed=3)
    s.mean[:] = (0.5 + 0.05 * rng.normal(size=(n, 3))).astype(np.float32)
    s.magnitude[:] = (s.magnitude * 10.0 ** rng.uniform(-4, 4, n)).astype(np.float32)
    return s


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp
    build.build()
    ugp.lib()
    r = scenes.random_rays(N, seed=11)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    rays = dict(o=t(r.o), d=t(r.d), t0=t(r.t0), t1=t(r.t1), u=t(scenes.uniforms24(1, N)), u2=t(scenes.uniforms24(2, N)),
                ex=torch.arange(N, dtype=torch.int32, device="cuda") % 7 - 1)
    made = {}

    def scene(kind):
        if kind not in made:
            s = {"room": lambda: scenes.room_scene(20_000, seed=4, n_clusters=6), "three": lambda: scenes.tiny_scene(3),
                 "heap": lambda: _heap(600)}[kind]()
            bvh = ugp.build_bvh(t(s.mean), t(s.quat), t(s.scale), t(s.magnitude))
            q = rays
            full = (ugp.trace_transmittance(bvh, q["o"], q["d"], q["t0"], q["t1"], exclude=q["ex"]),
                    ugp.sample_free_flight(bvh, q["o"], q["d"], q["t0"], q["t1"], q["u"], q["u2"], exclude=q["ex"]))
            made[kind] = (bvh, full)
        return made[kind]
    return torch, ugp, rays, scene


@pytest.mark.parametrize("kind", ["room", "three", "heap"])
@pytest.mark.parametrize("n", SIZES)
def test_first_rays_alone_give_the_same_bits(env, kind, n):
    torch, ugp, rays, scene = env
    bvh, (T_full, ff_full) = scene(kind)
    q = {k: v[:n].contiguous() for k, v in rays.items()}
    T = ugp.trace_transmittance(bvh, q["o"], q["d"], q["t0"], q["t1"], exclude=q["ex"])
    ff = ugp.sample_free_flight(bvh, q["o"], q["d"], q["t0"], q["t1"], q["u"], q["u2"], exclude=q["ex"])
    torch.cuda.synchronize()
    for a, b in zip(T + ff, T_full + ff_full):
        assert torch.equal(a, b[:n])
    assert int(ff[3].max()) == 0 and int(T[1].max()) == 0
