"""Scenes of few primitives take the kernels with a lane per ray from fewer rays on. At the edges of that rule (600 rays
a primitive for transmittances, 12,000 and 250 a primitive for free flights) the results keep their bits."""
import numpy as np
import pytest

from paper_2406_09733_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 8, 64, 300])
def test_results_keep_their_bits_at_the_edges(p):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_09733_gb300 import build, ugp
    build.build()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    s = scenes.tiny_scene(max(p, 2), seed=p).subset(np.arange(p))
    bvh = ugp.build_bvh(t(s.mean), t(s.quat), t(s.scale), t(s.magnitude))
    N = 360_000
    r = scenes.random_rays(N, seed=12)
    rays, us = [t(r.o), t(r.d), t(r.t0), t(r.t1)], [t(scenes.uniforms24(1, N)), t(scenes.uniforms24(2, N))]
    T, ff = ugp.trace_transmittance(bvh, *rays), ugp.sample_free_flight(bvh, *rays, *us)
    for n in (600 * p, 600 * p + 1, 12_000 + 250 * p, 12_001 + 250 * p):
        q, v = [x[:n].contiguous() for x in rays], [x[:n].contiguous() for x in us]
        got = ugp.trace_transmittance(bvh, *q) + ugp.sample_free_flight(bvh, *q, *v)
        torch.cuda.synchronize()
        for a, b in zip(got, T + ff):
            assert torch.equal(a, b[:n]), n
    assert int(T[1].max()) == 0 and int(ff[3].max()) == 0
