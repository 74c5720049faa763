"""Builds and renders when a launch fails: no later kernel runs on what the failed one
did not write (it would index by keys, jobs or counters that are not there), the error is
returned, and returned once."""
import pytest

from tests.fake_runtime import LAUNCH_ERROR, load

ENTRY = r"""
// The download of the SAH build's control words says: no node left, `mid` subtrees.
int fake_lbvh(unsigned n) {
  return rt::build_lbvh((float4*)at(0), (float*)at(1), 0, n, (float4*)at(2), (float4*)at(3), (uint64_t*)at(4),
                        (int32_t*)at(5), at(6), ~(size_t)0, (uint32_t*)at(7), 0);
}
int fake_sah(unsigned n, unsigned mid) {
  for (unsigned& w : g_word) w = 0;
  g_word[4] = mid;
  return rt::build_sah_tree((float4*)at(0), (int32_t*)at(1), n, (float4*)at(2), at(3), (uint32_t*)at(4), 0);
}
int fake_render(int tiles, int counts) {
  rt::Workspace ws;
  ws.accum = (uint32_t*)at(0); ws.wq = (float4*)at(1); ws.pool = (float4*)at(2); ws.pool_flag = (uint32_t*)at(3);
  ws.counters = (uint32_t*)at(4);
  ws.cap_p = 1024; ws.cap_s = 64; ws.cap_r = 64; ws.n_warps = 1u << 20;
  rt::RenderArgs a = {};
  a.cam.W = 8 * tiles; a.cam.H = a.cam.rows = 4; a.cam.tiles_x = tiles; a.cam.tiles_y = 1;
  a.sc.n_prims = 10; a.sc.n_lights = 1; a.color_scale = 1.f; a.eyes = 3u; a.resolve = true;
  a.out_L = (float*)at(5); a.out_R = (float*)at(6);
  a.ray_counts = counts ? (uint64_t*)at(7) : nullptr;
  return rt::render(a, ws, 0);
}
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return load(tmp_path_factory.mktemp("fake"), ["lbvh.o", "sah.o", "trace.o"], ENTRY)


@pytest.mark.parametrize("call", [("fake_lbvh", 1), ("fake_lbvh", 200), ("fake_lbvh", 5000), ("fake_lbvh", 3_000_000),
                                  ("fake_sah", 100, 1), ("fake_sah", 300, 2), ("fake_sah", 100_000, 700),
                                  ("fake_render", 3, 1), ("fake_render", 100_000, 0)], ids=str)
def test_a_chain_ends_at_its_first_failed_launch(fake, call):
    run = getattr(fake, call[0])
    fake.fake_begin(0, -1)
    assert run(*call[1:]) == 0
    launches = fake.fake_launches()
    assert launches >= 2
    for at in range(launches):
        fake.fake_begin(0, at)
        assert run(*call[1:]) == LAUNCH_ERROR, at
        assert fake.fake_launches() == at + 1, "a kernel was launched on what the failed one did not make"
        fake.fake_begin(0, -1)
        assert run(*call[1:]) == 0, "the failure is reported once"
