"""The host side of the network's kernels when a launch fails, and on a second device."""
import pytest

from tests.fake_runtime import LAUNCH_ERROR, load

ENTRY = r"""
int fake_train(unsigned W, unsigned H) {
  rt::nn::TrainBuffers t = {};
  size_t i = 0;
  t.params = (float*)at(i++); t.m = (float*)at(i++); t.v = (float*)at(i++);
  for (int l = 0; l < 4; ++l) { t.wf[l] = (__nv_bfloat16*)at(i++); t.wb[l] = (__nv_bfloat16*)at(i++); }
  for (int l = 0; l < 3; ++l) { t.act[l] = (__nv_bfloat16*)at(i++); t.dz[l] = (__nv_bfloat16*)at(i++); }
  t.g8 = (__nv_bfloat16*)at(i++); t.mask = (uint32_t*)at(i++);
  t.wpart = (float*)at(i++); t.loss_part = (float*)at(i++); t.loss = (float*)at(i++);
  return rt::nn::train_step((__nv_bfloat16*)at(i), (float*)at(i + 1), t, W, H, 1e-3f, 1u, nullptr, (uint32_t*)at(i + 2), 0);
}
int fake_forward(int fp8, unsigned W, unsigned H) {
  __nv_bfloat16* wf[4];
  uint8_t* w8[3];
  float* inv[3];
  const float scale[3] = {1.f, 1.f, 1.f};
  for (int l = 0; l < 4; ++l) wf[l] = (__nv_bfloat16*)at(l);
  for (int l = 0; l < 3; ++l) { w8[l] = (uint8_t*)at(4 + l); inv[l] = (float*)at(7 + l); }
  __nv_bfloat16* feat = (__nv_bfloat16*)at(10);
  float *params = (float*)at(11), *prob = (float*)at(12);
  uint32_t* err = (uint32_t*)at(13);
  if (fp8) return rt::nn::forward_fp8(feat, params, wf, w8, inv, scale, prob, W, H, err, 0, 1);
  return rt::nn::forward(feat, params, wf, nullptr, prob, W, H, err, 0, 1);
}
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return load(tmp_path_factory.mktemp("fake"), ["nn.o", "trace.o"], ENTRY)


@pytest.mark.parametrize("W,H", [(960, 540), (33, 9)])
def test_a_step_ends_at_its_first_failed_launch(fake, W, H):
    fake.fake_begin(0, -1)
    assert fake.fake_train(W, H) == 0
    steps = fake.fake_launches()
    assert steps == 4
    for at in range(steps):
        fake.fake_begin(0, at)
        assert fake.fake_train(W, H) == LAUNCH_ERROR
        assert fake.fake_launches() == at + 1, "a kernel was launched on what the failed one did not make"
        fake.fake_begin(0, -1)
        assert fake.fake_train(W, H) == 0, "the failure is reported once"


@pytest.mark.parametrize("W,H", [(960, 540), (33, 9)])     # either weight-gradient kernel
def test_a_second_device_allows_the_shared_memory_too(fake, W, H):
    for device in (0, 1, 0, 2):
        fake.fake_begin(device, -1)
        assert fake.fake_forward(0, W, H) == 0, device
        assert fake.fake_forward(1, W, H) == 0, device
        assert fake.fake_train(W, H) == 0, device
