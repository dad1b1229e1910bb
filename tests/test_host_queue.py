"""What the host code may rely on while the device lags behind it (tests/fake_device.cpp)."""
import pytest

import host_cpp
from paper_1804_04797_gb300 import sv

SOURCES = ['capi.cpp', 'capi_tasks.cpp', 'capi_batch.cpp', 'plan.cpp', 'interp.cpp', 'generator.cpp']


@pytest.fixture(scope='module')
def fake_device(tmp_path_factory):
    return host_cpp.build(tmp_path_factory.mktemp('fake_device'), 'fake_device', SOURCES)


@pytest.mark.parametrize('jit,precision', [(-1, sv.SV_PREC_PLAIN), (1, sv.SV_PREC_PLAIN), (0, sv.SV_PREC_F16X3)])
def test_sources_of_queued_copies_stay_as_they_are(fake_device, jit, precision):
    # (memory that is given back is overwritten at once)
    r = host_cpp.run(fake_device, 'uploads', jit, precision, env={'MALLOC_PERTURB_': '165'})
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize('how,passes', [('support', (0, 3)), ('whole', (0, 2)), ('product', (0, 3))])
def test_a_state_that_was_not_finished_is_reported_by_the_call_that_reads_it(fake_device, how, passes):
    for fail in (-1, *passes):
        r = host_cpp.run(fake_device, 'gave_up', how, fail)
        assert r.returncode == 0, r.stdout + r.stderr


def test_a_segment_s_plan_serves_no_other_call(fake_device):
    r = host_cpp.run(fake_device, 'segments')
    assert r.returncode == 0, r.stdout + r.stderr


def test_a_batch_s_amplitudes_are_read_on_its_device(fake_device):
    r = host_cpp.run(fake_device, 'other_device')
    assert r.returncode == 0, r.stdout + r.stderr


def test_the_tensor_form_runs_where_its_operand_images_find_no_room(fake_device):
    r = host_cpp.run(fake_device, 'no_room')
    assert r.returncode == 0, r.stdout + r.stderr
