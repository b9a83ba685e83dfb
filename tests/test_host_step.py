"""The packed header functions of the step on the host: tests/host_step.cu
(to_modes, from_modes and moments on pairs, load_force, noise_unit,
one_to_two, DensitySink's pair put, SphereTest)."""
from test_host_headers import _build_and_run


def test_packed_header_functions(tmp_path):
    out = _build_and_run(tmp_path, "host_step", "")
    assert out.split()[-2:] == ["failed", "0"], out
