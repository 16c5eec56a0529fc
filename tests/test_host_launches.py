"""The library's host code on a CUDA runtime without a device: scratch slots, kernel attributes per device, routes."""
import pytest

from fake_runtime import FakeRuntime

P = 0x7F0000000000      # an address nothing on the host reads


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    f = FakeRuntime(tmp_path_factory.mktemp("fake"))
    f.record_arg("dp_gemm_kernel", 15)                # the slot of cut tiles' parts
    f.record_arg("w4a4_gemm_tc_kernel", 17)           # the first unit of split tiles' parts
    f.record_arg("w4a4_gemm_decode_tc_kernel", 15)    # the slot of cut units' parts
    return f


def linear_dp(fake, n, d_in, d_out, bits_x, bits_w, asym=False):
    z = P if asym else None
    return fake.call("cat_linear_dp", P, bits_x, asym, P, z, P, bits_w, P, z, n, d_in, d_out, P, None, None)


def linear_e8(fake, n, d_in, d_out):
    return fake.call("cat_w4a4_linear_e8", P, P, P, P, n, d_in, d_out, P, None, None)


def linear(fake, n, d_in, d_out):
    return fake.call("cat_w4a4_linear", P, P, P, P, n, d_in, d_out, P, None, None)


def test_launches_in_a_row_have_different_slots_of_scratch(fake):
    """The kernels of a family share one scratch array: the launches that may overlap, whatever their template
    arguments, must not be handed the same slot by counters of their own."""
    cut = [linear_dp(fake, 1000, 14336, 4096, 8, 8), linear_dp(fake, 1000, 14336, 6144, 4, 4),
           linear_dp(fake, 512, 8192, 9980, 4, 8), linear_dp(fake, 300, 6144, 9980, 8, 4, True)]
    split = [linear_e8(fake, 256, 8192, 3000), linear(fake, 256, 8192, 3000), linear_e8(fake, 4096, 14336, 4096),
             linear_e8(fake, 200, 8192, 128)]
    units = [linear(fake, 16, 4096, 28672), linear(fake, 32, 4096, 28672)]
    for calls in (cut, split, units):
        launches = [c[0] for c in calls]
        assert all(len(c) == 1 for c in calls) and all(x.cooperative for x in launches)
        assert len({x.kernel for x in launches}) > 1
        assert all(a.arg != b.arg for a, b in zip(launches, launches[1:])), launches


def test_small_split_launches_share_no_scratch(fake):
    """One split tile takes 16 of the 76 pairs: as many such launches as fit the device, twice, have scratch of their own."""
    launches = [linear_e8(fake, 200, 8192, 128)[0] for _ in range(9)] + [linear(fake, 200, 8192, 128)[0]]
    assert all(x.grid == 32 and x.cooperative for x in launches)
    first = sorted(x.arg for x in launches)
    assert all(b - a >= 16 for a, b in zip(first, first[1:])) and first[-1] + 16 <= 320, first
