"""The library's host code on a CUDA runtime without a device: scratch slots, kernel attributes per device, routes."""
import ctypes

import numpy as np
import pytest

from fake_runtime import FakeRuntime

P = 0x10 << 40          # an address that holds nothing


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    f = FakeRuntime(tmp_path_factory.mktemp("fake"))
    f.record_arg("dp_gemm_kernel", 14)                # the slot of cut tiles' parts
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


def entry_calls(fake):
    """One call, at least, of every kernel that needs an attribute of its own: shared memory or a wide cluster."""
    blocks = fake.buffer(8 * 512 * 128)
    for dtype in (0, 1):
        for n, d, k in ((1, 64, 64), (16, 4096, 128), (32, 4096, 32), (3, 4096, 256), (100, 256, 32), (100, 4096, 128),
                        (300, 4096, 256), (9000, 4096, 128), (2600, 192, 64), (40, 20480, 128), (9000, 8192, 256)):
            yield "cat_transform_quantize_act", P, dtype, n, d, k, P, P, P, None
            yield "cat_transform_quantize_act_dp", P, dtype, n, d, k, P, 8, 1, P, P, P, None
            yield "cat_transform_quantize_act_dp", P, dtype, n, d, k, P, 8, 0, P, P, None, None
        for n, d, k in ((512, 4096, 128), (512, 512, 256), (20000, 4096, 128), (3000, 256, 64), (9000, 512, 256)):
            yield "cat_calib_cov", P, dtype, n, d, k, P, 0, None
        yield "cat_block_row_stats", P, dtype, 100, 512, 128, P, 0, P, P, P, None
        yield "cat_quantize_weights", P, dtype, 300, 512, 128, 2, blocks, 512, None, blocks, P, P, None
        yield "cat_quantize_weights_dp", P, dtype, 300, 512, 128, 2, blocks, 512, None, 8, 1, blocks, P, P, P, None
    yield "cat_fwht_rows", P, 10, 32768, None
    for n, d_in, d_out in ((1, 4096, 6144), (32, 4096, 28672), (16, 4096, 28672), (27, 14336, 4096), (32, 32768, 260),
                           (201, 4096, 6144), (200, 8192, 128), (2048, 4096, 6144)):
        yield "cat_w4a4_linear", P, P, P, P, n, d_in, d_out, P, None, None
    for n, d_in, d_out in ((2048, 4096, 6144), (256, 8192, 1000), (256, 8192, 3000), (200, 8192, 128), (1100, 4096, 5312)):
        yield "cat_w4a4_linear_e8", P, P, P, P, n, d_in, d_out, P, None, None
        yield "cat_w4a4_linear_sqnr_e8", P, P, P, P, n, d_in, d_out, P, P, P, None
    for bits_x, bits_w in ((4, 4), (8, 4), (4, 8), (8, 8)):
        for n, d_in, d_out in ((1, 4096, 64), (2048, 4096, 6144), (1000, 14336, 4096), (1000, 14336, 6144), (512, 8192, 9980)):
            yield "cat_linear_dp", P, bits_x, 0, P, None, P, bits_w, P, None, n, d_in, d_out, P, None, None


def test_every_kernel_is_allowed_its_launch_on_every_device(fake):
    """Shared memory beyond 48 KB and clusters of 16 are allowed per device: what one device was asked does not hold for
    another, so the same calls are launched the same way on two devices of a process."""
    first, second = [], []
    for found, device in ((first, 3), (second, 5)):
        fake.device(device)
        for name, *args in entry_calls(fake):
            found += fake.call(name, *args)
    fake.device(0)
    assert {x.device for x in first} == {3} and {x.device for x in second} == {5}
    same = [x._replace(device=0, arg=0) for x in first]
    assert same == [x._replace(device=0, arg=0) for x in second]
    assert any(x.cluster == 16 for x in first) and sum(x.smem > 48 * 1024 for x in first) > 50


def transform_kernel(fake, n, d, k, dtype, code_bytes):
    name, planes = ("cat_transform_quantize_act_e8", (None,)) if code_bytes else ("cat_transform_quantize_act", ())
    launches = fake.call(name, P, dtype, n, d, k, P, *planes, P, P, None)
    return next(name for name in ("few", "rows", "tc_fused", "tc", "") if f"transform_quant_{name}_kernel".replace("__", "_")
                in launches[0].kernel)


@pytest.mark.parametrize("code_bytes", [False, True])
@pytest.mark.parametrize("k,whole,tiled", [
    (16, [(5, 64), (512, 384), (65536, 384)], [(33, 416), (512, 3072), (65536, 1024), (5, 3072)]),
    (32, [(100, 32), (512, 256), (65536, 576), (2432, 768)], [(2433, 768), (100, 800), (512, 2048)]),
    (64, [(40, 64), (65536, 512), (2432, 640)], [(2433, 640), (100, 704), (512, 1024)]),
    (128, [(40, 128), (512, 512), (14592, 128), (7296, 256), (4864, 384), (2432, 512)],
     [(14593, 128), (7297, 256), (4865, 384), (2433, 512), (33, 640)]),
    (256, [(33, 256), (65536, 256)], [(33, 512)]),
])
def test_small_transforms_take_whole_rows_where_that_is_faster(fake, k, whole, tiled, code_bytes):
    """float32 rows (few rows of k >= 32 have a kernel of their own): blocks and rows at the rule's lines, both code forms."""
    for n, d in whole:
        assert transform_kernel(fake, n, d, k, 0, code_bytes) == "rows", (n, d)
    for n, d in tiled:
        assert transform_kernel(fake, n, d, k, 0, code_bytes) == "", (n, d)


def decode_route(fake, n, d_in, d_out, sums):
    """What n <= 32 tokens run on: whole units, a cluster of 2, 4 or 8 a unit, equal cuts, or mma.sync ("+": and the
    SQNR sums in a launch of their own)."""
    launches = (fake.call("cat_w4a4_linear_sqnr", P, P, P, P, n, d_in, d_out, P, P, P, None) if sums else
                linear(fake, n, d_in, d_out))
    first = launches[0]
    form = "mma" if "gemm_decode_kernel" in first.kernel else "cut" if first.cooperative else str(first.cluster)
    return form + "+" * (len(launches) - 1)


@pytest.mark.parametrize("n,d_in,d_out,plain,sums", [
    (1, 4096, 6144, "2", "2"), (16, 4096, 14336, "1", "1"), (27, 14336, 4096, "4", "4"), (16, 1024, 24001, "cut", "cut"),
    (16, 2048, 7530, "1", "1"), (30, 864, 4096, "1", "1"), (16, 4096, 1024, "8", "8"), (32, 256, 64, "1", "1"),
    (9, 32, 20000, "cut", "cut"), (16, 14336, 16384, "2", "2+"),
    # rows too long for one CTA: mma.sync for up to 8 tokens and many units, for 17 to 24 past a cluster of 4
    (2, 14336, 22016, "mma", "mma+"), (8, 10240, 28672, "mma", "mma+"), (9, 14336, 22016, "2", "2+"), (2, 14336, 1024, "8", "8"),
    (32, 20480, 28672, "8", "8+"), (24, 20480, 8192, "mma", "mma+"), (32, 28672, 4096, "8", "8+"), (24, 5120, 2048, "mma", "4"),
    (16, 100000, 4096, "mma", "mma+"), (32, 49152, 1024, "mma", "mma+"),
])
def test_decode_gemm_takes_the_fastest_form(fake, n, d_in, d_out, plain, sums):
    """The split that was measured fastest, on 152 SMs with 76, 36 and 15 clusters of 2, 4 and 8 resident."""
    assert (decode_route(fake, n, d_in, d_out, False), decode_route(fake, n, d_in, d_out, True)) == (plain, sums)


@pytest.mark.parametrize("n,d_in,d_out,width,grid,split", [
    (2048, 4096, 6144, 224, 152, False), (4096, 14336, 4096, 256, 152, True), (8192, 8192, 28672, 256, 152, True),
    (256, 8192, 3000, 192, 128, True), (600, 4096, 15000, 224, 152, False),
    # one partial wave of long rows: many wide parts in two are no use, in four they are
    (3000, 12640, 768, 128, 144, False), (1000, 12640, 2048, 128, 128, False), (1000, 14336, 768, 192, 128, True),
    (5978, 14336, 2048, 256, 152, False),
])
def test_byte_code_gemm_takes_the_fastest_tiles(fake, n, d_in, d_out, width, grid, split):
    """The tile width and whether the last wave is split along K, as measured, on 76 pairs."""
    launch, = linear_e8(fake, n, d_in, d_out)
    assert f"w4a4_gemm_tc_kernel<true, {width}>" in launch.kernel
    assert (launch.grid, launch.cooperative) == (grid, int(split))


@pytest.mark.parametrize("n,rows", [(1, 8), (8, 8), (9, 16), (64, 64), (121, 128), (127, 128), (128, 128), (300, 128)])
def test_digit_plane_gemm_loads_the_token_rows_there_are(fake, n, rows):
    """Boxes of as many token rows as there are in whole swizzle atoms, never more than a CTA's 128."""
    for bits_x, bits_w in ((4, 4), (8, 4), (4, 8), (8, 8)):
        linear_dp(fake, n, 4096, 6144, bits_x, bits_w)
        assert fake.box_rows()[:2] == [32, rows]                  # y's, then the tokens'


@pytest.mark.parametrize("d,k,device", [(112, 16, False), (128, 16, True), (128, 32, False), (160, 32, True), (64, 64, True),
                                        (128, 128, True), (512, 256, False)])
def test_transforms_of_a_few_small_blocks_are_built_on_the_host(fake, d, k, device):
    """Fewer than 8 blocks of 16 or 5 of 32 channels take longer on the device than on the host's cores."""
    sigma = np.tile(np.eye(k), (d // k, 1, 1)).astype(np.float64)
    sx, T = fake.buffer(sigma.nbytes), fake.buffer(d * k * 4)
    ctypes.memmove(sx, sigma.ctypes.data, sigma.nbytes)
    fake.lib.fake_reset()
    fake.lib.cat_quantize_weights(P, 0, 300, d, k, 2, sx, 512, None, T, P, P, None)   # (no kernel ran: Sigma_w is 0)
    kernels = [fake.lib.fake_kernel(i).decode() for i in range(fake.lib.fake_launches())]
    assert any("jacobi_kernel" in name for name in kernels) == device


@pytest.mark.parametrize("n,d_in,d_out,bits_x,bits_w,lanes", [
    (300, 3072, 4990, 8, 8, 2), (2500, 6144, 1030, 8, 8, 1), (1500, 6144, 3396, 6, 8, 1), (1000, 6144, 4990, 8, 6, 4),
    (300, 6144, 9980, 8, 4, 2), (512, 8192, 9980, 4, 4, 2), (300, 8192, 9980, 4, 4, 2), (512, 8192, 9980, 4, 8, 2),
    (1000, 8192, 6144, 4, 8, 4),
])
def test_digit_plane_gemm_cuts_its_last_waves(fake, n, d_in, d_out, bits_x, bits_w, lanes):
    """The shapes whose accumulators are checked for cut tiles take that path, with every kind of operand: in columns of
    all token tiles or tile by tile."""
    fake.record_arg("dp_gemm_kernel", 13)
    launch, = linear_dp(fake, n, d_in, d_out, bits_x, bits_w)
    fake.record_arg("dp_gemm_kernel", 14)
    planes = tuple(1 if b <= 4 else 2 for b in (bits_x, bits_w))
    assert f"dp_gemm_kernel<{planes[0]}, {planes[1]}, {128 if planes == (2, 2) else 256}, true, {str(d_out % 4 != 0).lower()}>" in launch.kernel
    assert launch.cooperative and launch.grid == 152 and launch.arg == lanes
