"""GEMMs that cut tiles along d_in, on several streams at once: calls of different kinds, made in turn, have scratch of
their own, so every accumulator is the exact one."""
import numpy as np
import pytest
import torch

import dp_planes
import sm4x8
import workloads as WL

pytestmark = pytest.mark.gpu

cat = pytest.importorskip("paper_2603_04359_gb300")
DEV = "cuda"


def dp_call(n, d_in, d_out, bits_x, bits_w):
    rng = np.random.default_rng(n + d_out)
    qx, qw = (rng.integers(-2 ** (b - 1) + 1, 2 ** (b - 1), s) for b, s in ((bits_x, (n, d_in)), (bits_w, (d_out, d_in))))
    xp, wp = (torch.from_numpy(dp_planes.encode(q, b, False)).to(DEV) for q, b in ((qx, bits_x), (qw, bits_w)))
    ones = torch.ones(max(n, d_out), device=DEV)
    ref = torch.from_numpy(qx).to(DEV).double() @ torch.from_numpy(qw).to(DEV).double().T

    def run(acc, y):
        cat.cat_linear_dp(xp, bits_x, ones[:n], wp, bits_w, ones[:d_out], y=y, acc_out=acc)
    return run, ref


def w4a4_call(n, d_in, d_out, code_bytes):
    rng = np.random.default_rng(n + d_out)
    qx, qw = WL.random_codes(rng, (n, d_in)), WL.random_codes(rng, (d_out, d_in))
    xq, wq = (torch.from_numpy(sm4x8.pack(q)).to(DEV) for q in (qx, qw))
    ones = torch.ones(max(n, d_out), device=DEV)
    ref = torch.from_numpy(qx).to(DEV).double() @ torch.from_numpy(qw).to(DEV).double().T
    if code_bytes:
        xq, wq = cat.cat_codes_to_e4m3(xq), cat.cat_codes_to_e4m3(wq)

    def run(acc, y):
        (cat.cat_w4a4_linear_e8 if code_bytes else cat.cat_w4a4_linear)(xq, ones[:n], wq, ones[:d_out], y=y, acc_out=acc)
    return run, ref


@pytest.mark.parametrize("make", [
    lambda: [dp_call(1000, 14336, 4096, 8, 8), dp_call(1000, 14336, 6144, 4, 4)],       # cut last waves of two bit widths
    lambda: [w4a4_call(256, 8192, 1000, True), w4a4_call(256, 8192, 3000, True)],       # split tails, 256 and 192 wide
    lambda: [w4a4_call(16, 2048, 24001, False), w4a4_call(32, 2048, 24001, False)],     # cut units, 16 and 32 tokens
    lambda: [w4a4_call(200, 8192, 128, i % 2 == 0) for i in range(4)],                  # a quarter of the device each
], ids=["digit_planes", "byte_codes", "weight_streaming", "small_splits"])
def test_cut_tiles_on_several_streams(make):
    calls = make()
    streams = [torch.cuda.Stream() for _ in calls]
    outs = [[(torch.empty(ref.shape, dtype=torch.int32, device=DEV), torch.empty(ref.shape, device=DEV)) for _ in range(4)]
            for _, ref in calls]
    torch.cuda.synchronize()
    for _ in range(5):
        for i in range(4):                                # (their scratch fits in turn)
            for (run, _), stream, out in zip(calls, streams, outs):
                with torch.cuda.stream(stream):
                    run(*out[i])
        torch.cuda.synchronize()
        assert cat.cat_device_status()[0] == 0
        for (_, ref), out in zip(calls, outs):
            for acc, y in out:
                assert torch.equal(acc.double(), ref) and torch.equal(y, acc.float())
                acc.fill_(-1)
