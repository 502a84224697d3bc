"""Local cluster positions at every length remainder and alignment of the arrays,
against the oracle bit for bit (one subtraction and one product, both rounded)."""
import numpy as np
import pytest

import oracle as orc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2101_11489_gb300 as sst  # noqa: E402

N_FEDS = 7


@pytest.mark.parametrize("offsets", [(0, 0, 0), (4, 4, 4), (1, 0, 0), (0, 2, 0), (0, 0, 3), (1, 1, 1)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 7, 1023, 1024, 1025, 1_300_003])  # the last: more than one pass of the grid
def test_local_x_alignments(n, offsets):
    rng = np.random.default_rng(n)
    pitch = rng.uniform(0.05, 0.3, N_FEDS * 96).astype(np.float32)
    det = rng.integers(0, N_FEDS * 96, n).astype(np.uint32)
    bary = rng.uniform(0.0, 256.0, n).astype(np.float32)
    want = orc.local_x(det, bary, pitch)
    outside = rng.random(n) < 0.1  # module ids outside the detector
    det[outside] = rng.integers(N_FEDS * 96, 2**32, int(outside.sum()), dtype=np.uint64).astype(np.uint32)
    want[outside] = np.nan
    ctx = sst.sst_create(0, N_FEDS)
    try:
        sst.sst_pitch_upload(ctx, pitch)
        buf = [torch.zeros(n + 8, dtype=t, device="cuda") for t in (torch.int32, torch.float32, torch.float32)]
        d, b, x = (t[o:o + n] for t, o in zip(buf, offsets))
        d.copy_(torch.from_numpy(det.view(np.int32)))
        b.copy_(torch.from_numpy(bary))
        sst.sst_local_x(ctx, d, b, n, x)
        whole = buf[2].cpu().numpy()
        assert np.array_equal(whole[offsets[2]:offsets[2] + n], want, equal_nan=True)
        assert not whole[:offsets[2]].any() and not whole[offsets[2] + n:].any()
        sst.sst_local_x(ctx, d, b, n, b)  # in place
        assert np.array_equal(b.cpu().numpy(), want, equal_nan=True)
    finally:
        sst.sst_destroy(ctx)
