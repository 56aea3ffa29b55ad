"""The GPU weight quantiser at the sizes where its split can go wrong (a tensor in one CTA's registers, over
a cluster, past its registers, slices that end inside a thread's groups), with tied medians, unaligned
tensors and the flat path of other types and layouts, bit for bit against the oracle."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_05911_gb300 import aecct as A
from test_gpu_aap import _unpack

torch = pytest.importorskip("torch")


def check(tensors, host):
    delta = np.linspace(0.7, 2.2, len(host)).astype(np.float32)
    codes, scale, wq = A.aap_ternarize(tensors, delta, 1e-8, want_weights=True)
    torch.cuda.synchronize()
    for j, t in enumerate(host):
        ref_t, ref_sc = O.ternary(t, delta=float(delta[j]), eps=1e-8)
        assert (_unpack(codes[j].cpu().numpy()) == ref_t.reshape(-1)).all(), f"tensor {j}"
        assert scale[j].cpu().numpy().view(np.int32) == np.float32(ref_sc).view(np.int32)
        want = (np.float32(ref_sc) * ref_t.astype(np.float32)).reshape(-1)
        assert wq[j].shape == tensors[j].shape
        assert (wq[j].cpu().numpy().reshape(-1).view(np.int32) == want.view(np.int32)).all()


@pytest.mark.gpu
@pytest.mark.parametrize("size", [4, 8, 2044, 2048, 8188, 8192, 8196, 16384, 16388, 65536, 65540, 131072, 300004])
@pytest.mark.parametrize("kind", ["normal", "ties", "two scales"])
def test_sizes(size, kind):
    rng = np.random.default_rng(size)
    w = rng.standard_normal(size).astype(np.float32)
    if kind == "ties":
        w = np.round(w * 2) / 2
    if kind == "two scales":  # the two middle order statistics far apart
        w[: size // 2] = np.abs(w[: size // 2]) * 1e-3 + 1e-4
        w[size // 2:] += np.sign(w[size // 2:]) * 10
    host = [w.astype(np.float32), rng.standard_normal(size).astype(np.float32)]
    check([torch.from_numpy(t).cuda() for t in host], host)


@pytest.mark.gpu
def test_unaligned_and_other_layouts():
    rng = np.random.default_rng(3)
    base = torch.from_numpy(rng.standard_normal(4000).astype(np.float32)).cuda()
    views = [base[1:1025], base[2:3002].reshape(50, 60), base[3:7]]  # contiguous, 4, 8 and 12 bytes past 16
    check(views, [v.cpu().numpy() for v in views])
    mixed = [base[:64].reshape(8, 8).t(), base[64:128].half(), base[128:192]]  # the flat path
    check(mixed, [v.float().contiguous().cpu().numpy() for v in mixed])
