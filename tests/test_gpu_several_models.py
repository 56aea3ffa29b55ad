"""Several decoders alive at once: models of one width share their kernels and differ in the size of the
attention plan that a launch asks shared memory for.  Creating one must not change what another's launches
may ask for."""
import time

import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_05911_gb300 import aecct as A
from paper_2410_05911_gb300 import inputs as I

torch = pytest.importorskip("torch")


# (codes in the order of creation): the largest plan first, then smaller ones; d = 32 has the kernel at two
# CTAs per SM for batches of more groups than SMs
@pytest.mark.gpu
@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("codes", [("bch31_16", "polar64_32", "hamming7_4"), ("hamming7_4", "bch31_16", "polar64_32"),
                                   ("polar64_32", "ldpc128_64", "bch31_16")], ids="-".join)
def test_decoders_of_one_width_side_by_side(codes, d):
    models = [I.random_model(I.make_code(c), d, 2, seed=5, spe_noise=True) for c in codes]
    decs = [A.Decoder(m) for m in models]
    batches = [np.random.Generator(np.random.PCG64(i)).standard_normal((2100, m.n)).astype(np.float32)
               for i, m in enumerate(models)]
    refs = [O.decode(m, y[:4])["logits"] for m, y in zip(models, batches)]
    for i in (0, 1, 2, 0):
        for B in (4, 2100):
            _, _, logits = decs[i].decode(torch.from_numpy(batches[i][:B]).cuda())
            torch.cuda.synchronize()
            assert decs[i].synchronize() == A.AECCT_OK
            assert (logits[:4].cpu().numpy().view(np.int32) == refs[i].view(np.int32)).all(), (codes[i], B)
    for dec in decs:
        dec.close()


@pytest.mark.gpu
@pytest.mark.parametrize("d", [32, 64])
def test_create_with_a_plan_for_every_word_count(d):
    # 24 tokens: plans for one to five words to a CTA; a decoder without plans has the same uploads
    code = I.ldpc_regular_code(16, 8, 3, 6, seed=1)
    model = I.random_model(code, d, 1, seed=5, spe_noise=True, full_precision=True)

    def fastest(mode):
        times = []
        for _ in range(20):
            t0 = time.perf_counter()
            st, h = A.create_handle(model, attention_mode=mode)
            times.append(time.perf_counter() - t0)
            assert st == A.AECCT_OK
            A.load().aecct_destroy(h)
        return min(times)

    plans, none = fastest(2), fastest(1)
    assert plans <= none + 0.2e-3, (plans, none)
