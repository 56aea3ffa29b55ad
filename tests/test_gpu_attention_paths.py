"""The attention paths that the decoder picks by itself against the per-row walk (attention_mode 1),
bit for bit, at the sizes where a path can go wrong: key lists that end inside, at and past a 16-key
block and the score cache, lists whose rows are not consecutive, more words than a group holds."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2410_05911_gb300 import aecct as A
from paper_2410_05911_gb300 import inputs as I

torch = pytest.importorskip("torch")


def random_code(n, m, weight, seed):
    """A code whose variables join `weight` random checks each (every check at least one variable)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    H = np.zeros((m, n), np.uint8)
    for j in range(n):
        H[rng.permutation(m)[:weight], j] = 1
    H[np.arange(m), np.arange(m) % n] = 1
    return I.LinearCode(f"random({n},{n - m})", n, n - m, H, np.zeros((1, n), np.uint8))


def both(model, B, seed, mode=0):
    rng = np.random.Generator(np.random.PCG64(seed))
    y = torch.from_numpy(rng.standard_normal((B, model.n)).astype(np.float32)).cuda()
    got = []
    for attention in (mode, 1):
        dec = A.Decoder(model, attention_mode=attention)
        got.append([t.clone() for t in dec.decode(y)] + [dec.query()["attention_mode"]])
        torch.cuda.synchronize()
        assert dec.synchronize() == A.AECCT_OK
        dec.close()
    return got


def same(got):
    a, b = got
    assert torch.equal(a[2].view(torch.int32), b[2].view(torch.int32)), "logits"
    assert torch.equal(a[0], b[0]) and torch.equal(a[1], b[1])


# (n, m, column weight): union lists below, at and above 16, 64 and 96 keys, up to 128 tokens
TASKS = [(7, 3, 2), (18, 14, 2), (17, 15, 3), (33, 31, 1), (64, 32, 4), (65, 31, 3), (96, 32, 3), (97, 31, 2),
         (110, 18, 3), (120, 8, 2)]


@pytest.mark.gpu
@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("n,m,weight", TASKS, ids=lambda v: str(v))
def test_warp_tasks_equal_per_row_walk(n, m, weight, d):
    if d == 128 and (n + 31) // 32 * 32 + m > 128:
        pytest.skip("warp tasks at d = 128 hold one padded word in 128 rows")
    for mask_mode in (0, 1):
        model = I.random_model(random_code(n, m, weight, n + d), d, 2, seed=n, spe_noise=True)
        model.mask_mode = mask_mode
        got = both(model, 5, seed=m, mode=2)
        assert got[0][3] == 2 and got[1][3] == 1
        same(got)


@pytest.mark.gpu
@pytest.mark.parametrize("d", [32, 64, 128])
def test_warp_tasks_keep_an_infinite_value_with_its_queries(d):
    # one token's embedding so large that its V overflows: the rows that do not attend to it keep the
    # finite attention outputs (recorded O operand) that the per-row walk gives them
    code = random_code(40, 20, 2, 3)
    model = I.random_model(code, d, 1, seed=5, spe_noise=True)
    model.emb[7] = 1.0e38
    model.w_scale[0, 2] = 1.0e4
    rng = np.random.Generator(np.random.PCG64(2))
    y = torch.from_numpy(np.clip(rng.standard_normal((3, code.n)), -2, 2).astype(np.float32)).cuda()
    caps = []
    for mode in (2, 1):
        dec = A.Decoder(model, attention_mode=mode)
        cap = dec.set_capture(3)
        dec.decode(y)
        torch.cuda.synchronize()
        caps.append({k: cap[k].cpu().numpy() for k in ("alpha", "acc")})
        dec.close()
    finite = np.isfinite(caps[1]["alpha"][:, 0, 1])
    assert finite.any() and not finite.all()
    assert (np.isfinite(caps[0]["alpha"][:, 0, 1]) == finite).all()
    assert (caps[0]["alpha"][:, 0, 1][finite] == caps[1]["alpha"][:, 0, 1][finite]).all()
    assert (caps[0]["acc"][:, 0, 1][finite] == caps[1]["acc"][:, 0, 1][finite]).all()


# LDPC codes of 129 to 639 tokens (staged over a cluster) at both widths, lists of one block (HPSA) and
# more (the code-aware mask), an odd token count, several words to a group, a batch that ends inside one
STAGED = [(86, 64, 3), (100, 50, 6), (128, 64, 3), (131, 60, 5), (200, 57, 8), (426, 213, 3)]


@pytest.mark.gpu
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("mask_mode", [0, 1])
@pytest.mark.parametrize("n,m,weight", STAGED, ids=lambda v: str(v))
def test_staged_attention_equals_per_row_walk(n, m, weight, mask_mode, d):
    if weight == 3 and n == 2 * m:
        code = I.ldpc_regular_code(n, m, 3, 6, seed=n)
    else:
        code = random_code(n, m, weight, n + d)
    model = I.random_model(code, d, 2, seed=n, spe_noise=True, activation=1 if weight == 5 else 0)
    model.mask_mode = mask_mode
    got = both(model, 2 * 152 // 3 + 5 if n <= 128 else 3, seed=m)
    assert got[0][3] == 3 and got[1][3] == 1
    same(got)


@pytest.mark.gpu
def test_staged_attention_takes_what_the_buffers_hold():
    # 642 tokens: past the rows of the staged buffers, the per-row walk stays; and an explicit request for
    # staged attention at d = 64 is refused as before
    code = I.ldpc_regular_code(428, 214, 3, 6, seed=1)
    for d in (64, 128):
        dec = A.Decoder(I.random_model(code, d, 1, seed=1, spe_noise=True))
        assert dec.query()["attention_mode"] == 1
        dec.close()
    st, h = A.create_handle(I.random_model(I.make_code("ldpc128_64"), 64, 1, seed=1), attention_mode=3)
    assert st == A.AECCT_ERR_UNSUPPORTED and h is None


# d = 32: more groups than SMs run two CTAs on each SM, with half the score cache (48 keys)
@pytest.mark.gpu
@pytest.mark.parametrize("n,m,weight,variant", [(31, 15, 3, "relu"), (16, 14, 2, "alpha"), (33, 15, 3, "gelu"),
                                                (34, 15, 4, "full"), (64, 32, 4, "relu"), (110, 18, 3, "relu")])
def test_two_ctas_per_sm_equal_one(n, m, weight, variant):
    model = I.random_model(random_code(n, m, weight, n), 32, 2, seed=n, spe_noise=True,
                           activation=1 if variant == "gelu" else 0, full_precision=variant == "full")
    model.alpha_mode = 1 if variant == "alpha" else 0
    dec = A.Decoder(model)
    q = dec.query()
    assert q["attention_mode"] == 2
    B = q["words_per_group"] * (q["max_clusters"] + q["max_clusters"] // 2) + 1  # some CTAs take a second group
    rng = np.random.Generator(np.random.PCG64(n))
    y = torch.from_numpy(rng.standard_normal((B, n)).astype(np.float32)).cuda()
    cap = {k: v for k, v in dec.set_capture(3).items()}
    many = [t.clone() for t in dec.decode(y)]
    torch.cuda.synchronize()
    first = {k: v.clone() for k, v in cap.items()}
    # the same words a few at a time: one CTA per SM
    step = 100 * q["words_per_group"]
    few = [[t.clone() for t in dec.decode(y[s:s + step].contiguous())] for s in range(0, B, step)]
    torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK
    for i in range(3):
        got = torch.cat([f[i] for f in few])
        assert torch.equal(many[i].view(torch.uint8), got.view(torch.uint8))
    again = dec.set_capture(3)
    dec.decode(y[:3].contiguous())
    torch.cuda.synchronize()
    assert all(torch.equal(first[k].view(torch.uint8), again[k].view(torch.uint8)) for k in first)
    dec.close()


# the warp tasks are compiled with and without the capture: same outputs, also where only part of the batch is
# recorded and after the capture is off again
@pytest.mark.gpu
@pytest.mark.parametrize("d,many", [(32, False), (32, True), (64, False), (128, False)])
@pytest.mark.parametrize("variant", ["relu", "gelu", "full", "full-gelu"])
def test_plain_decode_equals_decode_with_capture(d, many, variant):
    model = I.random_model(random_code(31, 15, 3, d), d, 2, seed=d, spe_noise=True,
                           activation=1 if "gelu" in variant else 0, full_precision="full" in variant)
    dec = A.Decoder(model, attention_mode=2)
    q = dec.query()
    assert q["attention_mode"] == 2
    B = q["words_per_group"] * (q["max_clusters"] + 3) + 1 if many else q["words_per_group"] + 1
    rng = np.random.Generator(np.random.PCG64(d))
    y = torch.from_numpy(rng.standard_normal((B, model.n)).astype(np.float32)).cuda()
    got = []
    for cap_B in (0, 1, 0):
        dec.set_capture(cap_B)
        got.append([t.clone() for t in dec.decode(y)])
        torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK
    dec.close()
    for other in got[1:]:
        assert all(torch.equal(a.view(torch.uint8), b.view(torch.uint8)) for a, b in zip(got[0], other))


# one alpha per quantised matrix of a word, in CTAs of more words (18) than warps
@pytest.mark.gpu
@pytest.mark.parametrize("mode", [1, 2])
def test_word_alpha_of_more_words_than_warps(mode):
    model = I.random_model(random_code(5, 2, 1, 37), 32, 2, seed=5, spe_noise=True)
    model.alpha_mode = 1
    dec = A.Decoder(model, attention_mode=mode)
    assert dec.query()["words_per_group"] == 18
    y = np.random.Generator(np.random.PCG64(5)).standard_normal((37, 5)).astype(np.float32)
    r = O.decode(model, y)
    bits, syn, logits = dec.decode(torch.from_numpy(y).cuda())
    torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK
    dec.close()
    assert (logits.cpu().numpy().view(np.int32) == r["logits"].view(np.int32)).all()
    assert (bits.cpu().numpy() == r["bits"]).all() and (syn.cpu().numpy() == r["syndrome"]).all()


# batches that leave SMs idle put fewer words into a CTA than it holds: the same outputs as in a batch that
# fills every CTA, at the counts where the number of words changes
@pytest.mark.gpu
@pytest.mark.parametrize("d", [32, 64])
@pytest.mark.parametrize("n,m,weight,alpha", [(31, 15, 3, 0), (18, 14, 2, 1), (7, 3, 2, 0), (5, 2, 1, 1), (40, 20, 2, 0)])
def test_fewer_words_per_cta_equal_a_full_batch(n, m, weight, alpha, d):
    model = I.random_model(random_code(n, m, weight, n + d), d, 2, seed=n, spe_noise=True)
    model.alpha_mode = alpha
    dec = A.Decoder(model, attention_mode=2)
    G, sms = dec.query()["words_per_group"], torch.cuda.get_device_properties(0).multi_processor_count
    rng = np.random.Generator(np.random.PCG64(n))
    y = torch.from_numpy(rng.standard_normal((2 * G * sms + 1, n)).astype(np.float32)).cuda()
    full = [t.clone() for t in dec.decode(y)]
    for B in sorted({1, 2, sms - 1, sms, sms + 1, 2 * sms + 1, (G - 1) * sms, (G - 1) * sms + 1, G * sms - 1, G * sms}):
        if B == 0:
            continue
        got = dec.decode(y[:B].contiguous())
        assert all(torch.equal(a[:B].view(torch.uint8), b.view(torch.uint8)) for a, b in zip(full, got)), B
    assert dec.synchronize() == A.AECCT_OK
    dec.close()


# a word whose values are not finite reaches no other word, and costs about what any word does
@pytest.mark.gpu
@pytest.mark.parametrize("key,d", [("bch31_16", 32), ("bch31_16", 64), ("polar64_32", 64), ("bch63_36", 128)])
def test_words_with_a_nan_among_others(key, d):
    model = I.random_model(I.make_code(key), d, 2, seed=3, spe_noise=True)
    dec = A.Decoder(model)
    assert dec.query()["attention_mode"] == 2
    y = torch.from_numpy(np.random.Generator(np.random.PCG64(d)).standard_normal((4096, model.n)).astype(np.float32)).cuda()
    some, every = y.clone(), y.clone()
    some[::3, 3] = float("nan")
    every[:, 3] = float("nan")
    keep = torch.arange(4096, device="cuda") % 3 != 0
    want, got = dec.decode(y), dec.decode(some)
    assert all(torch.equal(a[keep].view(torch.uint8), b[keep].view(torch.uint8)) for a, b in zip(want, got))

    def fastest(v):
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            dec.decode(v)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times[2:])

    # a branch around every fold is 1.2 times the attention without; a walk key by key was 1.6 to 2.4 times the decode
    plain, nan = fastest(y), fastest(every)
    assert nan <= 1.4 * plain, (plain, nan)
    assert dec.synchronize() == A.AECCT_OK
    dec.close()


# two CTAs to an SM only where their shared memory fits: not with the plan of 32 words of four tokens
@pytest.mark.gpu
@pytest.mark.parametrize("n,m,weight,per_sm", [(3, 1, 1, 1), (4, 1, 1, 2), (5, 2, 1, 2), (31, 15, 3, 2), (110, 18, 3, 2)])
def test_two_ctas_per_sm_where_they_fit(n, m, weight, per_sm):
    model = I.random_model(random_code(n, m, weight, n), 32, 2, seed=n, spe_noise=True)
    dec = A.Decoder(model)
    q, props = dec.query(), torch.cuda.get_device_properties(0)
    sms, smem_sm = props.multi_processor_count, 233472  # 228 KB
    assert q["max_clusters"] == per_sm * sms
    assert per_sm * (q["smem_bytes"] + 1024) <= smem_sm
    B = 2 * q["words_per_group"] * sms + 3  # more groups than SMs
    y = np.random.Generator(np.random.PCG64(n)).standard_normal((B, n)).astype(np.float32)
    _, _, logits = dec.decode(torch.from_numpy(y).cuda())
    torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK
    dec.close()
    for part in (slice(0, 40), slice(B - 40, B)):
        assert (logits[part].cpu().numpy().view(np.int32) == O.decode(model, y[part])["logits"].view(np.int32)).all()


# staged attention against the oracle: both widths (d = 64 takes it by default only), short lists and long ones
@pytest.mark.gpu
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("mask_mode", [0, 1])
def test_staged_attention_matches_oracle(mask_mode, d):
    model = I.random_model(I.make_code("ldpc128_64"), d, 2, seed=11, spe_noise=True)
    model.mask_mode = mask_mode
    y = np.random.Generator(np.random.PCG64(12)).standard_normal((7, model.n)).astype(np.float32)
    dec = A.Decoder(model)
    assert dec.query()["attention_mode"] == 3
    bits, syn, logits = dec.decode(torch.from_numpy(y).cuda())
    torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK
    dec.close()
    r = O.decode(model, y)
    assert (logits.cpu().numpy().view(np.int32) == r["logits"].view(np.int32)).all()
    assert (bits.cpu().numpy() == r["bits"]).all() and (syn.cpu().numpy() == r["syndrome"]).all()


# full-precision linears: the attention outputs go to the O GEMM as bf16, by another store
@pytest.mark.gpu
@pytest.mark.parametrize("d", [64, 128])
@pytest.mark.parametrize("mask_mode", [0, 1])
def test_staged_attention_with_full_precision_linears_equals_per_row_walk(mask_mode, d):
    model = I.random_model(I.make_code("ldpc128_64"), d, 2, seed=13, spe_noise=True, activation=mask_mode, full_precision=True)
    model.mask_mode = mask_mode
    got = both(model, 107, seed=14)
    assert got[0][3] == 3 and got[1][3] == 1
    same(got)


# one alpha per quantised matrix of a word through the staged path's own exchange, several words to a CTA
@pytest.mark.gpu
@pytest.mark.parametrize("key,words", [("hamming7_4", 12), ("bch31_16", 2), ("polar64_32", 1)])
def test_staged_attention_with_word_alpha_matches_oracle(key, words):
    model = I.random_model(I.make_code(key), 128, 2, seed=15, spe_noise=True)
    model.alpha_mode = 1
    dec = A.Decoder(model, attention_mode=3)
    q = dec.query()
    assert (q["attention_mode"], q["words_per_group"]) == (3, words)
    y = np.random.Generator(np.random.PCG64(16)).standard_normal((2 * words + 1, model.n)).astype(np.float32)
    _, _, logits = dec.decode(torch.from_numpy(y).cuda())
    torch.cuda.synchronize()
    assert dec.synchronize() == A.AECCT_OK
    dec.close()
    assert (logits.cpu().numpy().view(np.int32) == O.decode(model, y)["logits"].view(np.int32)).all()
