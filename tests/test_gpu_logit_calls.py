"""The calls on a finished logits matrix at the edges of how they are cut up: vocabularies below, at and above the sizes at
which a row is spread over more CTAs (top-2: 1 to 8) or slices (arg-max: 1 to 64), one row to the largest number.  Against
the oracle's top2_probs (fp64) and numpy's arg-max; equal values test that ties go to the lowest id across slices.
Probabilities: fp32 sums of up to 70000 positive terms, error about sqrt(70000) * 2^-24 = 1.6e-5 at most, 1e-5 up to
32000, and well below where terms are added in slices."""
import numpy as np
import pytest
import torch

from oracle import specasr_oracle as O
from paper_2507_18181_b200 import binding as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("vocab", [1, 7, 1024, 1025, 4095, 4096, 8192, 16384, 32000, 70000])
@pytest.mark.parametrize("rows", [1, 5, 64, 256])
def test_top2_and_accept_of_a_logits_matrix(vocab, rows):
    rng = np.random.default_rng(vocab * 1000 + rows)
    logits = (rng.standard_normal((rows, vocab)) * 2).astype(np.float32)
    for r in range(0, rows, 3):                               # ties of the maximum, anywhere in the row
        at = rng.integers(0, vocab, size=3)
        logits[r, at] = logits[r].max() + 1
    d = torch.from_numpy(logits).cuda()
    ids = torch.full((rows, 2), -7, dtype=torch.int32, device="cuda")
    probs = torch.empty(rows, 2, device="cuda")
    B.specasr_top2_probs(d.data_ptr(), rows, vocab, ids.data_ptr(), probs.data_ptr())
    want_ids, want_probs = O.top2_probs(logits.astype(np.float64))
    assert np.array_equal(ids.cpu().numpy(), want_ids)
    assert np.allclose(probs.cpu().numpy(), want_probs, rtol=1e-5, atol=0)

    parent = np.arange(-1, rows - 1, dtype=np.int32)
    arg = logits.argmax(-1).astype(np.int32)                  # numpy: the first of equal maxima
    tokens = np.concatenate([[0], arg[:-1]]).astype(np.int32)
    if rows > 3 and vocab > 1:
        tokens[rows // 2] = (tokens[rows // 2] + 1) % vocab   # the chain breaks here
    want = O.accept(tokens, parent, arg)
    t, p = torch.from_numpy(tokens).cuda(), torch.from_numpy(parent).cuda()
    out = [torch.full((rows,), -7, dtype=torch.int32, device="cuda") for _ in range(2)]
    acc, bonus = torch.full((2,), -7, dtype=torch.int32, device="cuda"), torch.full((1,), -7, dtype=torch.int32, device="cuda")
    for _ in range(2):                                        # the second call finds the first one's leftovers
        B.specasr_accept_logits_static(d.data_ptr(), vocab, t.data_ptr(), p.data_ptr(), rows, out[0].data_ptr(),
                                       acc.data_ptr(), out[1].data_ptr(), bonus.data_ptr())
    a = int(acc[0])
    assert np.array_equal(out[0].cpu().numpy(), arg) and a == want["accept_len"] and int(bonus) == want["bonus"]
    path = out[1].cpu().numpy()
    assert list(path[:a + 1]) == list(want["path"]) and np.all(path[a + 1:] == -1)


@pytest.mark.parametrize("vocab,cut", [(32000, 28000), (32000, 20000), (32000, 1), (9000, 4000), (4096, 2048), (700, 300)])
def test_top2_of_rows_with_masked_values(vocab, cut):
    """-inf as a caller's mask: over the tail, the head (whole slices of a row and whole threads see nothing else), every
    other value, and all but two.  A masked value has probability 0 and changes nothing else (bound as above)."""
    rng = np.random.default_rng(cut)
    logits = (rng.standard_normal((4, vocab)) * 2).astype(np.float32)
    keep = logits[:, :2].copy()
    logits[0, max(cut, 2):] = -np.inf
    logits[1, :vocab - max(cut, 2)] = -np.inf
    logits[2, ::2] = -np.inf
    logits[3] = -np.inf
    logits[3, [cut // 2, vocab - 1]] = keep[3]
    d = torch.from_numpy(logits).cuda()
    ids = torch.full((4, 2), -7, dtype=torch.int32, device="cuda")
    probs = torch.empty(4, 2, device="cuda")
    B.specasr_top2_probs(d.data_ptr(), 4, vocab, ids.data_ptr(), probs.data_ptr())
    want_ids, want_probs = O.top2_probs(logits.astype(np.float64))
    assert np.array_equal(ids.cpu().numpy(), want_ids)
    assert np.allclose(probs.cpu().numpy(), want_probs, rtol=1e-5, atol=0)


@pytest.mark.parametrize("vocab", [2**31 - 1, 2**31 - 1500])
def test_widest_vocabularies(vocab):
    """One row of up to 2^31 - 1 tokens (8.6 GB): a thread's next index passes 2^31 there.  Everything is masked but three
    values, one in the last place, so that the expected probabilities are those of three numbers."""
    d = torch.full((vocab,), -float("inf"), device="cuda")
    at, val = [5, vocab // 2, vocab - 1], [0.25, 1.0, 2.0]
    for a, v in zip(at, val):
        d[a] = v
    ids, probs = torch.empty(1, 2, dtype=torch.int32, device="cuda"), torch.empty(1, 2, device="cuda")
    B.specasr_top2_probs(d.data_ptr(), 1, vocab, ids.data_ptr(), probs.data_ptr())
    e = np.exp(np.array(val))
    assert ids.tolist() == [[at[2], at[1]]]
    assert np.allclose(probs.cpu().numpy(), [[e[2] / e.sum(), e[1] / e.sum()]], rtol=1e-5, atol=0)
    t, p = torch.zeros(1, dtype=torch.int32, device="cuda"), torch.full((1,), -1, dtype=torch.int32, device="cuda")
    out = torch.full((4,), -7, dtype=torch.int32, device="cuda")
    B.specasr_accept_logits_static(d.data_ptr(), vocab, t.data_ptr(), p.data_ptr(), 1, out.data_ptr(), out[1:].data_ptr(),
                                   out[2:].data_ptr(), out[3:].data_ptr())
    assert out.tolist() == [vocab - 1, 0, 0, vocab - 1]
