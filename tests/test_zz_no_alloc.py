"""eig_gram_noalloc: the Gram product for callers that cannot allocate device memory (its scratch
is a fixed array inside the library).  Its result must equal eig_gram's on the same inputs, on
two calls in a row (the shared scratch keeps the previous call's contents), and the capped
grouping of a GPU with more SMs than the array has partials must still give A^T B (against the
oracle's FP64 product).  This file is collected last so that a run stopping at the first failure
has already run every other test."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
def test_gram_noalloc_matches_gram_on_two_calls(dt):
    from paper_2305_15552_gb300 import binding
    binding.load()
    rng = np.random.default_rng(11)
    for call, (n, nb) in enumerate([(200003, 16), (70001, 8)]):
        A = torch.tensor(rng.standard_normal((n, nb)), dtype=dt, device="cuda")
        B = torch.tensor(rng.standard_normal((n, nb)), dtype=dt, device="cuda")
        ref = binding.gram(A, B).cpu().numpy()
        got = binding.gram_noalloc(A, B).cpu().numpy()
        torch.cuda.synchronize()
        Ae, Be = A.double().cpu().numpy(), B.double().cpu().numpy()
        bound = np.abs(Ae).T @ np.abs(Be)
        tol = (2.0 ** -24 * 40 if dt == torch.float32 else 2.0 ** -53 * (n + 10)) * bound + 1e-300
        assert np.all(np.abs(got - ref) <= tol), f"call {call}"


def test_gram_noalloc_rejects_oversized_block():
    from paper_2305_15552_gb300 import binding
    binding.load()
    A = torch.ones(1000, 64, device="cuda")
    with pytest.raises(binding.EigError) as e:
        binding.gram_noalloc(A, A)
    assert e.value.status == binding.EIG_EINVAL


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("parts", [1, 7, 300])
def test_gram_noalloc_capped_partials_match_oracle(dt, parts):
    """More rows per CTA partial than eig_gram uses here (the 512-partial cap of a larger GPU,
    forced through eig_gram_noalloc_parts), checked element by element against O.gram."""
    from paper_2305_15552_gb300 import binding
    binding.load()
    rng = np.random.default_rng(5 + parts)
    n, nb = 100003, 16
    A = torch.tensor(rng.standard_normal((n, nb)), dtype=dt, device="cuda")
    B = torch.tensor(rng.standard_normal((n, nb)), dtype=dt, device="cuda")
    got = binding.gram_noalloc(A, B, max_parts=parts).cpu().numpy()
    Ae, Be = A.double().cpu().numpy(), B.double().cpu().numpy()
    ref = O.gram(Ae, Be)
    bound = np.abs(Ae).T @ np.abs(Be)
    tol = (2.0 ** -24 * 40 if dt == torch.float32 else 2.0 ** -53 * (n + 10)) * bound + 1e-300
    assert np.all(np.abs(got - ref) <= tol)


def test_gram_noalloc_parts_rejects_bad_cap():
    from paper_2305_15552_gb300 import binding
    binding.load()
    A = torch.ones(1000, 8, device="cuda")
    for bad in (0, 513):
        with pytest.raises(binding.EigError) as e:
            binding.gram_noalloc(A, A, max_parts=bad)
        assert e.value.status == binding.EIG_EINVAL


@pytest.mark.parametrize("dt", [torch.float32, torch.float64])
@pytest.mark.parametrize("n,nb", [(33, 8), (70001, 5), (200003, 16), (400000, 8), (100003, 32)])
@pytest.mark.parametrize("same", [False, True])
def test_gram_noalloc_equals_gram_bitwise(dt, n, nb, same):
    """The partials of eig_gram fit the fixed array, so both calls must group and round alike, also for a
    block with itself (of which eig_gram multiplies the upper tiles only)."""
    from paper_2305_15552_gb300 import binding
    binding.load()
    rng = np.random.default_rng(n + nb)
    A = torch.tensor(rng.standard_normal((n, nb)), dtype=dt, device="cuda")
    B = A if same else torch.tensor(rng.standard_normal((n, nb)), dtype=dt, device="cuda")
    assert torch.equal(binding.gram_noalloc(A, B), binding.gram(A, B))


@pytest.mark.parametrize("nb", [8, 16, 32])
def test_gram_totals_over_many_chunks(nb):
    """FP32 chunk sums (32 rows) into one partial: a block whose chunks hold one nonzero product each, 1
    in the first chunks (of every group of threads that may share the rows) and a constant far below
    it in the others.  Every chunk sum is exact, so the total may lose 2^-48 of itself per chunk (double
    that for both roundings of the pair), and the partials' FP64 sum a few 2^-53."""
    from paper_2305_15552_gb300 import binding
    binding.load()
    chunks, first = 65536, 32
    c = np.float32(5.603129e-08) * np.float32(2.0) ** -np.arange(nb, dtype=np.float32)
    a = np.zeros((chunks, 32, nb), np.float32)
    a[:first, 0] = 1.0
    a[first:, 0] = c
    A = torch.tensor(a.reshape(-1, nb), device="cuda")
    ones = torch.ones_like(A)
    want = first + (chunks - first) * c.astype(np.float64)
    for x, y in ((A, ones), (ones, A)):
        for parts in (1, 3):
            got = binding.gram_noalloc(x, y, max_parts=parts).cpu().numpy()
            got = got if x is A else got.T
            assert np.all(np.abs(got - want[:, None]) <= chunks * 2.0 ** -47 * want[:, None])
