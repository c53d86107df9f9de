"""The weight-streaming skinny GEMM of the decode kernel against a float64 matrix product."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

from paper_2506_03700_b200 import binding, synth


def _case(N, K, cols, mode, seed=7):
    W = synth.normal_tensor(seed, 11, (N, K), 0.05, torch.bfloat16, "cuda")
    X = synth.normal_tensor(seed, 12, (cols, K), 1.0, torch.float32, "cuda")
    Y, _ = binding.debug_gemm(W, X, mode)
    Wd, Xd = W.double().cpu().numpy(), X.double().cpu().numpy()
    ref = Xd @ Wd.T
    if mode == 1:
        g, u = ref[:, :N // 2], ref[:, N // 2:]
        ref = g / (1.0 + np.exp(-g)) * u
    return Y.double().cpu().numpy(), ref


# shapes: one tile; ragged last tile and several k chunks; k tail shorter than a chunk; more
# tiles than the grid holds at once (several groups per block); the 8B-shaped down projection
@pytest.mark.parametrize("N,K,cols", [(16, 64, 1), (48, 128, 3), (1000, 1216, 8), (5003, 512, 5), (40000, 192, 2),
                                      (4096, 14336, 6), (6144, 4096, 1)])
def test_streaming_gemm_matches_float64(N, K, cols):
    y, ref = _case(N, K, cols, 0)
    assert np.abs(y - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())


@pytest.mark.parametrize("N,K,cols", [(2 * 688, 256, 4), (2 * 14336, 4096, 6), (2 * 16, 64, 8)])
def test_streaming_gate_up_swiglu(N, K, cols):
    y, ref = _case(N, K, cols, 1)
    assert np.abs(y - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())


def test_result_of_a_column_does_not_depend_on_the_other_columns():
    """The same token in another column, alone or beside other tokens, gives the same bits."""
    N, K = 2048, 1536
    W = synth.normal_tensor(3, 11, (N, K), 0.05, torch.bfloat16, "cuda")
    X = synth.normal_tensor(3, 12, (8, K), 1.0, torch.float32, "cuda")
    full, _ = binding.debug_gemm(W, X, 0)
    for c in (0, 3, 7):
        alone, _ = binding.debug_gemm(W, X[c:c + 1].contiguous(), 0)
        assert torch.equal(alone[0], full[c])
    perm = [5, 2, 7, 0]
    mixed, _ = binding.debug_gemm(W, X[perm].contiguous(), 0)
    for j, c in enumerate(perm):
        assert torch.equal(mixed[j], full[c])


def test_bad_arguments_are_refused():
    W = torch.zeros(32, 48, dtype=torch.bfloat16, device="cuda")      # K not a multiple of 64
    X = torch.zeros(1, 48, dtype=torch.float32, device="cuda")
    with pytest.raises(binding.AdaError) as e:
        binding.debug_gemm(W, X, 0)
    assert e.value.code == -1


# ---------------------------------------------------------------- dense GEMM of the prompt pass (tcgen05)

@pytest.mark.parametrize("N,K,rows", [(64, 64, 128), (64, 256, 5), (200, 512, 128), (6144, 4096, 77), (4096, 14336, 128)])
def test_dense_gemm_matches_float64(N, K, rows):
    W = synth.normal_tensor(9, 11, (N, K), 0.05, torch.bfloat16, "cuda")
    X = synth.normal_tensor(9, 12, (rows, K), 1.0, torch.float32, "cuda")
    Y = binding.debug_dense_gemm(W, X)
    ref = X.double().cpu().numpy() @ W.double().cpu().numpy().T
    assert torch.isfinite(Y).all()
    assert np.abs(Y.double().cpu().numpy() - ref).max() <= 2e-5 * max(1.0, np.abs(ref).max())
    # accumulate form: the product is added to what the output holds
    Y2 = torch.ones_like(Y)
    binding.debug_dense_gemm(W, X, Y2)
    assert np.abs(Y2.double().cpu().numpy() - (ref + 1.0)).max() <= 2e-5 * max(1.0, np.abs(ref).max())


# deepest accumulator: an eighth of the depth, 256 to 512
@pytest.mark.parametrize("N,K,rows,depth", [(3072, 2048, 100, 256), (2048, 2048, 21, 256), (16384, 2048, 128, 256), (5120, 3008, 64, 320),
                                            (4096, 4096, 77, 512), (4096, 14336, 9, 512)])
def test_sums_of_the_dense_gemm(N, K, rows, depth):
    """The error that the sums add to that of the operand's split.  The tensor core truncates after every addition of sixteen
    products, twice per sixteen k (high and low parts): half a unit in the last place on average, 0.36 * 2^-23 of a partial sum
    that is two thirds of the final one, i.e. 2.9e-8 of the result per addition at most, half of it where the digits are
    spread evenly; 1e-7 for the fp32 additions of the accumulators."""
    W = synth.normal_tensor(9, 11, (N, K), 0.05, torch.bfloat16, "cuda")
    X = synth.normal_tensor(9, 12, (rows, K), 1.0, torch.float32, "cuda")
    hi = X.bfloat16()
    lo = (X - hi.float()).bfloat16()
    ref = (hi.double() + lo.double()) @ W.double().T
    err = (binding.debug_dense_gemm(W, X).double() - ref).norm() / ref.norm()
    assert err <= 1.6e-8 * (2 * depth / 16) + 1e-7, err


def _product(N, K, rows, pairs=0, seed=9):
    W = synth.normal_tensor(seed, 11, (N, K), 0.05, torch.bfloat16, "cuda")
    X = synth.normal_tensor(seed, 12, (rows, K), 1.0, torch.float32, "cuda")
    return W, X, binding.debug_dense_product(W, X, pairs=pairs)


# tiles of 256 weight rows x one position tile against `pairs` pairs of CTAs: one short of a wave, a wave, one more, two waves and one
# more; several position tiles; depths that are no multiple of a chunk or leave a last group shorter
@pytest.mark.parametrize("N,K,rows,pairs", [
    (73 * 256, 1088, 100, 74), (74 * 256, 1088, 64, 74), (75 * 256, 1088, 33, 74), (149 * 256, 576, 40, 74),
    (4 * 256, 3008, 100, 5), (5 * 256, 3008, 100, 5), (6 * 256, 3008, 256, 5), (11 * 256, 3008, 256, 5), (3 * 256 - 60, 5504, 300, 7),
    (4096, 14336, 777, 74), (6144, 4096, 2048, 74), (2048, 8192, 513, 74), (256, 14336, 257, 74), (64, 64, 2048, 74), (300, 192, 1, 74)])
def test_divided_products_match_float64(N, K, rows, pairs):
    W, X, Y = _product(N, K, rows, pairs)
    ref = X.double() @ W.double().T
    assert torch.isfinite(Y).all()
    # the split of X leaves 2^-17 of an element at most, 2.5e-6 of a result in the 2-norm; the sums 1.1e-6 (test_sums_of_the_dense_gemm)
    assert (Y.double() - ref).norm() <= 3e-6 * ref.norm()
    assert (Y.double() - ref).abs().max() <= 2e-5 * max(1.0, ref.abs().max())
    Y2 = binding.debug_dense_product(W, X, torch.ones_like(Y), pairs=pairs)
    assert (Y2.double() - (ref + 1.0)).abs().max() <= 2e-5 * max(1.0, ref.abs().max())


@pytest.mark.parametrize("N,K", [(2048, 8192), (4096, 3008), (19 * 256, 5504)])
def test_rows_of_a_divided_product_do_not_depend_on_how_many_there_are(N, K):
    W, X, Y = _product(N, K, 2048)
    for rows in (32, 97, 256, 260, 600, 1111):
        assert torch.equal(binding.debug_dense_product(W, X[:rows].contiguous()), Y[:rows]), rows
