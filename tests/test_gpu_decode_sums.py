"""The sums of a decode on their way out: pairs of row groups that several warps share, that one warp has to itself and that have
one group only, odd and even numbers of tokens, clusters of every size, and many rows of 16 tokens in one launch."""
import pytest
import torch

from paper_2305_14152_b200 import binding
from gpu_util import kernels_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [1, 2, 3, 5, 8, 9, 13, 16])
@pytest.mark.parametrize("N,K,bits,g", [(8, 128, 4, 0), (1048, 1536, 3, 0), (2072, 4224, 4, 128), (520, 9088, 3, 64), (22016, 2048, 3, 0)])
def test_sums_of_all_shapes(N, K, bits, g, M):
    gen = torch.Generator(device="cuda").manual_seed(N + M)
    w = binding.quantize_rtn(torch.randn((N, K), generator=gen, device="cuda"), bits, g)
    X = torch.randn((M, K), generator=gen, device="cuda").bfloat16()
    table = (w.scales * (1 + 0.1 * torch.rand((3,) + tuple(w.scales.shape), generator=gen, device="cuda"))).contiguous()
    ids = torch.randint(0, 3, (M,), generator=gen, device="cuda", dtype=torch.int32)
    codes = binding.unpack(w.qweight, K, bits).double().view(N, w.G, K // w.G) - w.zeros.double()[:, :, None]

    def check(Y, scales):
        for m in range(M):
            ref = (codes * scales[m].double()[:, :, None]).view(N, K) @ X[m].double()
            # bf16 has eight significant bits: rounding to it moves a value in [2^e, 2^(e+1)) by up to 2^(e-8), 2^-8 of the
            # smallest; the sums before it are good to 1e-5 of the outputs' norm
            assert ((Y[m].double() - ref).abs() <= 2.0 ** -8 * ref.abs() + 1e-5 * ref.norm()).all()

    prepared = binding.decode_prepare(w)
    check(binding.qlinear_decode_prepared(w, prepared, X), [w.scales] * M)
    check(binding.qlinear_decode_prepared(w, prepared, X, scale_table=table, task_ids=ids), [table[t] for t in ids.tolist()])
    if M <= 8 and g != 64:
        check(binding.qlinear_decode(w, X), [w.scales] * M)
    binding.check_status()


def test_sixteen_tokens_of_many_rows_take_one_launch():
    w = binding.quantize_rtn(torch.randn((22016, 8192), device="cuda"), 3, 0)
    prepared, X = binding.decode_prepare(w), torch.randn((16, 8192), device="cuda").bfloat16()
    binding.qlinear_decode_prepared(w, prepared, X)
    names = [n for n in kernels_of(lambda: binding.qlinear_decode_prepared(w, prepared, X)) if "decode_prep_kernel" in n]
    assert len(names) == 1, names


def test_many_columns_of_grouped_weights_take_two_launches():
    """13 tokens at once would be worked through in nine chunks of K, seven and six fit a cluster's CTAs."""
    w = binding.quantize_rtn(torch.randn((8192, 22016), device="cuda"), 4, 128)
    prepared, X = binding.decode_prepare(w), torch.randn((13, 22016), device="cuda").bfloat16()
    names = [n for n in kernels_of(lambda: binding.qlinear_decode_prepared(w, prepared, X)) if "decode_prep_kernel" in n]
    assert len(names) == 2, names
