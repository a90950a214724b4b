"""Which kernel a linear takes, asked of the library on the CPU (148 SMs)."""
import pytest

from paper_2507_14959_b200 import binding

NONE, GELU, RESIDUAL, PATCH = 0, 1, 2, 3
TOKENS = 197


def test_arguments():
    for bad in ((100, 128, 1, NONE), (128, 100, 1, NONE), (128, 128, 0, NONE), (128, 128, 1, 4), (0, 128, 1, NONE)):
        with pytest.raises(binding.PolymorphError):
            binding.linear_kernel(*bad, adapters=False)
    with pytest.raises(binding.PolymorphError):
        binding.linear_kernel(128, 128, 1, NONE, False, n_sms=0)


@pytest.mark.parametrize("k_in,n_out,frames,width,split", [
    (3072, 768, 1, 64, 4), (3072, 768, 2, 128, 4), (3072, 768, 4, 128, 2), (3072, 768, 8, 192, 2), (3072, 768, 12, 256, 2), (3072, 768, 15, 256, 2),
    (2048, 512, 12, 256, 2), (2048, 512, 24, 256, 2), (4096, 1024, 6, 256, 2), (4096, 1024, 11, 256, 2), (3072, 768, 17, 192, 1)])
def test_long_k_with_adapters_is_split_while_the_sms_suffice(k_in, n_out, frames, width, split):
    """Each share of t keeps 16 significant bits there, which no other form does."""
    assert binding.linear_kernel(k_in, n_out, frames * TOKENS, RESIDUAL, True)[:3] == ("few rows", width, split)
