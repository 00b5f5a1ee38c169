"""The buffer of the training loss' partial sums holds one value per CTA of the packed last
convolution for every output width and batch (csrc/surrogate_packed.cu, conv_grid: past 152 blocks
of 32 channels the grid grows with the width)."""
import pytest

from paper_2606_12850_gb300 import build, sem


@pytest.fixture(scope="module")
def sizes():
    build.build()
    lib = sem.lib()  # host functions of the library's C++ side, int (int batch, int channels, int samples)
    return lib._ZN3sgk11loss_valuesEiii, lib._ZN3sgk18packed_loss_blocksEiii


@pytest.mark.parametrize("out_c", [1, 31, 32, 192, 4864, 4896, 19456, 19488, 19520, 65536])
@pytest.mark.parametrize("out_l", [1, 128, 129, 1000])
def test_loss_buffer_holds_every_block(sizes, out_c, out_l):
    loss_values, blocks = sizes
    for max_batch in (1, 2, 151, 256):
        have = loss_values(max_batch, out_c, out_l)
        assert have >= 608  # the general loss kernel's blocks
        if out_c % 32 == 0:
            for b in (1, max(1, max_batch // 2), max_batch):
                assert blocks(b, out_c, out_l) <= have


def test_wide_outputs_exceed_the_general_kernel_s_blocks(sizes):
    _, blocks = sizes
    assert blocks(256, 192, 1000) == 150
    assert blocks(1, 19456, 4) == 608 and blocks(1, 19488, 4) == 609
