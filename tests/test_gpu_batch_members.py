"""Batch members against the same simulations stepped one by one: a member without
particles, whose tile arrays were allocated anew (their memory is whatever the
allocator hands out), and a field set on a member between two calls.  Fields of a
vacuum run come from the same kernels in the same order: equal to the last bit.
"""
import numpy as np
import pytest

from paper_1204_0838_gb300 import pic, workloads as W

pytestmark = pytest.mark.gpu

LAM = W.LAMBDA0
SHAPE = (40, 20, 24)


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    pic.lib()


class _DirtyMemory(pic.TorchMemory):
    """Device memory full of a large positive (or negative) number."""

    def __init__(self, byte):
        super().__init__()
        self.byte = byte

    def _alloc(self, nbytes, ctx):
        ptr = super()._alloc(nbytes, ctx)
        if ptr is not None:
            self._live[ptr].fill_(self.byte)
            self._torch.cuda.synchronize()
        return ptr


def _vacuum(memory=None, seed=5):
    g = pic.Sim(*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM, periodic_x=False, precision="fp32", window=(1.0, 0.0),
                memory=memory)
    F = 0.1 * np.random.default_rng(seed).standard_normal((9,) + SHAPE)
    F[6:] = 0.0
    g.set_fields(F)
    return g


def _plasma():
    g = pic.Sim(*SHAPE, LAM / 8, LAM / 3, LAM / 2, LAM, periodic_x=False, precision="fp32", window=(1.0, 0.0))
    g.add_species([-1.0, 1.0], [0.01, 0.01], 1)
    return g


@pytest.mark.parametrize("byte", [0x3f, 0xcf])
def test_member_without_particles_and_with_smaller_tiles(byte):
    single, member, other = _vacuum(), _vacuum(_DirtyMemory(byte)), _plasma()
    pic.pic_set_tiles(member.h, 2, 3, 2)  # more tiles than at creation
    b = pic.pic_batch_create([member.h, other.h])
    try:
        pic.pic_batch_step(b, 3)
        pic.pic_batch_step(b, 2)
        single.step(5)
        assert member.info()["np"] == 0 and member.info()["step"] == 5
        for c in range(9):
            assert np.array_equal(member.field(c), single.field(c)), pic.COMPONENTS[c]
    finally:
        pic.pic_batch_destroy(b)


def test_field_set_on_a_running_member():
    single, member = _vacuum(), _vacuum()
    b = pic.pic_batch_create([member.h])
    new = 0.1 * np.random.default_rng(9).standard_normal((2,) + SHAPE)
    try:
        pic.pic_batch_step(b, 3)
        single.step(3)
        for s in (member, single):
            s.set_field(1, new[0])  # Ey
            s.set_field(5, new[1])  # Bz
        pic.pic_batch_step(b, 3)
        single.step(3)
        for c in range(9):
            assert np.array_equal(member.field(c), single.field(c)), pic.COMPONENTS[c]
    finally:
        pic.pic_batch_destroy(b)
