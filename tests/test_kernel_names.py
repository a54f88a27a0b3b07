"""The step kernels' names tell them apart: results kept by name (bench.py's by_kernel) must not fall
together."""
from paper_1909_08406_gb300 import lb


def test_every_kernel_has_its_own_name():
    ids = [lb.LB_KERNEL_DIRECT1, lb.LB_KERNEL_DIRECT2, lb.LB_KERNEL_DIRECT2R, lb.LB_KERNEL_STAGED,
           lb.LB_KERNEL_WARPSPEC, lb.LB_KERNEL_DIRECT2X, lb.LB_KERNEL_DIRECT2XL]
    names = [lb.KERNEL_NAMES[k] for k in ids]
    assert len(set(names)) == len(ids)
