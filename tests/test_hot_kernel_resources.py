"""Resource budgets of the kernels that the calls of every size run (see
test_kernel_resources.py for the others): FP64 Tsit5 in integer products and with a
lane per component, FP32-mixed over packed segments, and the neural Robertson's
lane groups. Registers set how many CTAs fit per SM; spills are bounded by what
the measured throughputs include."""
import concurrent.futures as cf

import pytest

from tests.test_kernel_resources import find, resources


@pytest.fixture(scope="module")
def res():
    names = ("gs_tsit5_soft.cu", "gs_packed.cu", "gs_tsit5_group.cu", "gs_nrob.cu")
    with cf.ThreadPoolExecutor(len(names)) as ex:
        return dict(zip(names, ex.map(resources, names)))


# translation unit, parts of the kernel's name, most registers, most spill stores (bytes)
BUDGETS = [
    # 4 CTAs of 128 threads per SM: 128 registers
    ("gs_tsit5_soft.cu", ("record_soft_kernel", "Lorenz", "Lb1ELb1ELb0E"), 128, 64),
    ("gs_tsit5_soft.cu", ("record_soft_kernel", "VanDerPol", "Lb1ELb1ELb0E"), 128, 0),
    ("gs_tsit5_soft.cu", ("record_soft_kernel", "Lorenz", "Lb0ELb0ELb0E"), 128, 0),  # forward only
    ("gs_tsit5_soft.cu", ("reverse_k1_soft_kernel", "Lorenz", "Lb0ELb1ELi4E"), 128, 256),
    ("gs_tsit5_soft.cu", ("reverse_k1_soft_kernel", "VanDerPol", "Lb0ELb1ELi4E"), 128, 0),
    # 10 and 8 CTAs per SM: 48 and 64 registers
    ("gs_packed.cu", ("record_packed_kernel", "Lorenz", "Lb0ELi4E"), 48, 0),
    ("gs_packed.cu", ("record_packed_kernel", "VanDerPol", "Lb0ELi4E"), 48, 0),
    ("gs_packed.cu", ("reverse_packed_kernel", "Lorenz"), 64, 64),
    ("gs_packed.cu", ("reverse_packed_kernel", "VanDerPol"), 64, 0),
    # small ensembles, one CTA per SM or a few: no spills
    ("gs_tsit5_group.cu", ("record_kernel", "LorenzGroup", "EdLb1ELb1ELb0E"), 168, 0),
    ("gs_tsit5_group.cu", ("reverse_k1_kernel", "LorenzGroup", "EdLb0ELb1E"), 168, 0),
    ("gs_tsit5_group.cu", ("record_kernel", "VanDerPolGroup", "EdLb0ELb0ELb0E"), 128, 0),  # (a context's)
    ("gs_tsit5_group.cu", ("reverse_k1_kernel", "VanDerPolGroup", "EdLb0ELb0E"), 128, 0),
    ("gs_nrob.cu", ("record_kernel", "NeuralRobertsonGroup", "EdLb1ELb1ELb0E"), 255, 0),
    ("gs_nrob.cu", ("reverse_k1_kernel", "NeuralRobertsonGroup", "EdLb0ELb1E"), 255, 2048),
]


@pytest.mark.parametrize("src,parts,most,spills", BUDGETS, ids=lambda v: "-".join(v) if isinstance(v, tuple) else None)
def test_budget(res, src, parts, most, spills):
    regs, spill = find(res[src], *parts)
    assert regs <= most and spill <= spills, (regs, spill)
