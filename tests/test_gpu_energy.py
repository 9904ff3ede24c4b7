"""Energies of int8 configurations (Eq. 1) against a numpy sum over the bonds, exactly, at
every load width the kernel picks: rows of 2, 4 and 16 bytes and odd base addresses."""
import numpy as np
import pytest

from paper_2501_17267_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    torch.cuda.init()
    from paper_2501_17267_gb300 import sg
    return sg


def energies(L, J3, spins):
    J = J3.reshape(L, L, L, 3).astype(np.int64)
    s = spins.reshape(-1, L, L, L).astype(np.int64)
    return sum((J[..., d] * s * np.roll(s, -1, axis=3 - d)).sum(axis=(1, 2, 3)) for d in range(3))


# (16, 4, 2 or 1 bytes a load; n below, at and above a block's 32 configurations)
@pytest.mark.parametrize("L,n,offset", [(2, 1, 0), (2, 70, 1), (4, 33, 0), (6, 32, 0), (6, 5, 3), (10, 31, 2), (12, 65, 0),
                                        (16, 100, 0), (16, 7, 4), (16, 9, 1), (48, 3, 0), (64, 40, 0), (34, 4, 0)])
def test_energies_at_every_load_width(sg, L, n, offset):
    import torch
    J3 = wl.random_couplings(L + n, L)
    spins = wl.random_spins(3 * L + n, (n, L ** 3))
    inst = sg.Instance.from_couplings(L, J3)
    flat = torch.zeros(n * L ** 3 + offset, dtype=torch.int8, device="cuda")
    view = flat[offset:].view(n, L ** 3)
    view.copy_(torch.from_numpy(spins))
    want = energies(L, J3, spins)
    assert np.array_equal(sg.energy(inst, view), want)
    assert np.array_equal(sg.energy(inst, spins), want)
    out = torch.empty(n, dtype=torch.int64, device="cuda")
    sg.energy_noalloc(L, torch.from_numpy(J3).cuda(), view, out)
    assert np.array_equal(out.cpu().numpy(), want)


@pytest.mark.parametrize("L,values", [(4, (0,)), (6, (2, -2)), (16, (3, -127, 127, -128))])
def test_every_value_that_is_no_spin_is_counted(sg, L, values):
    import torch
    inst = sg.Instance.from_couplings(L, wl.random_couplings(1, L))
    spins = wl.random_spins(2, (3, L ** 3))
    for k, v in enumerate(values):
        spins[k % 3, (7 * k * L + 5) % L ** 3] = v
    with pytest.raises(sg.SGError, match=f"{len(values)} spin values"):
        sg.energy(inst, torch.from_numpy(spins).cuda())


# (16, 4, 2 and 1 bytes a load) n such that a block walks over several configurations (3, 7, 7 and
# 14 with 152 SMs) and the last one over fewer; then more than 128 a block could have
@pytest.mark.parametrize("L,n,offset", [(64, 103, 0), (36, 320, 0), (34, 200, 0), (34, 200, 1), (2, 128 * 8 * 152 + 77, 0),
                                        (2, 128 * 8 * 152 + 77, 1)])
def test_energies_of_many_configurations_a_block(sg, L, n, offset):
    test_energies_at_every_load_width(sg, L, n, offset)
