"""The field read-outs of the C ABI: a packed selection (lbm_read_fields) equals
the fields read one by one, also where what follows a one-byte field of an odd
number of cells starts at an odd byte, in host and device memory; a destination
per field (lbm_read_fields_each) of any alignment; what both refuse."""
import ctypes as C

import numpy as np
import pytest

import inputs
from paper_1708_01613_gb300 import Simulation, load_library, make_config
from paper_1708_01613_gb300.lbm import FIELDS, LBM_EINVAL, LBM_OK

pytestmark = pytest.mark.gpu

RL, RG = inputs.RHO_LIQ_G55, inputs.RHO_GAS_G55
ORDER = sorted(FIELDS, key=lambda n: FIELDS[n][0])


def box(storage, comps, barrier):
    nx, ny = 121, 51  # an odd number of cells
    sim = Simulation(make_config(nx, ny, storage=storage, barrier=barrier, relabel_every=2, rho_ref=RL, components=comps,
                                 G=-1.0 if comps == 2 else -5.5, G_mg=2.5 if comps == 2 else 0.0, rupture_eps=1e-3))
    if comps == 2:
        sim.init_density(inputs.noise_density(nx, ny, seed=3), inputs.noise_density(nx, ny, seed=4, rho_mean=0.6))
    else:
        sim.init_bubbles([[48.0, 25.0, 11.0], [73.0, 25.5, 11.0]], RL, RG, 4.0)
    sim.step(3)
    return sim


def selections():
    yield ORDER
    yield ["mask", "pops"]
    yield ["ux", "mask", "rho_gas"]
    yield ["rho", "open", "pops", "rho_gas"]
    yield ["label", "owner", "mask", "open"]


@pytest.mark.parametrize("storage,comps,barrier", [("f32", 1, True), ("f16", 1, True), ("bf16", 1, False), ("f32", 2, True)])
@pytest.mark.parametrize("device,shift", [(False, 0), (True, 0), (True, 1), (True, 2)])
def test_packed_selection(storage, comps, barrier, device, shift):
    import torch

    sim = box(storage, comps, barrier)
    lib = load_library()
    one = {n: sim.read(n)[n] for n in ORDER}
    for names in selections():
        bits = sum(FIELDS[n][0] for n in names)
        total = int(lib.lbm_fields_bytes(sim.handle, bits))
        assert total == sum(one[n].nbytes for n in names)
        buf = torch.full((total + shift + 16,), 0xA5, dtype=torch.uint8, device="cuda" if device else "cpu")
        torch.cuda.synchronize()
        assert lib.lbm_read_fields(sim.handle, bits, C.c_void_p(buf.data_ptr() + shift), total, int(device)) == LBM_OK
        raw = buf.cpu().numpy()
        at = shift
        for n in sorted(names, key=ORDER.index):
            got = np.frombuffer(raw[at:at + one[n].nbytes].tobytes(), one[n].dtype).reshape(one[n].shape)
            assert np.array_equal(got, one[n]), (names, n)
            at += one[n].nbytes
        assert (raw[:shift] == 0xA5).all() and (raw[at:] == 0xA5).all()


@pytest.mark.parametrize("comps", [1, 2])
def test_destination_of_each_field_at_any_byte(comps):
    import torch

    sim = box("f32", comps, True)
    lib = load_library()
    one = {n: sim.read(n)[n] for n in ORDER}
    bufs = [torch.full((one[n].nbytes + 8,), 0x5A, dtype=torch.uint8, device="cuda") for n in ORDER]
    shifts = [k % 4 for k in range(1, len(ORDER) + 1)]
    torch.cuda.synchronize()
    ptrs = (C.c_void_p * len(ORDER))(*[b.data_ptr() + s for b, s in zip(bufs, shifts)])
    assert lib.lbm_read_fields_each(sim.handle, sum(FIELDS[n][0] for n in ORDER), ptrs, 1) == LBM_OK
    for n, b, s in zip(ORDER, bufs, shifts):
        raw = b.cpu().numpy()
        assert raw[s:s + one[n].nbytes].tobytes() == one[n].tobytes(), n
        assert (raw[:s] == 0x5A).all() and (raw[s + one[n].nbytes:] == 0x5A).all()


def test_refused_selections():
    sim = box("f32", 1, True)
    lib = load_library()
    rho = FIELDS["rho"][0]
    out = np.zeros((51, 121), np.float32)
    dst = C.c_void_p(out.ctypes.data)
    beyond = 2 * max(FIELDS[n][0] for n in ORDER)
    for bits in (0, beyond, rho | beyond):
        assert lib.lbm_read_fields(sim.handle, bits, dst, out.nbytes, 0) == LBM_EINVAL
        assert lib.lbm_read_fields_each(sim.handle, bits, (C.c_void_p * 2)(dst, dst), 0) == LBM_EINVAL
    assert lib.lbm_read_fields(sim.handle, rho, dst, out.nbytes - 1, 0) == LBM_EINVAL
    assert lib.lbm_read_fields(sim.handle, rho, None, out.nbytes, 0) == LBM_EINVAL
    assert lib.lbm_read_fields_each(sim.handle, rho, None, 0) == LBM_EINVAL
    assert lib.lbm_read_fields_each(sim.handle, rho | FIELDS["p"][0], (C.c_void_p * 2)(dst, None), 0) == LBM_EINVAL
    assert not out.any()
    assert lib.lbm_read_fields_each(sim.handle, rho, (C.c_void_p * 1)(dst), 0) == LBM_OK and out.all()
