"""The plan of a tall lattice: the z-chunk of least modelled cost among all ceil(nz / n), found without
trying every n (lbm_create of a tall lattice would take as long as that)."""
import time

import pytest

pytestmark = pytest.mark.gpu


def _params(nx, ny, nz):
    from paper_2201_06039_gb300 import lbm
    p = lbm.lbm_params_default()
    p.nx, p.ny, p.nz = nx, ny, nz
    return p


@pytest.mark.parametrize("dims", [(4, 4, 1), (33, 20, 2), (40, 10, 97), (64, 64, 96), (16, 16, 2003), (8, 8, 9973)])
def test_no_z_chunk_beats_the_plans(dims):
    from paper_2201_06039_gb300 import lbm
    nz = dims[2]
    lat = lbm.Lattice(_params(*dims))
    shape, zchunk, items, _ = lat.plan
    w, h = lbm.lbm_plan_shapes()[shape]
    tiles = -(-dims[0] // w) * -(-dims[1] // h)
    assert items == tiles * -(-nz // zchunk)
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count

    def cost(zc):   # rounds of items on the SMs, an item as long as its planes and 2.1 more
        return -(-tiles * -(-nz // zc) // sms) * (zc + 2.1)
    assert cost(zchunk) <= min(cost(-(-nz // n)) for n in range(1, nz + 1)) * (1 + 1e-12)
    lat.close()


def test_creating_a_tall_lattice_takes_no_time_of_its_own():
    """6 x 490 chunk lengths of 60000 planes against 6 x 60000: lbm_create took 2.6 ms here, 13 us on a cube."""
    from paper_2201_06039_gb300 import lbm

    def create(dims):
        best = 1e9
        p = _params(*dims)
        ws = lbm.Lattice(p)   # its workspace is used by every context below
        for _ in range(7):
            t = time.perf_counter()
            ctx = lbm.lbm_create(p)
            best = min(best, time.perf_counter() - t)
            lbm.lbm_destroy(ctx)
        ws.close()
        return best
    tall, cube = create((4, 4, 60000)), create((32, 32, 32))
    print(f"tall {1e6 * tall:.0f} us, cube {1e6 * cube:.0f} us")
    assert tall < 1e-3 + cube, (tall, cube)
