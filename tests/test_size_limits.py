"""Sizes that 32-bit numbering cannot hold are refused with EINVAL before
anything is allocated or launched."""
import pytest

from paper_1502_06447_gb300 import build, ecmc


@pytest.fixture(scope="module", autouse=True)
def _build():
    build.build()


@pytest.mark.parametrize("dims", [(1024, 1024, 512), (2**31 - 1, 2**31 - 1, 2**31 - 1)])
def test_replica_of_2_29_beads_is_refused(dims):
    """Staging keeps a bead's id in 29 bits (refused before a device is
    touched, so this runs on the CPU)."""
    with pytest.raises(ecmc.EcmcError) as e:
        ecmc.Batch([dict(dims=(8, 8, 8), spacing=1.05, N=8), dict(dims=dims, spacing=1.05, N=1)])
    assert e.value.code == -1 and "2^29" in str(e.value)


@pytest.mark.gpu
@pytest.mark.parametrize("kw,why", [
    (dict(tile_side=500.0), "cell grid"),                    # 5333^3 cells of 1.05 in the second replica
    (dict(tile_side=4.2, cell_side=100.0), "too many tiles"),  # 1333^3 tiles there
])
def test_batch_grids_past_31_bits_are_refused(kw, why):
    specs = [dict(dims=(8, 8, 8), spacing=100.0, N=1), dict(dims=(8, 8, 8), spacing=700.0, N=1)]
    b = ecmc.Batch(specs, seed=1)
    with pytest.raises(ecmc.EcmcError) as e:
        b.configure(dir_mode=ecmc.DIR_ISO, precision=ecmc.PREC_FP64, lanes=8, **kw)
    assert e.value.code == -1 and why in str(e.value)


@pytest.mark.gpu
def test_tiles_past_31_bits_are_refused():
    """Free spheres with a joint of one diameter: 1340^3 tiles of 1.0075 (the
    1285^3 cells of the box take 17 GB)."""
    with ecmc.Context.create_lattice((8, 8, 8), 168.75, 1, b_max=1.0) as ctx:
        with pytest.raises(ecmc.EcmcError) as e:
            ctx.configure(mode=ecmc.MODE_DOMAIN, precision=ecmc.PREC_FP64, tiles=(1340, 1340, 1340), cell_side=100.0)
        assert e.value.code == -1 and "too many tiles" in str(e.value)
