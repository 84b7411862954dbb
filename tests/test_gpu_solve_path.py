"""How the mixed form's solves run is decided once per chunk: a chunk with too many units for block-step
launches (more than n / 64, n >= 3000) stays with chains when it is cut into parts that by themselves are
below that number.  A part then launches at most the kernels that the whole chunk would, and the results are
the same bits."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2311_12134_gb300 import workload as wl

from ._util import ensure_built


def test_parts_keep_the_path_of_their_chunk():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()
    from paper_2311_12134_gb300 import binding as B
    # 2 atoms x 40 energies of 259 sites: 80 units of n = 4144, 64 < 80 <= 4 x 64
    w = wl.make_supercell(name="bcc2", kind="bcc", n_cells=1, a=5.42, counts=[1, 1], r_liz=3.0 * 5.42,
                          phases=[wl.PHASE_A, wl.PHASE_B], e_fermi=0.62, deltas=list(np.linspace(0.002, 0.004, 20)),
                          seed=3)
    lz = B.build_liz(w.pos, w.lattice, w.r_liz)
    assert 16 * lz.max_sites == 4144 and len(w.z) == 40
    need = B.tau_workspace_bytes(lz, w.lmax, len(w.z), B._prec("mixed"))[1]
    ws = torch.empty(need, dtype=torch.uint8, device="cuda")  # one chunk
    sp, ti = torch.as_tensor(w.species).cuda(), torch.as_tensor(w.tinv).cuda()
    launches, tau = {}, {}
    try:
        for streams in (1, 0):
            B.set_option("streams", streams)
            c0 = B.launch_count()
            t, st = B.tau_blocks(lz, w.lmax, sp, ti, w.z, "mixed", workspace=ws)
            launches[streams] = B.launch_count() - c0
            assert not np.any(st.cpu().numpy() & 0xff)
            tau[streams] = t.cpu().numpy()
    finally:
        B.set_option("streams", 0)
    assert launches[0] <= 2 * launches[1], launches
    assert np.array_equal(tau[0], tau[1])
