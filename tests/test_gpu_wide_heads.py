"""Adjoint heads of wide MLPs: in the GEMM's epilogue or in a kernel of their own, the same bits.

Which form a call takes depends on its rows.  A batch of k copies of one cluster has the same
activations, and so the same per-tensor FP8 scales, for every k, so each copy's results are those of the
cluster alone, whatever form its head took.  The cluster alone has too few row blocks for the fused
form; two copies fill the SMs with one row block each, four with two (so the barriers between the two
warps of a row are used again, and partial sums cross column tiles)."""
import numpy as np
import pytest

from gpu_util import lib_model
from synth import Arch, lattice_box, make_weights, weights_to_blob

pytestmark = pytest.mark.gpu

ARCHS = {
    "512": Arch(n_species=2, lmax=2, n_layers=3, channels=64, two_body=(64, 512), latent=(512,), edge=(16,)),
    "768_two_layers": Arch(n_species=2, lmax=1, n_layers=2, channels=64, two_body=(96, 512), latent=(768, 768), edge=()),
    "1024": Arch(n_species=2, lmax=1, n_layers=2, channels=64, two_body=(64, 1024), latent=(1024,), edge=()),
}
ROWS = 75 * 128   # one copy: 75 row blocks of 128 edges


def _cluster(r_c):
    """A cluster of just under ROWS edges, no cell."""
    s = lattice_box(700, (700 / 0.1) ** (1 / 3), seed=9)
    order = np.argsort(np.linalg.norm(s.pos - s.pos.mean(0), axis=1))
    d = np.linalg.norm(s.pos[order][:, None] - s.pos[order][None], axis=-1)
    close = np.tril((d < r_c) & (d > 0))
    n = int(np.searchsorted(2 * np.cumsum(close.sum(1)), ROWS))
    return s.pos[order[:n]], (np.arange(n) % 2).astype(np.int32)


@pytest.mark.parametrize("prec", ["fp8", "bf16", "tf32"])
@pytest.mark.parametrize("name", list(ARCHS))
def test_copies_of_a_cluster(name, prec):
    arch = ARCHS[name]
    pos, types = _cluster(arch.r_c)
    n = len(pos)
    m = lib_model(weights_to_blob(arch, make_weights(arch, 5)), precision=prec)
    forms, first = set(), None
    for k in (1, 2, 4):
        edges = m.neighbors_batched(np.arange(k + 1, dtype=np.int64) * n, np.tile(pos, (k, 1)), np.tile(types, k))
        assert 70 * 128 * k < edges <= ROWS * k
        m.profile(True)
        out = {q: v.cpu().numpy() for q, v in m.energy_forces().items()}
        rep, _ = m.profile_report()
        m.profile(False)
        forms.add(rep["head_bwd"]["launches"])   # (the last layer's is always one of them)
        if first is None:
            first = out
        for b in range(k):
            at = slice(b * n, (b + 1) * n)
            np.testing.assert_array_equal(out["E_atom"][at], first["E_atom"])
            np.testing.assert_array_equal(out["F"][at], first["F"])
    m.close()
    assert len(forms) > 1, forms
