"""Host code of the library on a CUDA runtime without a GPU (fake_cudart.c): what its calls queue,
on which stream, what they leave queued when they return, and what they do with the values that
kernels leave for the host.  Each test is a program of its own (the fake is preloaded)."""
import os
import subprocess
import sys
import textwrap

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PREAMBLE = """
    import ctypes, sys
    import numpy as np
    sys.path.insert(0, {root!r})
    from paper_2304_10061_gb300 import Allegro, AllegroError
    from synth import ARCHS, make_weights, weights_to_blob

    fake = ctypes.CDLL({fake!r})
    for f in (fake.fake_pending, fake.fake_total, fake.fake_pending_all):
        f.restype = ctypes.c_long
    fake.fake_pending.argtypes = fake.fake_total.argtypes = [ctypes.c_void_p]
    HOOK = ctypes.CFUNCTYPE(None, ctypes.c_char_p, ctypes.POINTER(ctypes.c_void_p))

    def param(args, k, ctype=ctypes.c_void_p):
        return ctype.from_address(args[k]).value

    ARCH = ARCHS["c1"]
    model = Allegro(weights_to_blob(ARCH, make_weights(ARCH, 0)))
    N = 64
    rng = np.random.default_rng(0)
    cell = np.eye(3) * 8.62
    pos = rng.uniform(0.0, 8.62, (N, 3))
    types = (np.arange(N) % 2).astype(np.int32)

    def evaluate():
        out = [np.zeros(k) for k in (model.n_struct, N, 3 * N, 9 * model.n_struct)]
        model._check(model._L.allegro_energy_forces(model._ctx, *[a.ctypes.data for a in out]))
        return out

    def status(call):
        try:
            call()
        except AllegroError as e:
            return e.status
        return 0
"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    import __graft_entry__ as g
    from paper_2304_10061_gb300.build import nvcc
    g.build()
    so = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc()))), "include")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-I", include, os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", so],
                   check=True)

    def run(script):
        text = textwrap.dedent(PREAMBLE).format(root=ROOT, fake=so) + textwrap.dedent(script)
        r = subprocess.run([sys.executable, "-c", text], env=dict(os.environ, LD_PRELOAD=so), capture_output=True,
                           text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]

    return run


def test_nothing_on_the_default_stream(fake):
    """The context's stream does not wait for the default stream: uploads on it have ended when
    allegro_create returns, and no clear is queued on it (a workspace cleared there was cleared
    while the first kernels wrote it)."""
    fake("""
        assert fake.fake_pending(None) == 0, fake.fake_pending(None)
        before = fake.fake_total(None)
        model.neighbors(pos, types, cell)
        evaluate()
        assert fake.fake_total(None) == before, fake.fake_total(None) - before
    """)


def test_calls_leave_nothing_queued(fake):
    """Every call has waited for what it queued when it returns, refused ones too: the stream may be
    changed and the caller's arrays may go."""
    fake("""
        def check(want, call):
            assert status(call) == want
            assert fake.fake_pending_all() == 0, fake.fake_pending_all()

        flat, nan = np.diag([8.62, 8.62, 0.0]), np.diag([8.62, 8.62, np.nan])
        offs = np.array([0, 30, N], np.int64)
        check(0, lambda: model.reserve(1000, 5000))
        check(1, lambda: model.neighbors(pos, types, flat))
        check(1, lambda: model.neighbors(pos, types, nan))
        check(1, lambda: model.neighbors(pos, types, None, [1, 0, 0]))
        check(1, lambda: model.neighbors_local(10, pos, types, flat))
        check(1, lambda: model.neighbors_batched(offs, pos, types, np.stack([cell, flat])))
        check(1, lambda: model.neighbors_batched(offs, pos, types, None, [1] * 6))
        check(1, lambda: model.md_verlet(pos.copy(), np.zeros((N, 3)), types, [1.0, 1.0], 1.0, 2, flat))
        check(0, lambda: model.neighbors_batched(offs, pos, types))
        check(0, evaluate)
        check(0, lambda: model.neighbors(pos, types, cell))
        check(0, evaluate)
        check(0, model.get_neighbors)
        check(0, lambda: model.md_verlet(pos.copy(), np.zeros((N, 3)), types, [1.0, 1.0], 1.0, 2, cell))
    """)


@pytest.mark.parametrize("skin", [0.0, 1.0])
@pytest.mark.parametrize("bit,want", [(1, 5), (8, 6)])
def test_md_reports_every_steps_errors(fake, bit, want, skin):
    """A device wait that ran out, or a non-finite energy or force, ends the MD run whichever of its
    evaluations raised it, and is gone in the next call."""
    fake(f"""
        BIT, WANT, SKIN = {bit}, {want}, {skin}
    """ + """
        seen = [0]

        @HOOK
        def hook(name, args):
            if b"struct_reduce_kernel" in name:   # the last kernel of an evaluation; its last parameter is the error word
                seen[0] += 1
                if seen[0] == at:
                    ctypes.c_int.from_address(param(args, 10)).value |= BIT

        fake.fake_on_launch(hook)
        model.set_md_skin(SKIN)
        for at in range(1, 6):   # evaluations 1..4 of three steps; 5: none of them
            seen[0] = 0
            got = status(lambda: model.md_verlet(pos.copy(), np.zeros((N, 3)), types, [1.0, 1.0], 1.0, 3, cell))
            assert got == (WANT if at < 5 else 0), (at, got)
            at = 0
            assert status(lambda: model.neighbors(pos, types, cell)) == 0
            assert status(evaluate) == 0
    """)


def test_profile_counts_the_edges_of_its_own_list(fake):
    """Bytes of the fill and column passes: those of the list they wrote, whatever list came before,
    and none for a pass that found its list too long for the arrays."""
    fake("""
        @HOOK
        def hook(name, args):
            if b"scan_one_kernel" in name and param(args, 4):   # the scan of the row counts leaves the total
                ctypes.c_int.from_address(param(args, 4)).value = edges

        fake.fake_on_launch(hook)
        offs = np.array([0, 30, N], np.int64)
        for build, label in ((lambda: model.neighbors(pos, types, cell), "nb_search_fill"),
                             (lambda: model.neighbors_batched(offs, pos, types), "nb_brute_fill")):
            for edges in (1000, 700, 90000, 20, 200000):
                model.profile(True)
                assert build() == edges
                rep, _ = model.profile_report()
                model.profile(False)
                assert rep[label]["bytes"] == 44 * edges + 64 * N, (edges, rep[label])
                assert rep["nb_csc"]["bytes"] == 16 * edges + 16 * N, (edges, rep["nb_csc"])
            edges = 100
            build()
    """)


@pytest.mark.parametrize("precision", ["fp32", "tf32", "bf16", "fp8"])
def test_every_array_a_gemm_names_is_there(fake, precision):
    """MLPs of 1 to 5 layers: each tensor map of an evaluation (operands, outputs, pre-activations) lies in an
    allocation.  (BF16 latent MLPs of three layers and more wrote a layer at address zero.)"""
    fake(f"""
        PRECISION = {precision!r}
    """ + """
        from synth import Arch

        @HOOK
        def hook(name, args):
            if b"scan_one_kernel" in name and param(args, 4):
                ctypes.c_int.from_address(param(args, 4)).value = 3000

        fake.fake_on_launch(hook)
        for layers, lmax, channels in ((1, 1, 16), (1, 2, 64), (2, 1, 32), (2, 2, 64), (2, 2, 32), (3, 2, 64), (2, 3, 16)):
            for depth in range(1, 6):
                for widths in ((64, 128, 256, 32, 96), (40, 24, 192, 256, 16), (256, 512, 64, 320, 128)):
                    if max(widths[:depth]) > 256 and PRECISION == "bf16" and channels * (lmax + 1) % 64:
                        continue   # (refused)
                    arch = Arch(n_species=2, lmax=lmax, n_layers=layers, channels=channels, two_body=widths[:depth],
                                latent=widths[:depth][::-1], edge=(8,))
                    model = Allegro(weights_to_blob(arch, make_weights(arch, 0)), precision=PRECISION)
                    assert model.neighbors(pos, types, cell) == 3000
                    evaluate()
                    model.close()
    """)
