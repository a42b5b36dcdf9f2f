"""Checkpoint and resume through the C ABI (GPU), and host-side rejection of
corrupted checkpoints (the fault is injected into the host buffer; nothing
invalid reaches the device)."""
import numpy as np
import pytest

from paper_1401_4076_gb300 import mucal as m

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_1401_4076_gb300 import _build_ext
    _build_ext.build_library()
    m.load_library()


DESCS = [(2, 24, 60, 70, 0, 0, 5), (3, 10, 90, 33, 0, 0, 900)]


def test_resume_is_bit_exact():
    with m.Mucal(DESCS) as a:
        for it in range(2):
            a.run_iteration(30, it)
            for s in range(2):
                a.update_weights(s)
        cks = [a.checkpoint(s) for s in range(2)]
        a.run_iteration(30, 2)
        Ha = [a.histogram(s) for s in range(2)]
        Wa = [a.update_weights(s)[0] for s in range(2)]
        Ea = [a.walker_state(s, 3)[2] for s in range(2)]
    with m.Mucal(DESCS) as b:
        for s in range(2):
            b.restore(s, cks[s])
        b.run_iteration(30, 2)
        for s in range(2):
            np.testing.assert_array_equal(b.histogram(s), Ha[s])
            np.testing.assert_array_equal(b.update_weights(s)[0], Wa[s])
            assert b.walker_state(s, 3)[2] == Ea[s]


def test_corrupted_checkpoints_are_rejected():
    with m.Mucal(DESCS[:1]) as a:
        a.run_iteration(10, 0)
        ck = a.checkpoint(0)
        H_before = a.histogram(0)
        info = a.info[0]
        W, V, words = info["n_walkers"], info["V"], (info["V"] + 31) // 32
        hdr = len(ck) - (W * words * 4 + W * V * 2 + W * 4 + info["n_bins"] * 17)
        bad = ck.copy()                     # a list entry off the lattice
        bad[hdr + W * words * 4: hdr + W * words * 4 + 2] = np.frombuffer(
            np.uint16(V + 5).tobytes(), np.uint8)
        with pytest.raises(m.MucalError) as ei:
            a.restore(0, bad)
        assert ei.value.code == m.MUCAL_ERR_INVALID_ARG
        bad = ck.copy()                     # an energy outside the window
        off = hdr + W * words * 4 + W * V * 2
        bad[off: off + 4] = np.frombuffer(np.int32(5).tobytes(), np.uint8)
        with pytest.raises(m.MucalError):
            a.restore(0, bad)
        bad = ck.copy()                     # wrong magic
        bad[0] ^= 0xFF
        with pytest.raises(m.MucalError):
            a.restore(0, bad)
        with pytest.raises(m.MucalError):   # wrong size
            a.restore(0, ck[:-1])
        # nothing was changed: the state still continues as before
        a.restore(0, ck)
        a.run_iteration(10, 0)
        assert a.histogram(0).sum() == H_before.sum()


def test_allocation_failure_is_reported_cleanly():
    """A system far larger than the device: the allocation fails inside the
    library, which returns MUCAL_ERR_OOM and frees what it had taken."""
    huge = (2, 1024, 100, 1 << 22, 0, 0, 0)      # bitsets alone would need 512 GiB
    with pytest.raises(m.MucalError) as ei:
        m.Mucal([huge])
    assert ei.value.code == m.MUCAL_ERR_OOM
    with m.Mucal([(2, 8, 10, 4, 0, 0, 1)]) as ok:    # the device is still usable
        ok.run_iteration(5, 0)
        assert ok.histogram(0).sum() == 4 * 5 * 10


@pytest.mark.parametrize("desc,launch", [
    # the table staged, rows per walker, masks from global memory
    ((2, 12, 40, 9, 0, 0, 4), dict(kernel=m.MUCAL_KERNEL_FIELD, lanes_per_walker=8, walkers_per_block=4)),
    ((2, 90, 2501, 5, 0, 0, 7), dict(kernel=m.MUCAL_KERNEL_GROUP, lanes_per_walker=8, walkers_per_block=4)),
    ((3, 17, 1201, 5, 0, 0, 8), dict(kernel=m.MUCAL_KERNEL_FIELD, lanes_per_walker=16, walkers_per_block=2)),
    ((3, 30, 1201, 11, 0, 0, 9), dict(kernel=m.MUCAL_KERNEL_FIELD, lanes_per_walker=8, walkers_per_block=8)),
    ((3, 30, 1201, 64, 0, 0, 9), dict(kernel=m.MUCAL_KERNEL_GROUP, lanes_per_walker=8, walkers_per_block=64)),
], ids=lambda x: f"L{x[1]}-{x[3]}" if isinstance(x, tuple) else None)
def test_rounds_on_a_restored_state_that_disagrees_with_itself(desc, launch):
    """Lists with repeated sites and bitsets of other sites pass the restore's
    checks.  The rounds with several commits then give no chain that means
    anything, but count every attempt at an energy of the window."""
    d, L, N, W, _, _, seed = desc
    V = L ** d
    words = (V + 31) // 32
    rng = np.random.default_rng(seed)
    with m.Mucal([desc]) as mc:
        mc.set_launch(bits_in_smem=1, thr_window=0, multi_commit=1, **launch)
        assert mc.launch()["multi_commit"] == 1
        ck = mc.checkpoint(0).copy()
        at = 64                                        # the header's bytes
        bits = ck[at:at + 4 * W * words].view(np.uint32).reshape(W, words)
        S = ck[at + 4 * W * words:at + 4 * W * words + 2 * W * V].view(np.uint16).reshape(W, V)
        bits[:, :V // 32] = rng.integers(1 << 32, size=(W, V // 32), dtype=np.uint32)
        S[:, ::2] = S[:, :1]
        for beta in (0.0, 1.0):
            mc.restore(0, ck)
            mc.set_weights(0, -beta * np.arange(-d * N, 1, dtype=np.float64))
            mc.run_iteration(3, 0)
            assert mc.histogram(0).sum() == 3 * N * W
            E = [mc.walker_state(0, w)[2] for w in range(W)]
            assert min(E) >= -d * N and max(E) <= 0
