"""Contexts of different sizes in several host threads.

The dynamic shared-memory limit of a kernel belongs to the function, not to the
call or the thread: a launch that needs more than a limit which another thread
has lowered is refused.  Every kernel whose request varies between contexts is
used here by contexts of different sizes at once; each thread's results have the
bits of the same calls alone.
"""
import threading

import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def run_threads(targets):
    errors = []

    def guard(f):
        try:
            f()
        except BaseException as e:  # noqa: BLE001 -- reported by the main thread
            errors.append(e)

    ts = [threading.Thread(target=guard, args=(f,)) for f in targets]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def test_cs_reconstructions_of_different_sizes():
    import paper_2605_09590_gb300 as pico
    jobs = []
    for n, levels, repeats in ((320, 4, 12), (64, 4, 40), (384, 4, 10), (64, 3, 40)):
        S = synth.coil_maps(n, n, 2, 1)
        mask = (np.random.default_rng(n).random((n, n)) < 0.6).astype(np.uint8)
        op = pico.Operator(S, mask=mask, power_iters=10, max_batch=1)
        x0 = torch.from_numpy(synth.phantom(n, 1).astype(np.complex64)).cuda().reshape(1, n, n)
        b = op.forward(x0)[0].contiguous()
        alone = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        pico.pico_cs_recon(op.ctx, b, 1e-3, 40, levels, alone)
        op.sync()
        jobs.append((op, b, levels, repeats, alone))
    start = threading.Barrier(len(jobs))

    def worker(op, b, levels, repeats, alone):
        x = torch.empty_like(alone)
        start.wait()
        for _ in range(repeats):
            pico.pico_cs_recon(op.ctx, b, 1e-3, 40, levels, x)
        op.sync()
        assert torch.equal(x, alone)

    run_threads([lambda j=j: worker(*j) for j in jobs])
    for j in jobs:
        j[0].close()


def gram_op(ny, nx=32, nc=4):
    import paper_2605_09590_gb300 as pico
    op = pico.Operator(synth.coil_maps(ny, nx, nc, 1), mask=synth.mask_pe(ny, 2, 8), power_iters=0, max_batch=4)
    op.set_tuning(gram_min_batch=1)
    return op


@pytest.mark.parametrize("solver", ["global", "columns"])
def test_gram_kernels_after_a_smaller_context_of_another_thread(solver, monkeypatch):
    """320 rows take 209 KB of shared memory per block, 256 rows 164 KB."""
    monkeypatch.setenv("PICO_COLCG_PERSIST", "0")   # the per-update kernel
    rng = np.random.default_rng(4)

    def solve(op):
        op.set_solver(solver)
        x = rhs[op.ny]
        y = op.cg(x, 6) if solver == "columns" else op.apply_normal(x)
        op.sync()
        return y

    rhs = {ny: torch.from_numpy((rng.standard_normal((2, ny, 32)) + 1j * rng.standard_normal((2, ny, 32)))
                                .astype(np.complex64)).cuda() for ny in (320, 256)}
    large, small = gram_op(320), gram_op(256)
    alone = solve(large)
    run_threads([lambda: solve(small)])
    assert torch.equal(solve(large), alone)
    large.close()
    small.close()


def test_gram_setups_of_different_sizes():
    """The set-up keeps a column's sensitivities in shared memory: coils x rows x 8 bytes.

    Changing the contraction depth builds the operator anew."""
    shapes = ((128, 3), (256, 64), (128, 5), (320, 70))
    start = threading.Barrier(len(shapes))
    rng = np.random.default_rng(5)
    cases = []
    for ny, nc in shapes:
        x = torch.from_numpy((rng.standard_normal((1, ny, 16)) + 1j * rng.standard_normal((1, ny, 16)))
                             .astype(np.complex64)).cuda()
        op = gram_op(ny, 16, nc)
        cases.append((op, x, op.apply_normal(x)))
        op.sync()

    def worker(op, x, alone):
        start.wait()
        for _ in range(1000):
            op.set_tuning(gram_kc=8)
            op.set_tuning(gram_kc=16)
        y = op.apply_normal(x)
        op.sync()
        assert torch.equal(y, alone)

    run_threads([lambda c=c: worker(*c) for c in cases])
    for c in cases:
        c[0].close()
