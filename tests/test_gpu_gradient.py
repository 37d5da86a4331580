"""Gradient of the exit-wave misfit (Sec. 2.1) on the GPU against the oracle,
central finite differences and autograd; the plain gradient baseline."""
import numpy as np
import pytest

import oracle as O
import synth
from emg_cases import Case, c64, gpu_params, make_context, oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch as t

    assert t.cuda.is_available()
    return t


def _gpu_gradient(lib, torch, ctx, z, q):
    zd = torch.from_numpy(c64(z)).cuda()
    qd = torch.from_numpy(c64(q)).cuda()
    gz = torch.empty_like(zd)
    gq = torch.empty_like(qd)
    phi = lib.emg_misfit_gradient(ctx.ctx, zd.data_ptr(), qd.data_ptr(), gz.data_ptr(), gq.data_ptr(), True)
    torch.cuda.synchronize()
    return phi, gz.cpu().numpy().astype(np.complex128), gq.cpu().numpy().astype(np.complex128)


@pytest.mark.parametrize("chunk", [6, 0])
@pytest.mark.parametrize("m", [16, 32, 64, 128, 256])
def test_gradient_matches_the_oracle(lib, torch, m, chunk):
    """16 positions in chunks of 6 (sums over several launches), and in the
    automatic chunk (one launch here)."""
    case = Case(n=2 * m + 40, m=m, side=4, noise_peak=1e4, seed=40 + m)
    p = oracle_params(minibatch=6)
    ctx = make_context(lib, case, p)
    lib.emg_set_gradient_chunk(ctx.ctx, chunk)
    phi, gz, gq = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
    ctx.close()
    phi_o, gz_o, gq_o = O.misfit_gradients(case.q0.astype(np.complex128), case.z0.astype(np.complex128),
                                           case.pos, case.a64)
    assert abs(phi - phi_o) <= 1e-5 * phi_o
    assert rel_err(gz, gz_o) <= 1e-5
    assert rel_err(gq, gq_o) <= 1e-5


def test_chunked_gradient_sums_are_bitwise_repeatable(lib, torch):
    """Several chunks: the sums of one chunk run beside the next chunk's patches on
    two buffer pairs.  Calls in a row, and a call after a misfit-only one, give
    bitwise the same gradients."""
    m = 64
    case = Case(n=2 * m + 40, m=m, side=5, noise_peak=1e4, seed=140)
    ctx = make_context(lib, case, oracle_params(minibatch=6))
    lib.emg_set_gradient_chunk(ctx.ctx, 5)               # 29 positions: 6 chunks
    first = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
    second = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
    zd = torch.from_numpy(c64(case.z0)).cuda()
    qd = torch.from_numpy(c64(case.q0)).cuda()
    lib.emg_misfit_gradient(ctx.ctx, zd.data_ptr(), qd.data_ptr(), 0, 0, True)
    third = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
    ctx.close()
    for other in (second, third):
        assert other[0] == first[0]
        assert np.array_equal(other[1], first[1]) and np.array_equal(other[2], first[2])
    phi_o, gz_o, gq_o = O.misfit_gradients(case.q0.astype(np.complex128), case.z0.astype(np.complex128),
                                           case.pos, case.a64)
    assert rel_err(first[1], gz_o) <= 1e-5 and rel_err(first[2], gq_o) <= 1e-5


def test_gradient_matches_central_differences(lib, torch):
    """Central differences (h = 1e-3) of the FP64 misfit at the same point."""
    case = Case(n=104, m=32, side=4, noise_peak=1e4, seed=9)
    ctx = make_context(lib, case, oracle_params(minibatch=8))
    _, gz, gq = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
    ctx.close()
    z = case.z0.astype(np.complex128)
    q = case.q0.astype(np.complex128)
    h = 1e-3
    rng = np.random.default_rng(2)
    for _ in range(4):
        i, j = rng.integers(20, 80, 2)
        for unit in (1.0, 1j):
            zp, zm = z.copy(), z.copy()
            zp[i, j] += h * unit
            zm[i, j] -= h * unit
            fd = (O.misfit(q, zp, case.pos, case.a64) - O.misfit(q, zm, case.pos, case.a64)) / (2 * h)
            got = gz[i, j].real if unit == 1.0 else gz[i, j].imag
            assert abs(got - fd) <= 1e-4 * np.max(np.abs(gz))
        i, j = rng.integers(0, 32, 2)
        for unit in (1.0, 1j):
            qp, qm = q.copy(), q.copy()
            qp[i, j] += h * unit
            qm[i, j] -= h * unit
            fd = (O.misfit(qp, z, case.pos, case.a64) - O.misfit(qm, z, case.pos, case.a64)) / (2 * h)
            got = gq[i, j].real if unit == 1.0 else gq[i, j].imag
            assert abs(got - fd) <= 1e-4 * np.max(np.abs(gq))


def test_autograd_function_uses_the_kernel_gradient(lib, torch):
    from paper_2511_01793_gb300 import autograd as AG

    case = Case(n=104, m=32, side=4, seed=10)
    ctx = make_context(lib, case, oracle_params(minibatch=8))
    _, gz, gq = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
    o = torch.from_numpy(case.z0).cuda().requires_grad_(True)
    q = torch.from_numpy(case.q0).cuda().requires_grad_(True)
    loss = 3.0 * AG.misfit(o, q, ctx)
    loss.backward()
    assert np.allclose(o.grad.cpu().numpy(), 3.0 * gz, rtol=1e-6, atol=1e-6 * np.abs(gz).max())
    assert np.allclose(q.grad.cpu().numpy(), 3.0 * gq, rtol=1e-6, atol=1e-6 * np.abs(gq).max())
    ctx.close()


def test_gradient_descent_baseline_reduces_the_misfit(lib, torch):
    from paper_2511_01793_gb300 import autograd as AG

    case = Case(n=104, m=32, side=5, step=8, seed=11, edge=False, pert=0.2)
    ctx = make_context(lib, case, oracle_params(minibatch=8))
    o = torch.from_numpy(case.z0).cuda()
    q = torch.from_numpy(case.q0).cuda()
    _, _, hist = AG.gradient_descent(ctx, o, q, 40)
    ctx.close()
    assert hist[-1] < 0.5 * hist[0]
    assert all(b <= a * (1 + 1e-6) for a, b in zip(hist, hist[1:]))


def test_full_size_gradient_workload(lib, torch):
    """Object 1024^2, probe 256^2, 1600 positions, Poisson 1e4: gradient vs the oracle."""
    import paper_2511_01793_gb300 as emg

    w = synth.make_workload("grad_n1024_m256")
    pr = w.params
    d = O.forward_intensity(w.q_true, w.z_true, w.pos)
    d = synth.poisson_noise(d, pr["peak"], np.random.Generator(np.random.PCG64(pr["noise_seed"]))).astype(np.float32)
    rng = np.random.default_rng(12)
    z = c64(synth.perturb(w.z_true, 0.2, rng))
    q = c64(synth.perturb(w.q_true, 0.2, rng))
    params = emg.emg_default_params(alpha=pr["alpha"], minibatch=pr["minibatch"])
    ctx = emg.Context(w.pos, d, pr["n"], pr["n"], params)
    phi, gz, gq = _gpu_gradient(lib, torch, ctx, z, q)
    ctx.close()
    phi_o, gz_o, gq_o = O.misfit_gradients(q.astype(np.complex128), z.astype(np.complex128), w.pos,
                                           np.sqrt(d.astype(np.float64)))
    assert abs(phi - phi_o) <= 1e-5 * phi_o
    assert rel_err(gz, gz_o) <= 1e-5
    assert rel_err(gq, gq_o) <= 1e-5


@pytest.mark.parametrize("m,n_pos,chunk", [(16, 2500, 0), (32, 1300, 1300), (64, 330, 7), (128, 160, 0), (256, 45, 20)])
def test_gradients_of_many_positions_by_every_split(lib, torch, m, n_pos, chunk):
    """More positions than clusters (each cluster then sums several probe gradients), several chunks,
    position lists longer than one pass of the sums, and either gradient alone: the gradients equal a
    plain FP64 evaluation to 1e-5, and the parts asked for alone equal the joint call bitwise."""
    rng = np.random.default_rng(m)
    n_rows, n_cols = m + 37, m + 50
    pos = np.stack([rng.integers(-m // 3, 50, n_pos), rng.integers(-m // 3, 60, n_pos)], 1).astype(np.int32)
    z = (rng.standard_normal((n_rows, n_cols)) + 1j * rng.standard_normal((n_rows, n_cols))).astype(np.complex64)
    q = (rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m))).astype(np.complex64)
    d = (rng.uniform(0.5, 2.0, size=(n_pos, m, m)) * 2 * m * m).astype(np.float32)
    c = lib.Context(pos, d, n_rows, n_cols, lib.emg_default_params(minibatch=4), obj=torch.from_numpy(z),
                    probe=torch.from_numpy(q))
    lib.emg_set_gradient_chunk(c.ctx, chunk)

    def call(obj, probe):
        g = torch.zeros_like(c.obj), torch.zeros_like(c.probe)
        phi = lib.emg_misfit_gradient(c.ctx, c.obj.data_ptr(), c.probe.data_ptr(), g[0].data_ptr() if obj else 0,
                                      g[1].data_ptr() if probe else 0)
        return phi, g[0].cpu().numpy(), g[1].cpu().numpy()

    phi, gz, gq = call(True, True)
    assert np.array_equal(call(True, False)[1], gz) and np.array_equal(call(False, True)[2], gq)
    z64, q64, a64 = z.astype(np.complex128), q.astype(np.complex128), np.sqrt(d.astype(np.float64))
    rz, rq, want = np.zeros_like(z64), np.zeros_like(q64), 0.0
    for k in range(n_pos):
        r0, c0 = pos[k]
        rows, cols = slice(max(r0, 0), min(r0 + m, n_rows)), slice(max(c0, 0), min(c0 + m, n_cols))
        zk = np.zeros((m, m), dtype=np.complex128)
        part = slice(rows.start - r0, rows.stop - r0), slice(cols.start - c0, cols.stop - c0)
        zk[part] = z64[rows, cols]
        f = np.fft.fft2(q64 * zk)
        want += 0.5 * np.sum((np.abs(f) - a64[k]) ** 2) / m ** 2
        e = q64 * zk - np.fft.ifft2(a64[k] * f / np.abs(f))
        rz[rows, cols] += (np.conj(q64) * e)[part]
        rq += np.conj(zk) * e
    assert abs(phi - want) <= 1e-5 * want
    assert np.linalg.norm(gz - rz) <= 1e-5 * np.linalg.norm(rz) and np.linalg.norm(gq - rq) <= 1e-5 * np.linalg.norm(rq)
    c.close()


@pytest.mark.parametrize("m", [32, 256])
@pytest.mark.parametrize("after", [0, 1])
def test_gradient_without_room_for_its_chunk_takes_the_minibatch(lib, torch, m, after):
    """Host-side fault injection: one of the automatic chunk's two buffers does not fit.  The call runs in
    chunks that the minibatch buffers hold, with bitwise their sums, and keeps no part of the failed
    allocation; a chunk that was asked for is still refused."""
    case = Case(n=2 * m + 40, m=m, side=4, seed=150 + m)
    p = oracle_params(minibatch=5)

    def call(chunk, fail):
        ctx = make_context(lib, case, p)
        lib.emg_set_gradient_chunk(ctx.ctx, chunk)
        free = torch.cuda.mem_get_info()[0]
        try:
            lib.emg_debug_fail_alloc(after if fail else -1)
            out = _gpu_gradient(lib, torch, ctx, case.z0, case.q0)
        finally:
            lib.emg_debug_fail_alloc(-1)
            lost = free - torch.cuda.mem_get_info()[0]
            ctx.close()
        return out, lost

    call(0, False)                                          # lazy CUDA state in place
    (phi, gz, gq), lost = call(0, True)
    want = call(5, False)[0]
    assert phi == want[0] and np.array_equal(gz, want[1]) and np.array_equal(gq, want[2])
    assert lost <= 4 << 20
    with pytest.raises(lib.EmgError) as e:
        call(case.n_pos, True)
    assert e.value.status == lib.EMG_ENOMEM


@pytest.mark.parametrize("n,n_pos,chunk", [(165, 160, 100), (640, 100, 0), (640, 100, 70)])
def test_gradients_of_few_positions_and_small_objects(lib, torch, n, n_pos, chunk):
    """m = 128: chunks of up to half a wave take clusters of 2, larger ones one CTA per position (100 and a
    remainder of 60 in one call); small objects are summed over smaller tiles.  Repeats bitwise and equals
    the sum of one-position calls to FP32 rounding."""
    m = 128
    rng = np.random.default_rng(n + chunk)
    pos = rng.integers(-m // 3, n - m // 2, size=(n_pos, 2)).astype(np.int32)
    z, q = (c64(rng.standard_normal(s) + 1j * rng.standard_normal(s)) for s in ((n, n + 3), (m, m)))
    d = (rng.uniform(0.5, 2.0, size=(n_pos, m, m)) * 2 * m * m).astype(np.float32)

    def call(sub, chunk):
        c = lib.Context(pos[sub], d[sub], n, n + 3, lib.emg_default_params(), obj=torch.from_numpy(z),
                        probe=torch.from_numpy(q))
        lib.emg_set_gradient_chunk(c.ctx, chunk)
        out = _gpu_gradient(lib, torch, c, z, q)
        again = _gpu_gradient(lib, torch, c, z, q)
        c.close()
        assert all(np.array_equal(a, b) for a, b in zip(out, again))
        return out

    phi, gz, gq = call(slice(None), chunk)
    parts = [call(slice(k, k + 1), 0) for k in range(n_pos)]
    want = sum(p[0] for p in parts), sum(p[1] for p in parts), sum(p[2] for p in parts)
    # FP32 sums of at most 160 terms against FP64 sums of the same terms
    assert abs(phi - want[0]) <= 1e-6 * want[0]
    assert rel_err(gz, want[1]) <= 2e-6 and rel_err(gq, want[2]) <= 2e-6
