"""The workspace limit holds for the FP64 form, whose digits take 20 MB per p + H position: a chunk's elements run in several
launches then, with the same bits."""
import numpy as np
import pytest

import wpccc_inputs as wi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("solve,mode", [("STAGE", 0), ("SCHUR", 0), ("SCHUR", 2)])
def test_propagate_stays_within_the_limit(solve, mode):
    import paper_2403_04252_gb300 as w
    basis, _ = wi.config_inputs("p_H_2c_n4l3")
    b, zg = np.linspace(0.4, 10.0, 12), np.array([-0.3, -0.2, -0.1, 0.0])
    out, held = [], []
    # one step of 12 paths: S and H twice for 36 positions, their FP32 factors in mode 2, and the carried matrices take
    # 0.39 (0.49) GB, the digits of 36 positions 0.8 GB more
    for limit in (8 << 30, 600 << 20):
        g = w.Basis(basis)
        g.set_solve_mode(getattr(w, "SOLVE_" + solve))
        g.set_workspace_limit(limit)
        c = torch.zeros((b.size, g.N), dtype=torch.complex128, device="cuda")
        c[:, 0] = 1.0
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        out.append(g.propagate(b, 1.5, zg, c=c, precision_mode=mode))
        torch.cuda.synchronize()
        held.append(free - torch.cuda.mem_get_info()[0])
        g.close()
    assert torch.equal(out[0], out[1])
    # the workspace beside what a first call loads (kernels, streams, work lists)
    assert held[1] <= (600 << 20) + (64 << 20), held


def test_short_memory_shrinks_the_digits_scratch_then_takes_the_cuda_cores():
    import paper_2403_04252_gb300 as w
    basis, _ = wi.config_inputs("p_H_2c_n4l3")
    b, zg, zs = np.linspace(0.4, 10.0, 12), np.array([-0.1, 0.0]), np.linspace(-3.0, 3.0, 64)

    def amplitudes(n):
        c = torch.zeros((n, basis.N), dtype=torch.complex128, device="cuda")
        c[:, 0] = 1.0
        return c

    SH = [torch.zeros((64, basis.N, basis.N), dtype=torch.complex128, device="cuda") for _ in range(2)]
    SH0 = [torch.zeros_like(x) for x in SH]
    amps = [amplitudes(12), amplitudes(4), amplitudes(4)]
    start = [a.clone() for a in amps]

    def elements(g):
        g.matrix_elements(1.0, 1.5, zs, SH[0], SH[1])
        return SH

    def propagate(g):
        return [g.propagate(b, 1.5, zg, c=amps[0].copy_(start[0]))]

    def batch(g):
        for a, s in zip(amps[1:], start[1:]):
            a.copy_(s)
        x = w.Batch([(g, b[:4], 1.5, zg), (g, b[4:8], 1.5, zg)], amps[1:], precision_mode=0)
        x.launch()
        x.status()
        x.close()
        return amps[1:]

    def run(call):
        g = w.Basis(basis)                       # its own workspace each time
        out = call(g)
        torch.cuda.synchronize()
        g.close()
        return [x.clone() for x in out] if call is not elements else out

    def with_free(nbytes, call):
        torch.cuda.empty_cache()
        g = w.Basis(basis)
        hold = torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")
        try:
            out = call(g)
            torch.cuda.synchronize()
        finally:
            del hold
            g.close()
            torch.cuda.empty_cache()
        return out

    # 64 positions' digits 1.3 GB; 36 positions' digits 0.7 GB beside 0.4 GB of matrices; two sets of 12 positions with
    # 0.24 GB of digits and 0.13 GB of matrices each: the same bits from a smaller scratch
    for call, nbytes in ((propagate, 600 << 20), (batch, 400 << 20)):
        ample = run(call)
        short = [x.clone() for x in with_free(nbytes, call)]
        assert all(torch.equal(x, y) for x, y in zip(ample, short)), call.__name__
    run(elements)
    for x, y in zip(SH0, SH):
        x.copy_(y)
    with_free(400 << 20, elements)
    assert all(torch.equal(x, y) for x, y in zip(SH, SH0))
    # 14 MB hold two positions of the CUDA cores' form, but not one position's digits: that form's bits, which the
    # no-allocation call has
    few, few0 = [x[:2] for x in SH], [x[:2] for x in SH0]
    with_free(14 << 20, lambda g: g.matrix_elements(1.0, 1.5, zs[:2], few[0], few[1]))
    digits = [x.clone() for x in few0]
    g = w.Basis(basis)
    g.matrix_elements_noalloc(1.0, 1.5, zs[:2], few0[0], few0[1])
    torch.cuda.synchronize()
    g.close()
    assert all(torch.equal(x, y) for x, y in zip(few, few0))
    assert not all(torch.equal(x, y) for x, y in zip(few, digits))


def test_overlap_norms_on_a_nearly_full_device():
    import paper_2403_04252_gb300 as w
    basis, _ = wi.config_inputs("p_H_2c_n4l3")
    n = 64
    rng = np.random.default_rng(3)
    c = torch.from_numpy(rng.standard_normal((n, basis.N)) + 1j * rng.standard_normal((n, basis.N))).cuda()
    b, v, z = np.linspace(0.4, 10.0, n), np.full(n, 1.5), np.linspace(-3.0, 3.0, n)
    out = []
    # S and H take 0.3 GB for 64 paths, the digits 1.3 GB
    for nbytes in (8 << 30, 500 << 20):
        g = w.Basis(basis)
        torch.cuda.empty_cache()
        hold = torch.empty(torch.cuda.mem_get_info()[0] - nbytes, dtype=torch.uint8, device="cuda")
        try:
            out.append(g.overlap_norms(b, v, z, c).clone())
            torch.cuda.synchronize()
        finally:
            del hold
            g.close()
            torch.cuda.empty_cache()
    assert torch.equal(out[0], out[1])
