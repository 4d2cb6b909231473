"""The FP64 form's tensor-core contraction takes more scratch per position than the CUDA cores' form: where the device's
memory holds only the latter, the calls take that one instead of failing."""
import numpy as np
import pytest

import wpccc_inputs as wi

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_fp64_calls_fall_back_to_the_cuda_cores_when_memory_is_short():
    import paper_2403_04252_gb300 as w
    basis, _ = wi.config_inputs("p_H_2c_n4l3")
    b, zg = np.linspace(0.4, 10.0, 40), np.array([-0.1, 0.0])      # 120 positions in one chunk

    def run():
        g = w.Basis(basis)                                         # its own workspace each time
        c = g.propagate(b, 1.5, zg)
        torch.cuda.synchronize()
        g.close()
        return c

    ample = run()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    # 120 positions: S and H 1.1 GB, tables 0.5 GB on the CUDA cores, 2.6 GB with the digits
    hold = torch.empty(free - int(2.8e9), dtype=torch.uint8, device="cuda")
    try:
        short = run()
    finally:
        del hold
        torch.cuda.empty_cache()
    # the same sums in another order: one step's four stages with a solve of condition below 300 each
    assert (short - ample).abs().max().item() < 4 * 380 * 2.0 ** -53 * 300
