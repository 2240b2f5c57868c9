"""Stream order and capture.  Single calls and the first launch of a batch are launched with
programmatic stream serialization and wait in the kernel for what came before them: that must
cover events of other streams, copies and other libraries' kernels.  Under stream capture the
same calls are recorded (the first of each as an ordinary launch), and a replay gives what the
calls give."""
import pytest

import workloads as WL

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def roi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    from paper_2608_23048_gb300 import _build
    _build.build()
    import paper_2608_23048_gb300 as roi
    return roi


def _same(a, b):
    import torch
    return all(torch.equal(x.view(torch.int16) if x.dtype == torch.bfloat16 else x.view(torch.int32),
                           y.view(torch.int16) if y.dtype == torch.bfloat16 else y.view(torch.int32))
               for x, y in zip(a, b))


class Calls:
    """Every kind of call on one set of tensors, writing fresh outputs."""

    def __init__(self, roi, N, M, rows, cols, tau):
        import torch
        self.roi, self.N, self.M, self.tau = roi, N, M, tau
        self.W, self.phi, self.dWm = WL.make_inputs(rows, cols, "normal", 5 + M, device=torch.device("cuda"))
        self.st = roi.NoiseState(3, 1, 2, 1.0, 0)
        self.X = WL.make_tokens(9, cols, 5, device=torch.device("cuda"))
        need = roi.roi_masked_linear_workspace_size(9, rows, cols)
        self.ws = torch.empty(max(16, need), dtype=torch.uint8, device="cuda")

    def outputs(self):
        import torch
        bits = lambda: torch.zeros(self.roi.hard_words(*self.phi.shape), dtype=torch.int32, device="cuda")  # noqa: E731
        z, w = (lambda: torch.zeros_like(self.phi)), (lambda: torch.zeros_like(self.W))
        return [w(), bits(), z(), w(), z(), z(), z(), bits(), w(), torch.zeros(9, len(self.phi), device="cuda"), w(), bits(), z()]

    def run(self, out, phi, stream=None):
        roi, N, M, tau, W, dWm, st = self.roi, self.N, self.M, self.tau, self.W, self.dWm, self.st
        Wm, hard, dphi, dW, p, m, v, exp, Wp, Y, bWm, bhard, bdphi = out
        roi.roi_mask_fwd_ex(phi, W, N, M, tau, st, Wm, None, hard, stream=stream)
        roi.roi_mask_bwd(phi, W, st, N, M, dWm, tau, dphi, dW, stream=stream)
        p.copy_(phi)
        roi.roi_mask_bwd_adamw(p, W, st, N, M, dWm, tau, m, v, roi.AdamW(1e-3, 0.9, 0.95, 1e-8, 0.05, 3), stream=stream)
        roi.roi_hard_mask_export(p, N, M, exp, W, Wp, stream=stream)
        if (N, M) in ((2, 4), (4, 8), (2, 8)):
            roi.roi_masked_linear_fwd(self.X, p, W, N, M, tau, st, Y, self.ws, stream=stream)
        half = phi.shape[0] // 2 // 8 * 8
        E = half * phi.shape[1] // 32
        roi.roi_mask_fwd_batch([(phi[:half], W[:half], st, bWm[:half], None, bhard[:E]),
                                (phi[half:], W[half:], st, bWm[half:], None, bhard[E:])], N, M, tau, stream=stream)
        roi.roi_mask_bwd_batch([(phi[:half], W[:half], st, dWm[:half], bdphi[:half], None),
                                (phi[half:], W[half:], st, dWm[half:], bdphi[half:], None)], N, M, tau, stream=stream)
        return out


CASES = [(2, 4, 0.3, 512, 4096), (2, 4, 1.0, 64, 1024), (4, 8, 0.5, 512, 4096), (8, 16, 0.2, 512, 4096),
         (16, 32, 0.2, 64, 1024), (1, 4, 0.5, 128, 1024), (3, 7, 0.5, 160, 7 * 128), (20, 24, 0.05, 16, 24 * 32)]


@pytest.mark.parametrize("N,M,tau,rows,cols", CASES)
def test_calls_wait_for_other_streams_and_copies(roi, N, M, tau, rows, cols):
    import torch
    c = Calls(roi, N, M, rows, cols, tau)
    want = c.run(c.outputs(), c.phi)
    torch.cuda.synchronize()
    side, main = torch.cuda.Stream(), torch.cuda.Stream()
    host = c.phi.cpu().pin_memory()
    other = c.outputs()
    for rep in range(12):
        phi = torch.full_like(c.phi, float(rep))
        out = c.outputs()
        torch.cuda.synchronize()
        with torch.cuda.stream(main):
            # a launch that lets its successor in before it ends
            roi.roi_mask_fwd_ex(c.phi, c.W, N, M, tau, c.st, other[0], None, other[1], stream=main)
            if rep % 3 == 0:
                with torch.cuda.stream(side):
                    torch.cuda._sleep(400_000)
                    phi.copy_(c.phi)
                main.wait_stream(side)
            elif rep % 3 == 1:
                phi.copy_(host, non_blocking=True)
            else:
                torch.cuda._sleep(200_000)
                phi.copy_(c.phi)
            c.run(out, phi, main)
            # read by the next kernel of the stream, with no wait of the host's
            copies = [x.clone() for x in out]
        main.synchronize()
        assert _same(want, copies) and _same(want, out), rep
    roi.roi_device_status()


@pytest.mark.parametrize("N,M,tau,rows,cols", CASES)
def test_captured_calls_replay(roi, N, M, tau, rows, cols):
    import torch
    c = Calls(roi, N, M, rows, cols, tau)
    want = c.run(c.outputs(), c.phi)
    torch.cuda.synchronize()
    phi, out = c.phi.clone(), c.outputs()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        c.run(out, phi, torch.cuda.current_stream())
    for rep in range(3):
        for x in out:
            x.zero_()
        phi.copy_(c.phi)
        graph.replay()
        torch.cuda.synchronize()
        assert _same(want, out), rep
    roi.roi_device_status()
