"""The stream of rotations from the QL recurrence to the warps that apply them: eigenproblems whose
rotations fill the ring several times over, again and again, with other work on the SMs. A count
that some lanes of the copying warp saw and others did not would leave a sweep uncopied."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


# one CTA; clusters of eight; of sixteen at the largest order (360000 rotations, 176 rings)
@pytest.mark.parametrize("m", [48, 140, 600])
def test_repeated_and_concurrent(cuda, m):
    from paper_1007_4400_gb300 import gevp
    rng = np.random.default_rng(9700 + m)
    V = np.linalg.qr(rng.standard_normal((m, m)) + 1j * rng.standard_normal((m, m)))[0]
    lam = np.linspace(-2, 5, m)
    G = torch.from_numpy((V * lam) @ V.conj().T).to(cuda)
    G = 0.5 * (G + G.conj().T)
    lam = torch.from_numpy(lam).to(cuda)
    side = torch.cuda.Stream()
    busy = torch.randn(2048, 2048, device=cuda)
    for _ in range(8):
        with torch.cuda.stream(side):     # other work comes and goes on the SMs meanwhile
            for _ in range(20):
                busy = torch.tanh(busy @ busy)
        th, Z = gevp.heev_small(G)
        assert (th - lam).abs().max().item() <= 1e-12 * 5
        assert (G @ Z - Z * th).abs().max().item() <= 1e-12 * 5
        assert (Z.conj().T @ Z - torch.eye(m, dtype=Z.dtype, device=cuda)).abs().max().item() <= 1e-12
    torch.cuda.synchronize()
