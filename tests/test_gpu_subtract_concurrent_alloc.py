"""Masks of a subtract that runs while the host maps and unmaps device memory.

Mapping memory stalls loads in flight.  A warp's last read of a stage has to be
over before the stage is given back for the next tile's bytes, stalled or not.
"""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu

W, H, K = 1920, 1080, 10


def _clip(n, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    m = W * H
    row = torch.arange(m, device="cuda") // W
    base = torch.rand(m, device="cuda", generator=g) * 150 + 40
    D = torch.empty((n, m), dtype=torch.uint8, device="cuda")
    for t in range(n):
        x = base + 3 * torch.randn(m, device="cuda", generator=g) + 40 * ((row + 2 * t) % H < 60)
        D[t] = x.clamp(0, 255).to(torch.uint8)
    return D, base


@pytest.mark.parametrize("n", [200, 100])      # two blocks of frames and a ring of three; one block
@pytest.mark.parametrize("mode", ["modulus", "complex", "background"])
def test_masks_while_memory_is_mapped(n, mode):
    from paper_1512_04205_gb300 import cdmd as C

    D, base = _clip(n, 31)
    m = W * H
    g = torch.Generator(device="cuda").manual_seed(7)
    Phi = torch.randn((m, K, 2), device="cuda", generator=g)
    Phi[:, 0, 0], Phi[:, 0, 1] = base, 0.0
    Phi = torch.view_as_complex(Phi)
    lam = torch.zeros(K, dtype=torch.complex128, device="cuda")
    lam[0] = 1.0
    for c in range(1, K):
        pair = (c + 1) // 2                     # 1 .. 4: conjugate neighbours, then a real one
        im = 0.0 if c == K - 1 else 0.02 * pair if c % 2 else -0.02 * pair
        if mode == "complex":
            im = 0.03 * c                       # no conjugate partners: real and imaginary part
        lam[c] = complex(1.0 - 0.01 * pair, im)
    beta = torch.full((K,), 0.5, dtype=torch.complex128, device="cuda")
    beta[0] = 1.0
    ctx = C.Context(0)
    want_bg = mode == "background"              # the kernel that writes the background too
    words = (m + 31) // 32
    masks = [torch.empty((n, words), dtype=torch.int32, device="cuda") for _ in range(8)]
    bg = torch.empty((n, m), dtype=torch.float32, device="cuda") if want_bg else None

    def subtract(mask):
        C.cdmd_subtract(ctx, D, Phi, beta, lam, 25.0, want_bg=want_bg, mask=mask, bg=bg)

    for x in masks:
        subtract(x)
    torch.cuda.synchronize()
    quiet = masks[0].clone()
    assert 0 < int((quiet != 0).sum()) < quiet.numel()
    for x in masks:
        assert torch.equal(x, quiet)
    wrong = 0
    for it in range(24):
        for x in masks:
            x.zero_()
        torch.cuda.synchronize()
        for x in masks:
            subtract(x)
        t0 = time.perf_counter()
        while time.perf_counter() - t0 < 0.0002 * (it % 4):
            pass
        held = [torch.empty((200 << 20) + (it << 20), dtype=torch.uint8, device="cuda") for _ in range(3)]
        torch.cuda.synchronize()
        wrong += sum(not torch.equal(x, quiet) for x in masks)
        del held
        torch.cuda.empty_cache()
    C.cdmd_status_sync(ctx)
    assert wrong == 0
