"""Padded leading dimensions: every product path gives the same bits whether the
matrices are packed or lie in larger storage (ld = rows + 3), and leaves the padding
alone. Odd orders, so that vectorised loads meet every alignment a column can have."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
PAD = 3


def padded(t):
    """The same matrix in storage with PAD more rows, filled with NaN."""
    rows, cols = t.shape
    buf = torch.full((cols, rows + PAD), complex(float("nan"), float("nan")), dtype=t.dtype,
                     device=t.device)
    buf[:, :rows] = t.mT
    return buf, buf.mT[:rows, :]


def run(lib, op, kw, N, n, pad):
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    rnd = lambda r, c: torch.randn(c, r, dtype=torch.complex128, device="cuda", generator=g).mT
    Z = rnd(N, N)
    A = lib.colmajor((Z + Z.mH) / (4 * N ** 0.5))
    V, Yb = rnd(N, n), rnd(N, n)
    if op == "rr":
        V = lib.colmajor(torch.linalg.qr(V)[0])
    bufs = []

    def place(t):
        if not pad:
            return lib.colmajor(t.clone())
        b, v = padded(t)
        bufs.append((b, t.shape[0]))
        return v

    A, V, Yb = place(A), place(V), place(Yb)
    out = [V]
    degs = np.full(n, 4, dtype=np.int32)
    with lib.Context(lib.default_params(N, n, 0, **kw)) as ctx:
        if op == "filter":
            ctx.chase_filter(A, V, n, degs, 0.3, 0.9, -1.2,
                             precision=kw.get("precision", lib.CHASE_FP64))
        elif op == "qr":
            ctx.chase_qr(V, n, 1e3)
        elif op == "rr":
            ritz = torch.zeros(n, dtype=torch.float64, device="cuda")
            ctx.chase_rayleigh_ritz(A, V, n, ritz)
            out.append(ritz)
        elif op == "residuals":
            r = torch.zeros(n, dtype=torch.float64, device="cuda")
            ctx.chase_residuals(A, V, torch.zeros_like(r), n, r)
            out.append(r)
        else:
            Ab, Vb = place(torch.zeros_like(A)), place(torch.zeros_like(V))
            ctx.chase_filter_vjp(A, V, n, 6, 0.3, 0.9, -1.2, Yb, Ab, Vb)
            out += [Ab, Vb]
    torch.cuda.synchronize()
    for b, rows in bufs:
        assert bool(torch.isnan(b[:, rows:].real).all())
    return [o.clone() for o in out]


@pytest.mark.parametrize("op,mode", [(o, m) for o in ("filter", "qr", "rr", "residuals", "vjp")
                                     for m in ("core", "tensor")] + [("filter", "mixed")])
@pytest.mark.parametrize("N,n", [(131, 30), (517, 70)])
def test_padding_changes_nothing(lib, op, mode, N, n):
    kw = dict(fp64_tensor=int(mode == "tensor"))
    if mode == "mixed":
        kw["precision"] = lib.CHASE_MIXED_BF16X3
    packed, strided = run(lib, op, kw, N, n, False), run(lib, op, kw, N, n, True)
    for a, b in zip(packed, strided):
        assert torch.equal(torch.view_as_real(a) if a.is_complex() else a,
                           torch.view_as_real(b) if b.is_complex() else b)
