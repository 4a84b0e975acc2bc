"""The byte-matrix converters and the operators on bytes and bit rows, at the edges of their runs (whole rows, rows cut
into segments, one-row runs), at every alignment of the caller's buffers, and with outputs that are or overlap inputs.
Plain torch on the same bytes is the reference."""
import pytest
import torch

pkg = pytest.importorskip("paper_2408_10369_gb300")
from paper_2408_10369_gb300 import bmlp  # noqa: E402

pytestmark = pytest.mark.gpu
PACKED = bmlp.BMLP_FMT_PACKED64


@pytest.fixture(scope="module")
def ctx():
    c = pkg.Context(0)
    yield c
    c.close()


def matrix(n, offset, seed, density=0.3):
    """n x n random bytes (0, 1 and other nonzero values) that start `offset` bytes into their allocation."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    buf = torch.zeros(n * n + 16, dtype=torch.uint8, device="cuda")
    m = buf[offset:offset + n * n].view(n, n)
    m.copy_((torch.rand((n, n), generator=g, device="cuda") < density) * torch.randint(1, 256, (n, n), generator=g, device="cuda"))
    return m


def guarded(n, offset):
    """An output matrix with guard bytes on both sides."""
    buf = torch.full((n * n + 32,), 0xA5, dtype=torch.uint8, device="cuda")
    return buf, buf[offset:offset + n * n].view(n, n)


def intact(buf, offset, n):
    return bool((buf[:offset] == 0xA5).all()) and bool((buf[offset + n * n:] == 0xA5).all())


@pytest.mark.parametrize("n", [1, 2, 7, 15, 16, 17, 63, 64, 65, 127, 300, 1000, 3157, 4099])
@pytest.mark.parametrize("offset", [0, 1, 8, 15])
def test_byte_operators(ctx, n, offset):
    a, b = matrix(n, offset, 1), matrix(n, (offset * 3) % 16, 2)
    type_rows, type_cols = torch.rand(n, device="cuda") < 0.7, torch.rand(n, device="cuda") < 0.7
    pack = lambda v: torch.zeros((n + 63) // 64, dtype=torch.int64, device="cuda").index_add_(  # noqa: E731
        0, v.nonzero().view(-1) >> 6, torch.ones_like(v.nonzero().view(-1)) << (v.nonzero().view(-1) & 63))
    buf, out = guarded(n, offset)
    ctx.transpose(a, n, out)
    assert torch.equal(out, (a.T != 0).to(torch.uint8)) and intact(buf, offset, n)
    ctx.union(a, b, n, out)
    assert torch.equal(out, ((a | b) != 0).to(torch.uint8)) and intact(buf, offset, n)
    ctx.negate(a, n, out, rows=pack(type_rows), cols=pack(type_cols))
    assert torch.equal(out, ((a == 0) & type_rows[:, None] & type_cols[None, :]).to(torch.uint8)) and intact(buf, offset, n)
    ctx.negate(a, n, out)
    assert torch.equal(out, (a == 0).to(torch.uint8)) and intact(buf, offset, n)
    # bytes -> bit rows -> bytes through a closure of a symmetric idempotent relation (one class of related constants)
    cls = torch.rand(n, device="cuda") < 0.5
    a.copy_((cls[:, None] & cls[None, :]) * 7)
    ctx.rms(a, n, out, reflexive=True)
    want = (cls[:, None] & cls[None, :]) | torch.eye(n, dtype=torch.bool, device="cuda")
    assert torch.equal(out, want.to(torch.uint8)) and intact(buf, offset, n)


@pytest.mark.parametrize("n", [16384, 16385, 20011])
def test_long_rows(ctx, n):
    """Rows cut into segments of 16,384 columns."""
    a = matrix(n, 5, 3, 0.01)
    buf, out = guarded(n, 3)
    ctx.transpose(a, n, out)
    assert torch.equal(out, (a.T != 0).to(torch.uint8)) and intact(buf, 3, n)
    ctx.negate(a, n, out)
    assert torch.equal(out, (a == 0).to(torch.uint8)) and intact(buf, 3, n)


@pytest.mark.parametrize("n", [65, 1000, 4096])
def test_overlapping_outputs(ctx, n):
    """In place, and outputs that overlap an input elsewhere: as if the inputs had been copied first."""
    a, b = matrix(n, 0, 4), matrix(n, 0, 5)
    want = ((a | b) != 0).to(torch.uint8)
    x = a.clone()
    ctx.union(x, b, n, x)
    assert torch.equal(x, want)
    buf = torch.zeros(n * n + n, dtype=torch.uint8, device="cuda")
    shifted, at = buf[n:].view(n, n), buf[:n * n].view(n, n)
    shifted.copy_(a)
    ctx.union(shifted, b, n, at)
    assert torch.equal(at, want)
    x = a.clone()
    ctx.negate(x, n, x)
    assert torch.equal(x, (a == 0).to(torch.uint8))
    x = a.clone()
    ctx.transpose(x, n, x)
    assert torch.equal(x, (a.T != 0).to(torch.uint8))


@pytest.mark.parametrize("n", [1, 63, 64, 130, 300, 2000, 8257])
def test_packed_operators(ctx, n):
    """Bit rows whose padding bits are set on input: ignored, and clear on output."""
    w = (n + 63) // 64
    g = torch.Generator(device="cuda").manual_seed(n)
    bits = lambda: torch.randint(-2**62, 2**62, (n, w), generator=g, device="cuda") | (1 << 62)  # noqa: E731
    a, b = bits(), bits()
    valid = torch.full((w,), -1, dtype=torch.int64, device="cuda")
    if n % 64:
        valid[-1] = (1 << (n % 64)) - 1
    out = torch.empty_like(a)
    ctx.union(a, b, n, out, fmt=PACKED)
    assert torch.equal(out, (a | b) & valid)
    ctx.negate(a, n, out, fmt=PACKED)
    assert torch.equal(out, ~a & valid)
    ctx.transpose(a, n, out, fmt=PACKED)
    unpack = lambda m: ((m[:, :, None] >> torch.arange(64, device="cuda")) & 1).reshape(n, -1)[:, :n]  # noqa: E731
    assert torch.equal(unpack(out), unpack(a).T)
    assert n % 64 == 0 or not bool((out[:, -1] & ~valid[-1]).any())
    x = a.clone()
    ctx.transpose(x, n, x, fmt=PACKED)
    assert torch.equal(x, out)
