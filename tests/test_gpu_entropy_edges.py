"""Entropy stage at the edges of its kernels: containers equal to the oracle's
encoding of their own codes for streams that end around a warp's group of 1024
symbols, escapes whose codeword and payload fit 32 bits or do not, and
codebooks from one present symbol to all of them with frequencies that take
every number of radix passes."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 31, 1023, 1024, 1025, 2047, 3073, 5000])
@pytest.mark.parametrize("tol", [1e-2, 1e-5, 1e-8, 1e-12])
@pytest.mark.parametrize("D", [4, 8192])
def test_escapes_and_partial_groups(oracle, n, tol, D):
    from paper_2503_06322_gb300 import hpdr as H
    u = np.cumsum(np.random.default_rng(n).standard_normal(n))
    buf = H.hpdr_compress(torch.from_numpy(u).cuda(), tol, dict_size=D)
    h = oracle.parse_header(buf.cpu().numpy())
    sym, esc = oracle.decode(h["words"], h["chunk"], h["N"], h["K"], h["lengths"], esc_width=h["esc_width"])
    ln = oracle.code_lengths(oracle.histogram(sym, D))
    words, chunk, bits = oracle.encode(sym, ln, K=h["K"], esc_k=esc)
    assert np.array_equal(h["lengths"], ln)
    assert np.array_equal(h["chunk"], chunk) and h["total_bits"] == bits
    assert np.array_equal(h["words"], words)
    rec = H.hpdr_decompress(buf).cpu().numpy()
    assert np.abs(rec - u).max() <= tol * np.abs(u).max()


@pytest.mark.parametrize("present,top", [(1, 5), (2, 1), (3, 300), (33, 3), (1024, 2), (1025, 70000), (4097, 40),
                                         (8191, 300), (8192, 900)])
def test_codebooks(oracle, present, top):
    from paper_2503_06322_gb300 import hpdr as H
    D, K = 8192, 1024
    rng = np.random.default_rng(present)
    freq = rng.integers(1, 4, size=present)
    freq[rng.integers(present)] = top
    sym = np.repeat(rng.permutation(D)[:present].astype(np.uint16), freq)
    sym = sym[rng.permutation(sym.size)]
    ln_ref = oracle.code_lengths(oracle.histogram(sym, D))
    words_ref, chunk_ref, bits_ref = oracle.encode(sym, ln_ref, K=K)
    ln, chunk, words, bits = H.hpdr_huffman_encode(torch.from_numpy(sym.view(np.int16)).cuda(), D=D, K=K)
    assert np.array_equal(ln.cpu().numpy(), ln_ref) and bits == bits_ref
    assert np.array_equal(words.cpu().numpy().view(np.uint32), words_ref)
    dec = H.hpdr_huffman_decode(words, bits, chunk, sym.size, ln, D=D, K=K)
    assert np.array_equal(dec.cpu().numpy().view(np.uint16), sym)


@pytest.mark.parametrize("n", [1, 7, 16, 33, 1023, 1024, 1025, 4099, 200003])
@pytest.mark.parametrize("shift", [0, 1, 8])
def test_byte_keys_in_place(oracle, n, shift):
    """Byte keys counted, encoded and decoded as bytes, or through 16-bit
    symbols where the pointer does not allow it (shift bytes into a buffer)."""
    from paper_2503_06322_gb300 import hpdr as H
    x = np.clip(np.round(np.random.default_rng(n).laplace(128, 6.0, size=n)), 0, 255).astype(np.uint8)
    store = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
    keys = store[shift:shift + n]
    keys.copy_(torch.from_numpy(x))
    out = torch.zeros(H.lossless_bound(n, 1, 128), dtype=torch.uint8, device="cuda")
    buf = H.hpdr_lossless_compress(keys, K=128, out=out)
    b = buf.cpu().numpy()
    ln = oracle.code_lengths(oracle.histogram(x.astype(np.uint16), 256))
    words, chunk, bits = oracle.encode(x.astype(np.uint16), ln, K=128)
    off_chunk, off_bits = (int(v) for v in b[40:56].view(np.uint64))
    assert b[:4].tobytes() == b"HPDL" and int(b[60:64].view(np.uint32)[0]) == oracle.crc32(b[:60].tobytes())
    assert np.array_equal(b[64:320], ln) and int(b[32:40].view(np.uint64)[0]) == bits
    assert np.array_equal(b[off_chunk:off_chunk + 8 * chunk.size].view(np.uint64), chunk)
    assert not b[320:off_chunk].any() and not b[off_chunk + 8 * chunk.size:off_bits].any()
    assert np.array_equal(b[off_bits:].view(np.uint32), words)
    back = torch.full((n + 16,), 7, dtype=torch.uint8, device="cuda")
    H.hpdr_lossless_decompress(buf, out=back[shift:shift + n])
    got = back.cpu().numpy()
    assert np.array_equal(got[shift:shift + n], x)
    assert (got[:shift] == 7).all() and (got[shift + n:] == 7).all()
