"""Chunks above 1024 symbols, which a warp encodes in pieces: whole pieces and parts of
them, chunks that are and are not complete, codewords above 26 bits and escapes that
send a piece to the general path, bytes, against the oracle's encoding."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

CHUNKS = [1152, 1920, 2048, 32640, 32768]


def check(oracle, sym, D, K):
    from paper_2503_06322_gb300 import hpdr as H
    ln_ref = oracle.code_lengths(oracle.histogram(sym, D))
    words_ref, chunk_ref, bits_ref = oracle.encode(sym, ln_ref, K=K)
    ln, chunk, words, bits = H.hpdr_huffman_encode(torch.from_numpy(sym.view(np.int16)).cuda(), D=D, K=K)
    assert np.array_equal(ln.cpu().numpy(), ln_ref) and bits == bits_ref
    assert np.array_equal(chunk.cpu().numpy().view(np.uint64), chunk_ref)
    assert np.array_equal(words.cpu().numpy().view(np.uint32), words_ref)
    dec = H.hpdr_huffman_decode(words, bits, chunk, sym.size, ln, D=D, K=K)
    assert np.array_equal(dec.cpu().numpy().view(np.uint16), sym)
    return ln_ref


@pytest.mark.parametrize("K", CHUNKS)
@pytest.mark.parametrize("n", [1, 100, 1024, 1025, 3000, 32769, 70001])
def test_pieces(oracle, K, n):
    rng = np.random.default_rng(n)
    for D, scale in ((4, 0.5), (8192, 40.0), (32768, 3000.0)):
        sym = np.clip(np.round(rng.laplace(D // 2, scale, n)), 0, D - 1).astype(np.uint16)
        check(oracle, sym, D, K)


@pytest.mark.parametrize("K", CHUNKS)
def test_long_codewords(oracle, K):
    f = [1, 1]
    while len(f) < 30:
        f.append(f[-1] + f[-2])
    sym = np.repeat(np.arange(30, dtype=np.uint16), f)
    sym = sym[np.random.default_rng(1).permutation(sym.size)]
    assert check(oracle, sym, 256, K).max() > 26


@pytest.mark.parametrize("K", CHUNKS)
@pytest.mark.parametrize("tol", [1e-3, 1e-6, 1e-10])
def test_escapes(oracle, K, tol):
    from paper_2503_06322_gb300 import hpdr as H
    u = np.cumsum(np.random.default_rng(K).standard_normal((70, 1003)), axis=1)
    buf = H.hpdr_compress(torch.from_numpy(u).cuda(), tol, chunk=K)
    h = oracle.parse_header(buf.cpu().numpy())
    sym, esc = oracle.decode(h["words"], h["chunk"], h["N"], h["K"], h["lengths"], esc_width=h["esc_width"])
    ln = oracle.code_lengths(oracle.histogram(sym, 8192))
    words, chunk, bits = oracle.encode(sym, ln, K=K, esc_k=esc)
    assert np.array_equal(h["lengths"], ln)
    assert np.array_equal(h["chunk"], chunk) and h["total_bits"] == bits
    assert np.array_equal(h["words"], words)
    assert np.abs(H.hpdr_decompress(buf).cpu().numpy() - u).max() <= tol * np.abs(u).max()


@pytest.mark.parametrize("K", CHUNKS)
@pytest.mark.parametrize("n", [5000, 100001])
def test_byte_keys(oracle, K, n):
    from paper_2503_06322_gb300 import hpdr as H
    x = np.clip(np.round(np.random.default_rng(n).laplace(128, 6.0, size=n)), 0, 255).astype(np.uint8)
    buf = H.hpdr_lossless_compress(torch.from_numpy(x).cuda(), K=K)
    b = buf.cpu().numpy()
    words, chunk, bits = oracle.encode(x.astype(np.uint16), oracle.code_lengths(oracle.histogram(x.astype(np.uint16), 256)), K=K)
    off_chunk, off_bits = (int(v) for v in b[40:56].view(np.uint64))
    assert np.array_equal(b[off_chunk:off_chunk + 8 * chunk.size].view(np.uint64), chunk)
    assert np.array_equal(b[off_bits:].view(np.uint32), words)
    assert np.array_equal(H.hpdr_lossless_decompress(buf).cpu().numpy(), x)
