"""GPU tests of the top-k similarity table (through the C ABI) against the
oracle.  The table is integer output decided by floating point: the oracle
reproduces the library's normalised bf16 embedding exactly and decides on
exact similarities of it, while the tensor cores sum the d exact products in
fp32, within eps = 2 d 2^-24 of the exact value (unit vectors).  So a row is
checked for what is unique -- every token whose exact similarity exceeds the
exact k-th largest by more than 2 eps is present, the first entry is the
token itself -- and for validity: k distinct tokens, in descending exact
similarity up to 2 eps, none outside missing by more than 2 eps.  Small
exact cases (a hand-worked table with ties) must match exactly."""
import json
import os

import numpy as np
import pytest
import torch

import oracle
from paper_2606_19528_gb300 import lora, synth
from tests import gpu_util as G

pytestmark = pytest.mark.gpu

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden")


def run_table(bits, k, status=lora.LORA_OK):
    V, d = bits.shape
    E = G.dev_bf16(bits)
    table = torch.full((V, k), -1, dtype=torch.int32, device="cuda")
    ws = G.workspace(lora.lora_topk_workspace_size(V, d, k))
    lora.lora_topk_table(E, V, d, k, table, ws, ws.numel())
    torch.cuda.synchronize()
    assert lora.lora_read_status() == status
    return table.cpu().numpy()


def test_topk_handworked_exact():
    with open(os.path.join(GOLDEN, "topk_table_handworked_V4_d2.json")) as f:
        g = json.load(f)
    for E, want in ((g["E"], g["table_k4"]), (g["ties"]["E"], g["ties"]["table_k4"])):
        x = np.zeros((4, 8))
        x[:, :2] = np.array(E, dtype=np.float64)  # d padded to 8 with zeros: norms and products unchanged
        got = run_table(synth.to_bf16_bits(x), 4)
        assert got.tolist() == want, (got.tolist(), want)


def check_rows(bits, table, k, rows):
    V, d = bits.shape
    eps = 2.0 * d * 2.0 ** -24
    En = oracle.normalize_rows(bits)
    C = oracle.similarities(En, rows)
    for r, i in enumerate(rows):
        L = table[i]
        assert len(set(L.tolist())) == k and L.min() >= 0 and L.max() < V, i
        assert L[0] == i, (i, L[:4])
        c = C[r]
        cl = c[L]
        assert np.all(cl[:-1] >= cl[1:] - 2 * eps), i
        kth = np.sort(c)[::-1][k - 1]
        outside = np.ones(V, dtype=bool)
        outside[L] = False
        assert np.all(c[outside] <= cl[-1] + 2 * eps), i
        must = np.nonzero(c > kth + 2 * eps)[0]
        assert np.all(np.isin(must, L)), i


# V >= 32768 takes the sampled-threshold selection, smaller V the radix path
@pytest.mark.parametrize("V,d,k", [(5000, 256, 37), (1200, 64, 1024), (20000, 1024, 500), (32767, 64, 64),
                                   (32768, 64, 64), (40000, 64, 300), (70000, 128, 1024)],
                         ids=["V5000_d256_k37", "V1200_d64_k1024", "V20000_d1024_k500", "V32767_d64_k64",
                              "V32768_d64_k64_sampled", "V40000_d64_k300_sampled", "V70000_d128_k1024_sampled"])
def test_topk_table_parity(V, d, k):
    bits = synth.gen_E(0, 50, V, d)
    table = run_table(bits, k)
    rng = np.random.default_rng(V)
    rows = np.unique(np.concatenate([[0, V - 1, 511, 512], rng.integers(0, V, 60)]))
    check_rows(bits, table, k, rows)


# partial row groups and column chunks of the norms, several chunks of short rows, large k (a short sample)
@pytest.mark.parametrize("V,d,k", [(2001, 72, 16), (9003, 200, 130), (33001, 72, 1024), (17001, 64, 1000),
                                   (100, 8, 100)],
                         ids=["V2001_d72_k16", "V9003_d200_k130", "V33001_d72_k1024", "V17001_d64_k1000", "V100_d8_k100"])
def test_topk_table_edges(V, d, k):
    """The oracle's checks, and the same table when rows are scaled by powers of two (2^62 and 2^-50 take the two
    division paths of the normalisation; a scaled row normalises to the same bits)."""
    bits = synth.gen_E(0, 52, V, d)
    table = run_table(bits, k)
    rng = np.random.default_rng(V)
    rows = [r for r in (0, V - 1, 511, 512) if r < V]
    check_rows(bits, table, k, np.unique(np.concatenate([rows, rng.integers(0, V, 20)])))
    scale = np.array([1.0, 2.0 ** 62, 2.0 ** -50])[rng.integers(0, 3, V)]
    scaled = synth.to_bf16_bits(synth.bf16_bits_to_f64(bits) * scale[:, None])
    assert np.array_equal(run_table(scaled, k), table)


def test_topk_argument_errors():
    with pytest.raises(lora.LoraError) as e:
        lora.lora_topk_workspace_size(100, 12, 5)  # d not a multiple of 8
    assert e.value.code == lora.LORA_EINVAL
    with pytest.raises(lora.LoraError) as e:
        lora.lora_topk_workspace_size(100, 16, 101)  # k > V
    assert e.value.code == lora.LORA_EINVAL
    with pytest.raises(lora.LoraError) as e:
        lora.lora_topk_workspace_size(5000, 16, 1025)  # k beyond the selection's capacity
    assert e.value.code == lora.LORA_EINVAL


def test_topk_sampled_ties_and_fallback():
    """Rows 0..1999 are one vector u, rows 2000..4999 one vector v with
    cos(u, v) about 0.9, the rest random (V = 40000, k = 1000).  A u row's
    sampled threshold lands on v's similarity, so 5000 values pass it (more
    than the 4096 candidate slots) and the row falls back to the radix select;
    a v row passes 3000 tied values and stays on the sampled path.  Identical
    inputs give identical tensor-core sums, so the ties are exact and the
    lower index goes first: u rows list tokens 0..999, v rows 2000..2999."""
    V, d, k = 40000, 64, 1000
    bits = synth.gen_E(0, 51, V, d)
    x = synth.bf16_bits_to_f64(bits)
    u = x[7] / np.linalg.norm(x[7])
    w = x[11] - (x[11] @ u) * u
    v = 0.9 * u + np.sqrt(1 - 0.81) * w / np.linalg.norm(w)
    ub, vb = synth.to_bf16_bits(u[None, :]), synth.to_bf16_bits(v[None, :])
    bits = bits.copy()
    bits[0:2000] = ub
    bits[2000:5000] = vb
    table = run_table(bits, k)
    for i in (0, 1, 1999):
        assert table[i].tolist() == list(range(1000)), i
    for i in (2000, 4999):
        assert table[i].tolist() == list(range(2000, 3000)), i
    check_rows(bits, table, k, np.array([5000, 12345, V - 1]))


def test_topk_short_rows_ties_and_nan():
    """Short rows whose k-th similarity ties with thousands of others go to the radix select (lower index first), and
    so do rows with a NaN similarity: rows 0..2999 are one vector, and with an infinite element in row 3500 (its
    normalised row holds a NaN) every row of the table still lists k distinct tokens, each row's as without it but
    for that token (its own row, 4000 tied NaNs, lists the first k)."""
    V, d, k = 4000, 64, 100
    bits = synth.gen_E(0, 53, V, d)
    bits[:3000] = bits[7]
    table = run_table(bits, k)
    assert np.array_equal(table[[0, 1500, 2999]], np.tile(np.arange(k), (3, 1)))
    check_rows(bits, table, k, np.array([3000, 3400, V - 1]))
    bad = bits.copy()
    bad[3500, 3] = 0x7F80
    t2 = run_table(bad, k)
    for i in (3000, 3400, V - 1):
        rest = t2[i][t2[i] != 3500]
        assert len(set(t2[i].tolist())) == k and len(rest) >= k - 1
        assert np.array_equal(rest, table[i][table[i] != 3500][:len(rest)])


# just over the short rows, a length that is no multiple of 4, and the longest below the stored candidates
@pytest.mark.parametrize("V,k", [(8193, 1000), (20481, 1000), (32766, 64)])
def test_topk_row_sample_ties_and_nan(V, k):
    """Rows whose threshold comes from a sample of the row itself: rows 0..nu-1 are one vector u, rows nu..3899 one
    vector v with cos(u, v) about 0.9, so that u's k-th value is one of thousands of exact ties (the lower index
    first). A random row whose k-th similarity is v's has at most k - 1 above it and 3900 - nu ties: 999 + 3000 at
    k = 1000, 63 + 3880 at k = 64, so with a NaN at most 4000 of the 4096 candidates that the selection holds. With an
    infinite element in the last row every other row holds a NaN, and goes to the radix select; that row itself (V
    tied NaNs, more than the selection holds) is reported and left unwritten."""
    d = 64
    bits = synth.gen_E(0, 54, V, d)
    x = synth.bf16_bits_to_f64(bits)
    u = x[7] / np.linalg.norm(x[7])
    w = x[11] - (x[11] @ u) * u
    v = 0.9 * u + np.sqrt(1 - 0.81) * w / np.linalg.norm(w)
    bits = bits.copy()
    nu = max(k - 100, 20)
    bits[:nu] = synth.to_bf16_bits(u[None, :])
    bits[nu:3900] = synth.to_bf16_bits(v[None, :])
    table = run_table(bits, k)
    for i in (0, nu - 1):
        assert np.array_equal(table[i], np.arange(k)), i
    for i in (nu, 3899):
        assert np.array_equal(table[i], np.arange(nu, nu + k)), i
    check_rows(bits, table, k, np.array([4000, 7777, V - 1]))
    bad = bits.copy()
    bad[V - 1, 3] = 0x7F80
    t2 = run_table(bad, k, lora.LORA_EINVAL)
    for i in (0, nu, 4000, 7777):
        rest = t2[i][t2[i] != V - 1]
        assert len(set(t2[i].tolist())) == k and len(rest) >= k - 1, i
        assert np.array_equal(rest, table[i][table[i] != V - 1][:len(rest)]), i
