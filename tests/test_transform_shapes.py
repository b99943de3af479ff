"""Block shapes of the transforms' matrix products (csrc/dft.cu), restated for
every tube length that can reach them: a thread stages at most the 16 samples of
a K tile that the widest instantiation has registers for, and tables and threads
stay within a block's limits."""
import os
import re

SRC = os.path.join(os.path.dirname(__file__), "..", "paper_1704_04362_gb300", "csrc", "dft.cu")


def constant(text, name):
    return eval(re.search(r"constexpr int [^;]*\b%s = ([0-9 *]+)[,;]" % name, text).group(1))


def test_every_length_fits():
    text = open(SRC).read()
    dk, dn, dm = (constant(text, n) for n in ("DK", "DN", "DM"))
    table, threads = constant(text, "TABLE_BYTES_MAX"), constant(text, "DT_MAX")
    floor = re.search(r"p\.ty = std::max\((\d+), ", text)
    least = int(floor.group(1)) if floor else 1
    widest = max(int(n) for n in re.findall(r"launch_product_np<INV, (\d+)>", text))
    for n3 in range(1, 513):
        h = n3 // 2 + 1
        kp = -(-h // dk) * dk
        fit = max(1, table // (8 * kp * dn))
        groups = -(-h // dn)
        ty = max(least, -(-groups // -(-groups // fit)))
        for tx_log in (4, 5, 6):
            if tx_log > 4 and ty << tx_log > 256:
                continue
            nt, bm = ty << tx_log, dm << tx_log
            assert -(-dk * bm // nt) <= widest, n3
            assert nt <= threads, n3
            assert 8 * kp * ty * dn + 16 * dk * bm + 20 * bm + 8 * n3 <= 227 * 1024, n3
