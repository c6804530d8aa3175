"""Index arithmetic and dispatch rules of the kernels, evaluated on the host."""
from host_rules import evaluate


def test_production_histogram_entries_beyond_32_bits(tmp_path):
    """accepted calls have windows of more than 2^31 entries (bin, class)"""
    cases = [(80000, 36001, 36000),   # q = 10, L = 200, one window
             (26886, 80340, 80339),   # q = 255, L = 284, 6 windows that do not overlap
             (1, 7, 3)]
    assert evaluate(tmp_path, ["heo_index(%d, %d, %d)" % c for c in cases]) == [b * n + c for b, n, c in cases]


def test_leading_words_are_shifted_by_less_than_their_width(tmp_path):
    ks = range(-200, 300)
    taken = [k for k, ok in zip(ks, evaluate(tmp_path, ["leading_words(%d)" % k for k in ks])) if ok]
    assert taken and all(0 < 58 - k < 32 for k in taken)


def test_faulting_in_a_result_buffer_keeps_what_it_holds(tmp_path):
    """a read that fails later leaves the caller's buffer as it was; every page is
    looked at once, whatever the alignment"""
    assert evaluate(tmp_path, [r"""([] {
        std::vector<unsigned char> v(1000003);
        for (size_t i = 0; i < v.size(); ++i) v[i] = (unsigned char)(i * 7 + 1);
        rewl::host::fault_in(v.data() + 1, v.size() - 1);
        rewl::host::fault_in(v.data(), 0);
        rewl::host::fault_in(v.data() + 5, 1);
        for (size_t i = 0; i < v.size(); ++i)
            if (v[i] != (unsigned char)(i * 7 + 1)) return 0;
        return 1;
    })()"""]) == [1]
