// The forms of the tensor path's kernel for one 16-bit type (included by conv_tc_bf16.cu and conv_tc_f16.cu, which are
// translation units of their own so that they compile side by side).
#ifndef RTOSS_CONV_TC_FORMS_CUH
#define RTOSS_CONV_TC_FORMS_CUH

#include <utility>

#include "conv_tc_kernel.cuh"

namespace {

constexpr int kNone = RTOSS_ACT_NONE, kRelu = RTOSS_ACT_RELU, kSilu = RTOSS_ACT_SILU, kSiluX = kActSiluX;
constexpr int kKind1 = 1, kKindPxm = 2, kKind3 = 3;

// One convolution.  Without a residual: every activation, cut along K or not.  With one: the combinations the networks use
// (none and ReLU behind the sum, SiLU in front of it).  Behind a layout pass: SiLU in the exponential form, and NCHW.
template <int K, int A> using Plain = std::integer_sequence<int, form_of(K, A, false, 0, false), form_of(K, A, true, 0, false)>;
template <int K, int A> using Nchw = std::integer_sequence<int, form_of(K, A, false, 0, true), form_of(K, A, true, 0, true)>;
template <int K, int A, int R> using Resid = std::integer_sequence<int, form_of(K, A, false, R, false), form_of(K, A, true, R, false)>;
template <int K, bool S> using Elem = std::integer_sequence<int, form_of(K, kNone, S, 0, false) | kFormElem, form_of(K, kRelu, S, 0, false) | kFormElem,
                                                            form_of(K, kSilu, S, 0, false) | kFormElem, form_of(K, kSiluX, S, 0, false) | kFormElem>;
using Pxm = std::integer_sequence<int, form_of(kKindPxm, kNone, false, 0, false), form_of(kKindPxm, kRelu, false, 0, false),
                                  form_of(kKindPxm, kSilu, false, 0, false), form_of(kKindPxm, kSiluX, false, 0, false),
                                  form_of(kKindPxm, kNone, false, 0, true), form_of(kKindPxm, kRelu, false, 0, true),
                                  form_of(kKindPxm, kSiluX, false, 0, true)>;

// 3x3 of stride 2 in two activation stages a channel block
template <int A, bool N> using Half = std::integer_sequence<int, form_of(kKind3, A, false, 0, N) | kFormHalf, form_of(kKind3, A, true, 0, N) | kFormHalf>;

// A list of kernels as (form, function) pairs.
struct FormEntry {
    int form;
    void* kernel;
};
template <typename T, typename G, int... F>
void add_forms(FormEntry* list, int& n, std::integer_sequence<int, F...>) {
    const FormEntry add[] = {{F, reinterpret_cast<void*>(conv_tc_kernel<T, G, false, F>)}...};
    for (const FormEntry& e : add) list[n++] = e;
}

constexpr int kMostForms = 80;
struct FormTable {
    FormEntry one[kMostForms], shared[kMostForms];
    int n_one = 0, n_shared = 0;
};
template <typename T>
FormTable make_forms() {
    FormTable t;
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind1, kNone>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind1, kRelu>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind1, kSilu>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind1, kSiluX>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind3, kNone>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind3, kRelu>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind3, kSilu>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Plain<kKind3, kSiluX>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Nchw<kKind1, kNone>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Nchw<kKind1, kRelu>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Nchw<kKind1, kSiluX>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Nchw<kKind3, kNone>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Nchw<kKind3, kRelu>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Nchw<kKind3, kSiluX>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Resid<kKind1, kNone, 1>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Resid<kKind1, kRelu, 1>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Resid<kKind3, kSilu, 2>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Pxm());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kNone, false>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kRelu, false>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kSilu, false>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kSiluX, false>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kNone, true>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kRelu, true>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Half<kSiluX, true>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Elem<kKind1, false>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Elem<kKind1, true>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Elem<kKind3, false>());
    add_forms<T, TcLaunch1>(t.one, t.n_one, Elem<kKind3, true>());
    // several convolutions
    add_forms<T, TcLaunchN>(t.shared, t.n_shared, std::integer_sequence<int, form_of(kKind1, -1, false, 0, false), form_of(kKind1, kNone, false, 0, false),
                                                                       form_of(kKind1, kRelu, false, 0, false), form_of(kKind1, kSilu, false, 0, false),
                                                                       form_of(kKind3, -1, false, 0, false), form_of(kKind3, kNone, false, 0, false),
                                                                       form_of(kKind3, kRelu, false, 0, false), form_of(kKind3, kSilu, false, 0, false)>());
    return t;
}

const FormTable& forms();   // of the including unit's type

inline void* find_form(int form, bool shared) {
    const FormTable& t = forms();
    const FormEntry* list = shared ? t.shared : t.one;
    for (int i = 0; i < (shared ? t.n_shared : t.n_one); ++i)
        if (list[i].form == form) return list[i].kernel;
    return nullptr;
}
// Every form may use up to the whole shared memory of an SM (asked for per function and device; it also loads the
// function, so that no first launch of one falls into a stream capture).
inline int prepare_forms() {
    const FormTable& t = forms();
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < t.n_one && e == cudaSuccess; ++i) e = cudaFuncSetAttribute(t.one[i].kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    for (int i = 0; i < t.n_shared && e == cudaSuccess; ++i)
        e = cudaFuncSetAttribute(t.shared[i].kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    return (int)e;
}

}  // namespace

#endif
