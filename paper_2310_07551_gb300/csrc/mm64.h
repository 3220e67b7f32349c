// FP64 mode products on the tensor cores: operands cut into eight 8-bit
// digits per value, exact digit products on tcgen05, integer recombination.
// Internal interface (mm64.cu).
#pragma once

#include "ds_internal.h"

namespace ds {
namespace mm {

constexpr int kMaxCat = 6;      // operand pairs concatenated along the contraction
constexpr int kMaxProd = 24;    // products of one launch
constexpr int kSlab = 16;       // contraction indices per slab (one 32-byte row of FP16 digits)
constexpr int kDigits = 8;
constexpr int kRowBlock = 128;  // rows of a tensor image's block

// One operand's "fibre view": element (r, k) of source t sits at
// (r / I) (I n) + r % I + I k.  I = 1: fibres contiguous (mode 1, or a
// matrix whose row index strides); I > 1: fibre index contiguous.
// ncat sources of n contracted entries each are laid one after the other
// along the contraction, source t multiplied by scale[t].
struct View {
    const double *src[kMaxCat];
    double scale[kMaxCat];
    int ncat, n;
    int64_t I, rows, r0;        // rows r0 .. r0 + rows - 1
    int batch;                  // this many independent views, `stride` entries apart
    int64_t stride;
};

// The digit image of a view: blocks of `rb` rows; per block and slab the
// eight digit planes [rb][kSlab] in FP16, swizzled as the tensor core reads
// them; per row its exponent (low half) and the slab of its largest entry.  Per block,
// slab and row also a mask, a bit per entry that is big against the exponent, and a
// code, the slab's own magnitude.  A batch's images follow one another, each in whole
// blocks; so do its exponents, its masks and its codes.
struct Image {
    uint8_t *data;
    int *exps;
    uint16_t *masks, *codes;
    int rb, slabs;
    int64_t rows;
    void place(uint8_t *at, int batch);
};

// out(r, i) (+)= sum over the contraction of A(r, k) B(i, k); element (r, i)
// of out at (r / I) (I cols) + r % I + I i, I of A's view.  ib.data null: B is
// cut into digits with A, for this call.  A batch (of A and B alike) writes its
// outputs `stride` entries apart.
struct Product {
    View A, B;
    Image ia, ib;
    double *out;
    int accumulate;
    int64_t stride;
};

inline int slabs_of(int n, int ncat) { return ncat * ((n + kSlab - 1) / kSlab); }
inline int64_t pad_rows(int64_t rows, int rb) { return (rows + rb - 1) / rb * rb; }
// data
inline size_t image_bytes(int64_t rows, int rb, int slabs)
{
    return (size_t)pad_rows(rows, rb) * slabs * kSlab * 2 * kDigits;
}

// data, exponents, masks and codes of one image
inline size_t image_total(int64_t rows, int rb, int slabs)
{
    return image_bytes(rows, rb, slabs) + sizeof(int) * pad_rows(rows, rb) * (1 + slabs);
}
inline void Image::place(uint8_t *at, int batch)
{
    data = at;
    exps = (int *)(data + image_bytes(rows, rb, slabs) * batch);
    masks = (uint16_t *)(exps + pad_rows(rows, rb) * batch);
    codes = masks + pad_rows(rows, rb) * slabs * batch;
}

// room for what the digit products of `rows` x `cols` outputs may leave to the FMA
// chains: 24 bytes for each column of 32 rows of a tile (and, once for a launch, kAlign
// for their count)
inline size_t left_bytes(int64_t rows, int cols, int batch)
{
    return (size_t)pad_rows(rows, kRowBlock) / 32 * 24 * (cols + 64) * batch;
}

// cycles a pipeline wait may take (the test hook DS_WAIT_LIMIT_CYCLES, else ~2 s)
long long wait_limit_default();

// Scratch of run_products for digit images, and where launch times are recorded.
struct Context {
    uint8_t *ws = nullptr;
    size_t ws_bytes = 0;
    long long wait_limit = wait_limit_default();
    Prof *prof = nullptr;
};
constexpr size_t kAlign = 256;
inline size_t aligned(size_t b) { return (b + kAlign - 1) / kAlign * kAlign; }

// The fibres of mode mu of a tensor of sizes n[0 .. d-1] (first fastest) and
// the rows of a column-major n x n matrix (of its transpose) as views.
View tensor_view(int d, const int64_t *n, int mu, const double *X);
View matrix_view(int64_t n, const double *L, int transpose, double scale = 1.0);

// Independent products of one phase: cuts the operands into digits and runs
// the digit products, in as few launches as the scratch allows (products that
// share an operand tensor next to each other share its image; a tensor whose
// image exceeds the scratch goes in row blocks), or runs them on the FP64 pipe
// where that is faster (use_digits) or the scratch is too small for one block.
// Returns the number of launches.
int run_products(const Context &c, const Product *p, int count, cudaStream_t st);
// Scratch that run_products uses in full for a phase of `count` products with
// tensors of N points and n x n matrices, `cat` concatenated terms, matrices
// cut per call or not.
size_t scratch_bytes(int64_t N, int64_t n, int count, int cat, bool matrices);
// A view's images in all, for a batch.
inline size_t image_total(const View &v, int rb)
{
    const int slabs = v.ncat * ((v.n + kSlab - 1) / kSlab);
    return aligned(image_total(v.rows, rb, slabs) * v.batch);
}
// Y = X x_1 L_1 ... x_d L_d (L^T with transpose), chained mode products; tmp:
// two tensors of N = prod n entries.
void tucker_f64(const Context &c, int d, const int64_t *n, const double *X, double *Y, const double *const *L,
                int transpose, double *tmp, cudaStream_t st);

// Columns per tile (a multiple of 16, at most 64) for matrices of `cols`
// columns in a launch of `products` products of `rows` rows and `slabs` slabs.
int tile_cols(int64_t rows, int cols, int products, int slabs);

// Digit images of up to kMaxProd views (one launch); reset: null, or a word to zero.
void launch_split(const View *v, const Image *im, int count, int *reset, cudaStream_t st);
// Up to kMaxProd products on their images.  left: a word, zero before the call, and
// from kAlign on the products' left_bytes.  Returns the number of launches.
int launch_products(const Product *p, int count, uint8_t *left, long long wait_limit, cudaStream_t st);
// The same products on the FP64 pipe, four threads per output (one launch;
// images unused): small products.
void launch_products_fma(const Product *p, int count, cudaStream_t st);
// Whether a mode product of this shape runs on the tensor cores (count
// products in the launch).
bool use_digits(int64_t rows, int n, int count);

}  // namespace mm
}  // namespace ds
