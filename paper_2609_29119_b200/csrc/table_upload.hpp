// Device tables of a plan on their way from host vectors to the device.  A large table is copied by add() itself, into an
// allocation of its own; the small ones are collected into one allocation and one copy that finish() makes (twenty of each
// took most of the time of creating a small plan).
//
// Lifetime: no address of a caller's vector is kept, so none has to outlive its add(), whether it is a temporary, local to
// a helper or changed afterwards.
#pragma once
#include <cstddef>
#include <cstring>
#include <type_traits>
#include <vector>

namespace cqt {

// Upload: bool(const void *host, size_t bytes, void *&dev), allocates device memory, copies to it and sets dev; false:
// failed.  Nothing is uploaded or set after a failure.
template <class Upload>
class TableUpload {
  public:
    static constexpr size_t kLarge = 1 << 20;   // tables of more bytes are copied by themselves

    explicit TableUpload(Upload upload) : upload_(upload) {}
    TableUpload(const TableUpload &) = delete;

    // dst: set to the table's device address (null for an empty table), by finish() for a small one
    template <class T>
    void add(T *&dst, const std::vector<T> &src) {
        static_assert(std::is_trivially_copyable<T>::value, "tables are copied byte by byte");
        dst = nullptr;
        const size_t n = src.size() * sizeof(T);
        if (n == 0 || !ok_) return;
        if (n > kLarge) {
            void *dev = nullptr;
            ok_ = upload_(static_cast<const void *>(src.data()), n, dev);
            if (ok_) dst = static_cast<T *>(dev);
            return;
        }
        const size_t off = (small_.size() + 255) / 256 * 256;
        small_.resize(off + n);
        std::memcpy(small_.data() + off, src.data(), n);
        pieces_.push_back({reinterpret_cast<void **>(&dst), off});
    }

    bool finish() {
        void *base = nullptr;
        if (ok_ && !small_.empty()) ok_ = upload_(static_cast<const void *>(small_.data()), small_.size(), base);
        if (ok_)
            for (const Piece &p : pieces_) *p.dst = static_cast<char *>(base) + p.offset;
        return ok_;
    }

  private:
    struct Piece {
        void **dst;
        size_t offset;
    };
    Upload upload_;
    bool ok_ = true;
    std::vector<char> small_;
    std::vector<Piece> pieces_;
};

}  // namespace cqt
